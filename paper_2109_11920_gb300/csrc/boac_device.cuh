// boac_device.cuh -- device helpers shared by every kernel of the library:
// view angles, ray-sample coordinates, bilinear sampling and its transpose.
//
// Every kernel computes the continuous pixel coordinates (u, w) of ray sample
// (k, b) with sample_uw(), so the forward projector, the back-projector and
// the gradient all use bit-identical bilinear weights (the back-projector is
// the exact transpose of the projector in float32 up to summation order).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/boac.h"

namespace boac {

// Checked builds (-DBOAC_CHECKED, libboac_checked.so): the shared-memory
// index of every bilinear gather and scatter, and every scatter-schedule
// entry, is checked before use; an index out of range is counted in this
// translation unit's fault counter and the access is skipped (never a trap
// or a fault), so a checked run reports the fault count instead of
// corrupting memory.  Normal builds compile the checks away.
#ifdef BOAC_CHECKED
static __device__ int g_bounds_faults;
__device__ __forceinline__ bool index_ok(long long i, long long n) {
    if (i >= 0 && i < n) return true;
    atomicAdd(&g_bounds_faults, 1);
    return false;
}
// Host side, one per translation unit: read (and optionally clear) the count.
#define BOAC_FAULT_READER(name)                                                              \
    int name(int reset) {                                                                    \
        int v = 0;                                                                           \
        if (cudaMemcpyFromSymbol(&v, g_bounds_faults, sizeof(int)) != cudaSuccess) return -1; \
        if (reset) {                                                                         \
            const int z = 0;                                                                 \
            if (cudaMemcpyToSymbol(g_bounds_faults, &z, sizeof(int)) != cudaSuccess) return -1; \
        }                                                                                    \
        return v;                                                                            \
    }
#else
__device__ __forceinline__ constexpr bool index_ok(long long, long long) { return true; }
#endif

// cos/sin of phi_v = 2 pi v / V (Sec. V: views uniformly spaced over the full
// angular range).  The quadrant is taken exactly, so views a quarter turn
// apart are exact rotations of each other; the in-quadrant angle is
// evaluated in float64 and rounded once to float32.
__device__ __forceinline__ void view_cos_sin(int v, int V, float* cs, float* sn) {
    long long four_v = 4LL * (long long)v;
    int quadrant = (int)((four_v / V) % 4);
    long long rem = four_v % V;
    double th = 1.5707963267948966192 * (double)rem / (double)V;
    double s, c;
    sincos(th, &s, &c);
    float fc = (float)c, fs = (float)s;
    switch (quadrant) {
        case 0: *cs = fc; *sn = fs; break;
        case 1: *cs = -fs; *sn = fc; break;
        case 2: *cs = -fc; *sn = -fs; break;
        default: *cs = fs; *sn = -fc; break;
    }
}

// view_cos_sin for a whole CTA: one thread evaluates it.  An SM does two
// float64 operations a cycle, so a float64 sine and cosine by each of 1024
// threads take 20 us.  Called by all threads; contains a barrier.
__device__ __forceinline__ void cta_view_cos_sin(int v, int V, float* cs, float* sn) {
    __shared__ float value[2];
    if (threadIdx.x == 0) view_cos_sin(v, V, &value[0], &value[1]);
    __syncthreads();
    *cs = value[0];
    *sn = value[1];
}

// Continuous (column u, row w) pixel index of ray sample k of bin b in the
// view with (cs, sn): p = s (cs, sn) + t (-sn, cs), s = (b - c) dx,
// t = (k - c) dx, c = (n - 1) / 2 (bins and samples share the pixel pitch).
// The bin term is innermost so that loops along a ray can hoist it.
__device__ __forceinline__ void sample_uw(int k, int b, float cs, float sn, float c,
                                          float* u, float* w) {
    float bc = (float)b - c;
    float kc = (float)k - c;
    *u = fmaf(-kc, sn, fmaf(bc, cs, c));
    *w = fmaf(kc, cs, fmaf(bc, sn, c));
}

__device__ __forceinline__ bool inside_open(float u, float w, int n) {
    return u > -1.0f && u < (float)n && w > -1.0f && w < (float)n;
}

// Bilinear sample of a zero-padded shared-memory image.  `img` points at
// padded element (0, 0) = pixel (-1, -1); rows are P floats apart; the pad
// ring (pixels -1 and n) holds zeros.  Samples outside (-1, n)^2 are 0.
__device__ __forceinline__ float bilerp_padded(const float* img, int P, int n, float u, float w) {
    if (!inside_open(u, w, n)) return 0.0f;
    float fj = floorf(u), fi = floorf(w);
    float au = u - fj, aw = w - fi;
    const int idx = ((int)fi + 1) * P + ((int)fj + 1);
    if (!index_ok(idx, (long long)P * (n + 1))) return 0.0f;  // idx + P + 1 < P (n + 2) + 1
    const float* p = img + idx;
    float v00 = p[0], v01 = p[1], v10 = p[P], v11 = p[P + 1];
    float top = fmaf(au, v01 - v00, v00);
    float bot = fmaf(au, v11 - v10, v10);
    return fmaf(aw, bot - top, top);
}

// ---- packed sampling --------------------------------------------------
// The fused kernels issue an instruction on more than half of all cycles
// (about 130 per sample of a grid and iteration), a third of them here, so
// their sampling uses sm_103's two-wide float instructions: one instruction
// computes both coordinates of a sample or both rows of a bilinear read, and
// floor() and its integer come from one rounded addition instead of four
// trips through the conversion unit.  Every lane performs the operations of
// the scalar functions above in the same order, so the results are the same
// bits.  256 candidates x 50 iterations, 128 x 128, 120 views: 35.3 -> 33.5
// ms (the scalar form of the same floor gains nothing).
//
// floor() without the conversion unit: adding 1.5 * 2^23 with rounding
// towards -inf leaves 1.5 * 2^23 + floor(x) (|x| < 2^22), whose bit pattern
// is kFloorBits + floor(x).
constexpr float kFloorBias = 12582912.0f;
constexpr unsigned kFloorBits = 0x4B400000u;

__device__ __forceinline__ float2 pair(float x) { return make_float2(x, x); }
// a - b, both lanes
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, pair(-1.0f), a); }
// a - b c, both lanes, rounded once
__device__ __forceinline__ float2 sub2_mul(float2 a, float2 b, float2 c) {
    return __ffma2_rn(b, make_float2(-c.x, -c.y), a);
}

// A sample's cell in an image of side N padded to pitch P: `frac` the
// fractions (au, aw), `cell` the padded index of its top left neighbour,
// `in` whether the footprint touches the image.
template <int N, int P>
struct Cell {
    float2 frac;
    int cell;
    bool in;
    __device__ __forceinline__ explicit Cell(float2 pos) {
        const float2 t = __fadd2_rd(pos, pair(kFloorBias));
        frac = sub2(pos, __fadd2_rn(t, pair(-kFloorBias)));
        const unsigned bj = __float_as_uint(t.x), bi = __float_as_uint(t.y);
        // floor in [-1, N - 1]: the sample lies in [-1, N)^2 (at -1 every
        // weight of a pixel inside is 0)
        in = bj - (kFloorBits - 1) <= (unsigned)N && bi - (kFloorBits - 1) <= (unsigned)N;
        cell = (int)(bi * P + bj - (kFloorBits - 1u) * (P + 1u));
    }
};

// The samples of one ray column, k = k0, k0 + 1, ...: next() returns the
// position (u, w) that sample_uw gives and moves to the next sample.
struct ColumnWalk {
    float2 base, kc;
    float2 dir;
    __device__ __forceinline__ ColumnWalk(int k0, int b, float cs, float sn, float c) {
        const float bc = (float)b - c;
        base = make_float2(fmaf(bc, cs, c), fmaf(bc, sn, c));
        kc = pair((float)k0 - c);
        dir = make_float2(-sn, cs);
    }
    __device__ __forceinline__ float2 next() {
        const float2 pos = __ffma2_rn(kc, dir, base);
        kc = __fadd2_rn(kc, pair(1.0f));
        return pos;
    }
};

// The bilinear sample, and its transpose (g times each weight added), of the
// footprint at p with fractions frac, as bilerp_padded and scatter_padded
// compute them.
template <int P>
__device__ __forceinline__ float bilerp_cell(const float* p, float2 frac) {
    const float2 v0 = make_float2(p[0], p[P]), v1 = make_float2(p[1], p[P + 1]);
    const float2 tb = __ffma2_rn(pair(frac.x), sub2(v1, v0), v0);  // (top, bottom)
    return fmaf(frac.y, tb.y - tb.x, tb.x);
}
template <int P>
__device__ __forceinline__ void scatter_cell(float* p, float2 frac, float g) {
    const float g1 = __fmul_rn(g, frac.y);
    const float2 row = make_float2(__fsub_rn(g, g1), g1);  // weights of the footprint's rows
    const float2 au = pair(frac.x);
    const float2 left = __fadd2_rn(make_float2(p[0], p[P]), sub2_mul(row, row, au));
    const float2 right = __ffma2_rn(row, au, make_float2(p[1], p[P + 1]));
    p[0] = left.x;
    p[1] = right.x;
    p[P] = left.y;
    p[P + 1] = right.y;
}

// bilerp_padded at a position.
template <int N, int P>
__device__ __forceinline__ float bilerp_pos(const float* img, float2 pos) {
    const Cell<N, P> x(pos);
    if (!x.in || !index_ok(x.cell, (long long)P * (N + 1))) return 0.0f;
    return bilerp_cell<P>(img + x.cell, x.frac);
}

// Transpose of bilerp_padded: add g times each bilinear weight to the four
// neighbours (non-atomic read-modify-write; callers guarantee that no two
// threads touch the same pixel concurrently).
__device__ __forceinline__ void scatter_padded(float* img, int P, int n, float u, float w, float g) {
    if (!inside_open(u, w, n)) return;
    float fj = floorf(u), fi = floorf(w);
    float au = u - fj, aw = w - fi;
    const int idx = ((int)fi + 1) * P + ((int)fj + 1);
    if (!index_ok(idx, (long long)P * (n + 1))) return;
    float* p = img + idx;
    float g1 = g * aw, g0 = g - g1;          // row weights (1 - aw), aw
    float g01 = g0 * au, g00 = g0 - g01;     // (1-aw)(1-au), (1-aw) au
    float g11 = g1 * au, g10 = g1 - g11;     // aw (1-au), aw au
    p[0] += g00;
    p[1] += g01;
    p[P] += g10;
    p[P + 1] += g11;
}

// Bilinear sample of an unpadded global-memory image with per-neighbour
// bounds checks (plain kernels).
__device__ __forceinline__ float bilerp_global(const float* __restrict__ img, int n, float u, float w) {
    if (!inside_open(u, w, n)) return 0.0f;
    float fj = floorf(u), fi = floorf(w);
    float au = u - fj, aw = w - fi;
    int j0 = (int)fj, i0 = (int)fi;
    float v00 = 0.f, v01 = 0.f, v10 = 0.f, v11 = 0.f;
    bool jl = j0 >= 0, jh = j0 + 1 < n, il = i0 >= 0, ih = i0 + 1 < n;
    if (il && jl) v00 = __ldg(img + i0 * n + j0);
    if (il && jh) v01 = __ldg(img + i0 * n + j0 + 1);
    if (ih && jl) v10 = __ldg(img + (i0 + 1) * n + j0);
    if (ih && jh) v11 = __ldg(img + (i0 + 1) * n + j0 + 1);
    float top = fmaf(au, v01 - v00, v00);
    float bot = fmaf(au, v11 - v10, v10);
    return fmaf(aw, bot - top, top);
}

// Bilinear weight with which ray sample (u, w) reads pixel (i, j): the same
// products as scatter_padded (exact transpose of the forward weights).
__device__ __forceinline__ float pixel_weight(float u, float w, int i, int j, int n) {
    if (!inside_open(u, w, n)) return 0.0f;
    float fj = floorf(u), fi = floorf(w);
    int j0 = (int)fj, i0 = (int)fi;
    int dj = j - j0, di = i - i0;
    if ((unsigned)dj > 1u || (unsigned)di > 1u) return 0.0f;
    float au = u - fj, aw = w - fi;
    float r = di ? aw : 1.0f - aw;
    float cw = dj ? au : 1.0f - au;
    return r * cw;
}

// Transposed bilinear scatter of a whole sample grid, race-free without
// atomics: G (n x n samples, row pitch WP) is added into the padded
// accumulator img1 (row pitch P) with the weights of grid (cs, sn).  Samples
// are split into 9 classes by (k mod 3, b mod 3); two samples of one class
// are >= 3 lattice steps apart, i.e. more than 2 pixels apart along some
// image axis, so their 2x2 footprints are disjoint and a class is a plain
// read-modify-write pass.  Classes run in a fixed order (deterministic).
// Called by all NT threads of the CTA; ends with a barrier.
template <int N, int NT, int P, int WP>
__device__ __forceinline__ void scatter_classes(const float* __restrict__ W, float* img1, float cs,
                                                float sn, float c) {
#pragma unroll
    for (int cls = 0; cls < 9; ++cls) {
        const int pk = cls / 3, pb = cls % 3;
        const int nkc = (N - pk + 2) / 3, nbc = (N - pb + 2) / 3;
        for (int t = threadIdx.x; t < nkc * nbc; t += NT) {
            const int k = pk + 3 * (t / nbc), b = pb + 3 * (t % nbc);
            if (!index_ok(k * WP + b, (long long)N * WP)) continue;
            const float g = W[k * WP + b];
            float u, w;
            sample_uw(k, b, cs, sn, c, &u, &w);
            scatter_padded(img1, P, N, u, w, g);
        }
        __syncthreads();
    }
}

}  // namespace boac
