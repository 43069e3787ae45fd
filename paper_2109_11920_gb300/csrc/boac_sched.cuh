// boac_sched.cuh -- the bank-balanced scatter schedule of the fused
// kernels' race-free class scatter (built by a small kernel from the
// geometry alone, and kept on the device across calls by
// boac_schedcache.cu) and the scheduled scatter itself.
#pragma once

#include <cuda_runtime.h>

#include "boac_device.cuh"
#include "boac_internal.h"

namespace boac {

// ---- scatter schedule -------------------------------------------------
// The race-free class scatter adds each sample's back-projection weight to
// the four pixels of its bilinear footprint with plain read-modify-writes of
// shared memory.  In the natural order (32 lanes = 32 samples along a
// lattice row) the footprints of a warp's lanes fall on few banks for most
// grid angles (2.4-way conflicts on average at 128 x 128), and samples
// outside the image still take a lane.  The schedule lists, for every sample
// grid and class, the class's in-image samples in rounds of 32 whose
// footprint corners (0, 0) lie in 32 different banks of the padded
// accumulator (the other three corners are fixed offsets of it, so they
// differ too) and whose weights lie in 32 different banks of the sample
// buffer W -- a 32 x 32 bank assignment made greedily by one warp per
// (grid, class).  It depends on the geometry only; the order inside a class
// does not change any sum (footprints of one class are disjoint, so every
// pixel still receives its contributions class by class), so results are
// bit-identical to the natural order.  Every class has a fixed capacity of
// slots; slots after its last round hold kSchedEmpty, so the fused kernel
// can load a class's slots before it knows how many rounds it has.
template <int N>
struct SchedShape {
    static_assert(N <= 128, "entries pack k and b into 8 bits each");
    static constexpr int CLS_MAX = ((N + 2) / 3) * ((N + 2) / 3);  // samples of class (0, 0)
    // Capacity, in rounds of 32: two per warp of an 8n-thread CTA.  A class
    // is as slow as its busiest warp, and the greedy assignment below needs
    // more than 64 rounds for 43 % of the classes at 128 x 128 and 120 views
    // (53 to 85, for 1500 to 1849 samples): those ran a third round on a few
    // warps.  Samples beyond the capacity fill empty slots instead (256
    // candidates x 50 iterations, 128 x 128, 120 views: 37.6 -> 35.3 ms).
    static constexpr int ROUNDS = N / 2;
    static_assert(ROUNDS * 32 >= CLS_MAX && ROUNDS % 2 == 0, "a class fits its rounds");
    static constexpr int CLS_ENTRIES = ROUNDS * 32;
    static constexpr int CLS_WORDS = CLS_ENTRIES / 2;
};
// Slot of round r, lane l in a class's entries: rounds are stored in pairs,
// lane-interleaved, so that one 32-bit word per lane holds the lane's entry
// of both rounds (low half: the even round).
__host__ __device__ constexpr int sched_slot(int r, int lane) { return (r >> 1) * 64 + 2 * lane + (r & 1); }
constexpr unsigned short kSchedEmpty = 0xFFFFu;

__host__ __device__ constexpr size_t sched_entries(int n) {
    return n == 64 ? SchedShape<64>::CLS_ENTRIES : n == 96 ? SchedShape<96>::CLS_ENTRIES
                                                           : SchedShape<128>::CLS_ENTRIES;
}
// Per grid: 9 classes x CLS_ENTRIES entries (k << 8 | b, or kSchedEmpty).
inline size_t sched_bytes(int n, int ngrid) {
    return align256(sizeof(unsigned short) * 9 * sched_entries(n) * (size_t)ngrid);
}

// Tag of a cached schedule: the geometry and sample-buffer pitch it was
// built for (never 0).
__host__ __device__ constexpr unsigned long long sched_tag_value(int n, int V, int ngrid, int wp) {
    return 0xB0AC5C0000000000ull ^ ((unsigned long long)n << 40) ^ ((unsigned long long)(wp - n) << 31) ^
           ((unsigned long long)V << 20) ^ (unsigned long long)ngrid;
}

// One CTA per (grid, class), for a sample buffer of pitch WP (the W banks of
// the rounds).  With a tag that already holds `want` (a cached schedule of
// this geometry and pitch) every CTA returns at once.
// Two builds on different streams may write one kept schedule at the same
// time, and one stream's kernel may read it while the other's builder still
// writes.  So the entries depend on the geometry and the pitch alone (no order
// of arrival), they are worked out in shared memory, and each is stored once:
// every store writes the value that is there already or will be.
template <int N, int WP>
__global__ void __launch_bounds__(256) scatter_schedule_kernel(int V, unsigned short* __restrict__ sched,
                                                               const unsigned long long* tag,
                                                               unsigned long long want) {
    using S = SchedShape<N>;
    if (tag != nullptr && *reinterpret_cast<const volatile unsigned long long*>(tag) == want) return;
    constexpr int P = N + 1;  // the padded accumulator's pitch
    const int gi = blockIdx.x / 9, cls = blockIdx.x % 9;
    const int pk = cls / 3, pb = cls % 3;
    const int nbc = (N - pb + 2) / 3, cnt = ((N - pk + 2) / 3) * nbc;
    __shared__ unsigned short ent[S::CLS_MAX];  // samples grouped by (bank, W bank)
    __shared__ unsigned short key[S::CLS_MAX];  // (bank << 5 | W bank) of sample t, or empty
    __shared__ __align__(4) unsigned short slot[S::CLS_ENTRIES];  // the class's entries
    __shared__ int num[1024], start[1024], cur[1024];
    float cs, sn;
    cta_view_cos_sin(gi, V, &cs, &sn);  // grid gi's base view, as in the fused kernel
    const float c = 0.5f * (float)(N - 1);
    unsigned short* out = sched + ((size_t)gi * 9 + cls) * S::CLS_ENTRIES;
    for (int i = threadIdx.x; i < 1024; i += blockDim.x) num[i] = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        const int k = pk + 3 * (t / nbc), b = pb + 3 * (t % nbc);
        float u, w;
        sample_uw(k, b, cs, sn, c, &u, &w);
        unsigned short kk = kSchedEmpty;
        if (inside_open(u, w, N)) {
            const int q = ((int)floorf(w) + 1) * P + (int)floorf(u) + 1;
            kk = (unsigned short)(((q & 31) << 5) | ((k * WP + b) & 31));
            atomicAdd(&num[kk], 1);
        }
        key[t] = kk;
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // exclusive prefix sum over the 1024 cells
        const int lane = threadIdx.x;
        int s = 0;
        for (int i = 0; i < 32; ++i) s += num[lane * 32 + i];
        int incl = s;
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        int run = incl - s;
        for (int i = 0; i < 32; ++i) {
            start[lane * 32 + i] = run;
            cur[lane * 32 + i] = run;
            run += num[lane * 32 + i];
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        const unsigned short kk = key[t];
        if (kk != kSchedEmpty)
            ent[atomicAdd(&cur[kk], 1)] = (unsigned short)(((pk + 3 * (t / nbc)) << 8) | (pb + 3 * (t % nbc)));
    }
    for (int t = threadIdx.x; t < S::CLS_ENTRIES; t += blockDim.x) slot[t] = kSchedEmpty;
    __syncthreads();
    // A cell's samples in ascending order, not in the order in which the
    // atomics above let them arrive.
    for (int cell = threadIdx.x; cell < 1024; cell += blockDim.x) {
        unsigned short* e = ent + start[cell];
        for (int i = 1; i < num[cell]; ++i) {
            const unsigned short x = e[i];
            int j = i;
            for (; j > 0 && e[j - 1] > x; --j) e[j] = e[j - 1];
            e[j] = x;
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int r = 0;
        // Greedy rounds, lane q owning the samples whose footprint starts in
        // bank q: every lane with samples left proposes the free W bank
        // nearest above its own index; a W bank claimed by several lanes goes
        // to the lane with the most samples left; losers propose again among
        // the banks still free.
        const int lane = threadIdx.x;
        unsigned avail = 0;
        int left = 0;
        for (int x = 0; x < 32; ++x) {
            const int m = num[lane * 32 + x];
            if (m) avail |= 1u << x;
            left += m;
            cur[lane * 32 + x] = 0;  // taken so far
        }
        while (__any_sync(0xffffffffu, left > 0) && r < S::ROUNDS) {
            unsigned used = 0;
            int pick = -1;
            for (;;) {
                int cand = -1;
                const unsigned fr = avail & ~used;
                if (pick < 0 && fr) cand = (__ffs(__funnelshift_r(fr, fr, lane)) - 1 + lane) & 31;
                if (!__any_sync(0xffffffffu, cand >= 0)) break;
                const unsigned grp = __match_any_sync(0xffffffffu, cand);
                const unsigned pri = cand >= 0 ? ((unsigned)left << 5) | (unsigned)(31 - lane) : 0u;
                const bool win = cand >= 0 && pri == __reduce_max_sync(grp, pri);
                used |= __reduce_or_sync(0xffffffffu, win ? 1u << cand : 0u);
                if (win) {
                    const int cell = lane * 32 + cand;
                    pick = ent[start[cell] + cur[cell]];
                    if (++cur[cell] == num[cell]) avail &= ~(1u << cand);
                    --left;
                }
            }
            if (pick >= 0) slot[sched_slot(r, lane)] = (unsigned short)pick;
            ++r;
        }
        // Samples left after the last round's capacity: into the empty slots
        // of their accumulator bank (only the sample buffer's banks may then
        // clash), and those that find none into any empty slot (a class has
        // at most CLS_MAX <= CLS_ENTRIES samples: there is one for each).
        if (__any_sync(0xffffffffu, left > 0)) {
            __syncwarp();
            int cell = lane * 32;
            auto take = [&]() -> unsigned short {
                while (cur[cell] == num[cell]) ++cell;
                return ent[start[cell] + cur[cell]++];
            };
            for (int q = 0; q < r && left > 0; ++q)
                if (slot[sched_slot(q, lane)] == kSchedEmpty) {
                    slot[sched_slot(q, lane)] = take();
                    --left;
                }
            int at = 0;
            for (int l = 0; l < 32; ++l) {
                __syncwarp();
                if (lane == l)
                    for (; left > 0; --left) {
                        while (at < S::CLS_ENTRIES && slot[sched_slot(at >> 5, at & 31)] != kSchedEmpty) ++at;
                        if (at == S::CLS_ENTRIES) break;
                        slot[sched_slot(at >> 5, at & 31)] = take();
                    }
                at = __shfl_sync(0xffffffffu, at, l);
            }
        }
    }
    __syncthreads();
    // every entry once, two to a word
    for (int t = threadIdx.x; t < S::CLS_WORDS; t += blockDim.x)
        reinterpret_cast<unsigned*>(out)[t] = reinterpret_cast<const unsigned*>(slot)[t];
}

// Launch the schedule builder for images up to 128 x 128 and a sample
// buffer of pitch wp (n + 1 or n + 4): ngrid x 9 CTAs (skipped on the
// device when *tag == want).
inline int sched_launch(int n, int V, int ngrid, int wp, unsigned short* sched, cudaStream_t st,
                        const unsigned long long* tag = nullptr, unsigned long long want = 0) {
#define BOAC_SCHED_CASE(NV)                                                                              \
    case NV:                                                                                             \
        if (wp == NV + 4) scatter_schedule_kernel<NV, NV + 4><<<ngrid * 9, 256, 0, st>>>(V, sched, tag, want); \
        else if (wp == NV + 1) scatter_schedule_kernel<NV, NV + 1><<<ngrid * 9, 256, 0, st>>>(V, sched, tag, want); \
        else return BOAC_EINVAL;                                                                         \
        break;
    switch (n) {
        BOAC_SCHED_CASE(64)
        BOAC_SCHED_CASE(96)
        BOAC_SCHED_CASE(128)
        default: return BOAC_OK;
    }
#undef BOAC_SCHED_CASE
    return launch_status();
}

// The schedule of geometry (n, V, ngrid) and sample-buffer pitch wp for a
// launch on stream st: a kept one (built there when its tag does not name the
// geometry and pitch), or, when there is no room for it, built into ws
// (sched_bytes(n, ngrid) bytes of the caller's workspace).  Returns the
// schedule's address, or nullptr where none is kept and ws is nullptr;
// *status is BOAC_OK or the launch error.
const unsigned short* sched_prepare(int n, int V, int ngrid, int wp, unsigned short* ws, cudaStream_t st,
                                    int* status);

// Floats below a padded image (its last padding row starts at (N + 1) P)
// that the scatter's empty slots may add 0 to: two rows of up to 33 cells.
constexpr int kScatterPad = 33;

// A thread's words of one class of a grid's schedule (word t = tid + i NT:
// warp w's lanes hold rounds 2 (w + i NT / 32) and that + 1).
template <int N, int NT>
struct SchedSlots {
    static constexpr int CW = SchedShape<N>::CLS_WORDS;
    static constexpr int KE = (CW + NT - 1) / NT;
    unsigned e[KE];
    __device__ __forceinline__ void load(const unsigned short* __restrict__ cls_entries) {
        const unsigned* wds = reinterpret_cast<const unsigned*>(cls_entries);
#pragma unroll
        for (int i = 0; i < KE; ++i) {
            const int t = threadIdx.x + i * NT;
            e[i] = (i + 1) * NT <= CW || t < CW ? __ldg(wds + t) : 0xFFFFFFFFu;
        }
    }
};

// The class scatter of scatter_classes (boac_device.cuh), in schedule order.
// `cur` holds this thread's slots of class 0 (loaded by the caller ahead of
// time); each class loads the next class's slots before it works, so the
// loads are in flight across the class's work and its barrier.  The class
// loop is unrolled: as a loop it moves the loaded words between registers at
// the end of a class, which waits there for an L2 load of about the length of
// a class (256 candidates x 50 iterations: 31.1 -> 28.6 ms).  BRANCH:
// empty slots are skipped; else they add 0 in the padding, which the MLEM
// kernel prefers (256 candidates x 50 iterations: 31.1 against 31.6 ms) and
// the gradient kernel, shorter of registers, does not (64 candidates x 10
// iterations: 8.7 against 8.3 ms).  Preparing a slot, or the next
// class's first slot, between another slot's loads and stores is slower
// (31.6 to 36.1 ms).
//
// `side` is work that each thread does beside the classes (NoSideWork:
// none), begin(cls) at the start of class cls.
struct NoSideWork {
    __device__ __forceinline__ void begin(int) {}
};

template <int N, int NT, int P, int WP, bool BRANCH = false, class Side = NoSideWork>
__device__ __forceinline__ void scatter_scheduled(const float* __restrict__ W, float* img1, float cs, float sn,
                                                  float c, const unsigned short* __restrict__ sched,
                                                  SchedSlots<N, NT> cur, Side side = Side()) {
    constexpr int CE = SchedShape<N>::CLS_ENTRIES;
    static_assert(CE % 64 == 0, "rounds are stored in lane-interleaved pairs");
    constexpr int kPad = (N + 1) * P;  // the padding row below the image
    const int pad_cell = kPad + (((int)(threadIdx.x & 31u) - kPad) & 31);  // bank: the lane
#pragma unroll
    for (int cls = 0; cls < 9; ++cls) {
        SchedSlots<N, NT> nxt;
        if (cls < 8) nxt.load(sched + (cls + 1) * CE);
        side.begin(cls);
#pragma unroll
        for (int i = 0; i < 2 * SchedSlots<N, NT>::KE; ++i) {
            const unsigned e = cur.e[i >> 1];
            const bool high = i & 1;
            bool ok = high ? e < 0xFFFF0000u : (e & 0xFFFFu) != 0xFFFFu;
            // k and b as floats without the conversion unit: the byte above
            // the low byte of 2^15's mantissa, less 2^15 (exact: c is a
            // multiple of 1/2)
            const unsigned kf = __byte_perm(e, 0x47000000u, high ? 0x7434 : 0x7414);
            const unsigned bf = __byte_perm(e, 0x47000000u, high ? 0x7424 : 0x7404);
            const float2 kb = __fadd2_rn(make_float2(__uint_as_float(kf), __uint_as_float(bf)), pair(-32768.0f - c));
            const Cell<N, P> x(make_float2(fmaf(-kb.x, sn, fmaf(kb.y, cs, c)), fmaf(kb.x, cs, fmaf(kb.y, sn, c))));
            const int wi = (int)__dp4a(e, high ? (unsigned)WP << 24 | 1u << 16 : (unsigned)WP << 8 | 1u, 0u);
            // an entry is in (-1, n)^2 by construction (checked builds check)
            if (BRANCH && !ok) continue;
            ok = ok && index_ok(wi, (long long)N * WP) && index_ok(x.cell, (long long)P * (N + 1));
            float g = 0.0f;
            if (ok) g = W[wi];
            scatter_cell<P>(img1 + (ok ? x.cell : pad_cell), x.frac, g);
        }
        __syncthreads();
        cur = nxt;
    }
}

}  // namespace boac
