// boac_fused.cu -- batched MLEM in one persistent fused kernel (Sec. III,
// step 3: "a fixed number of MLEM iterations ... for each candidate set c_k",
// with the system matrix, forward- and back-projection on the GPU, Sec. III
// last paragraph).
//
// One CTA owns one candidate at a time and keeps its whole state on chip:
//   img0  F (padded n+2 rows x n+1 floats, zero ring)   -- mu during set-up
//   img1  back-projection accumulator (same layout)
//   W     n x (n+4) ray-sample buffer (F samples, then G = dx a r)
// and in its SM's tensor memory the attenuation of the grid in flight.
// The candidate's "system matrix" -- the attenuation of every ray sample --
// is built once per candidate into a per-CTA slot of the workspace (as
// exp2 exponents) and read back, coalesced, in every iteration: the next
// grid's exponents go into tensor memory while this grid is scattered, and
// the factors taken from them in the forward passes stay there for the
// back-projection weights.
//
// Four views share one sample grid: with bins and ray samples on the pixel
// pitch, the grids of phi, phi + pi/2, phi + pi and phi + 3pi/2 are the same
// set of points (a quarter turn maps the lattice onto itself), so sample
// (k, b) of view phi + pi is sample (n-1-k, n-1-b) of view phi, and the rays
// of phi + pi/2 and phi + 3pi/2 are the grid's rows.  One bilinear sampling of
// F serves four views (column sums for phi, phi + pi; row sums for the other
// two), and the four views' back-projection weights
//   G = dx (a_phi r_phi + a_{phi+pi} r_{phi+pi} + a_{phi+pi/2} r + a_{phi+3pi/2} r)
// are summed on the grid before ONE transposed-bilinear scatter.  View counts
// that are not a multiple of 4 use pairs (phi, phi + pi) the same way.
//
// The scatter is race-free and deterministic without atomics: the samples
// are split into 9 classes by (k mod 3, b mod 3); two samples of one class
// are >= 3 lattice steps apart, i.e. >= 3/sqrt(2) > 2 pixels apart along
// some image axis, so their 2x2 pixel footprints are disjoint.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "boac_fused_kernel.cuh"

namespace boac {

// ---------------------------------------------------------------- host side
// Launch shapes: for each image side, CTAs of 2n, 4n or 8n threads (at most
// 1024), with four or two views per sample grid: configuration id =
// 2 * shape + (1 for two views per grid).  Ids 6, 7 and 8 are the cluster
// kernel (boac_band.cu, four views per grid only): 5, 6 or 8 CTAs per
// candidate for 256 x 256 images, 2, 4 or 8 for 128 x 128.
// Ids 9 .. 16 are the fused kernel's cluster mode (images up to 128 x 128,
// four views per grid, CTAs of 8n threads) with 2, 3, 4, 6, 8, 9, 12 or 16
// CTAs per candidate, each on its share of the sample grids.
constexpr int kShapes = 3;
constexpr int kBandConfigs = 3;
constexpr int kTableConfigs = 2 * kShapes + kBandConfigs;
constexpr int kConfigs = kTableConfigs + kSplitConfigs;

template <int N, int NT, bool QUAD>
static int fused_launch_t(const FusedArgs& a, int slots, cudaStream_t st) {
    // once per device: allow the large dynamic shared-memory carve-out
    constexpr int kDev = 64;
    static bool attr_set[kDev];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDev) return launch_status();
    if (!attr_set[dev]) {
        if (cudaFuncSetAttribute(mlem_fused_kernel<N, NT, QUAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fused_smem_bytes<N, NT>(kMaxViews)) != cudaSuccess)
            return launch_status();
        attr_set[dev] = true;
    }
    cudaLaunchAttribute attr[1];
    overlap_attribute(&attr[0], a);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)slots, 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = fused_smem_bytes<N, NT>(a.V);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, mlem_fused_kernel<N, NT, QUAD>, a) != cudaSuccess) return launch_status();
    return launch_status();
}

template <int N, int NT, bool QUAD>
static FusedVariant make_variant() {
    return FusedVariant{N, NT, QUAD, 1, smem_of<N, NT>, (const void*)mlem_fused_kernel<N, NT, QUAD>,
                        fused_prepare_t<N, NT, QUAD>, fused_launch_t<N, NT, QUAD>, 1, nullptr,
                        fused_image_floats<N, NT>(), fused_tmem_columns<N, NT, QUAD>()};
}

template <int N, int NB>
static size_t band_smem_of(int) { return band_smem_bytes(N, NB); }
template <int N, int NB>
static int band_prepare_of(FusedArgs* a, cudaStream_t st) {
    return band_prepare(N, NB, *a, st);
}
template <int N, int NB>
static int band_launch_of(const FusedArgs& a, int clusters, cudaStream_t st) {
    return band_launch(N, NB, a, clusters, st);
}
template <int N, int NB>
static FusedVariant make_band_variant() {
    return FusedVariant{N, 4 * N, true, NB, band_smem_of<N, NB>, nullptr, band_prepare_of<N, NB>,
                        band_launch_of<N, NB>, 1, nullptr, 0, 0};
}

#define BOAC_SHAPES(NV)                                                                        \
    make_variant<NV, 2 * NV, true>(), make_variant<NV, 2 * NV, false>(),                       \
        make_variant<NV, 4 * NV, true>(), make_variant<NV, 4 * NV, false>(),                   \
        make_variant<NV, (8 * NV > 1024 ? 1024 : 8 * NV), true>(),                             \
        make_variant<NV, (8 * NV > 1024 ? 1024 : 8 * NV), false>()
#define BOAC_NO_BAND FusedVariant{}, FusedVariant{}, FusedVariant{}
static const FusedVariant* variant_table(int n) {
    static const FusedVariant t64[kTableConfigs] = {BOAC_SHAPES(64), make_band_variant<64, 2>(),
                                                    make_band_variant<64, 4>(), make_band_variant<64, 8>()};
    static const FusedVariant t96[kTableConfigs] = {BOAC_SHAPES(96), BOAC_NO_BAND};
    static const FusedVariant t128[kTableConfigs] = {BOAC_SHAPES(128), make_band_variant<128, 2>(),
                                                     make_band_variant<128, 4>(), make_band_variant<128, 8>()};
    static const FusedVariant t256[kTableConfigs] = {BOAC_SHAPES(256), make_band_variant<256, 5>(),
                                                     make_band_variant<256, 6>(), make_band_variant<256, 8>()};
    switch (n) {
        case 64: return t64;
        case 96: return t96;
        case 128: return t128;
        case 256: return t256;
        default: return nullptr;
    }
}

// Default configuration of the one-CTA kernel: the largest CTA that keeps
// >= 64 registers per thread at the occupancy shared memory allows; four
// views per grid when V % 4 == 0.
static int single_cta_config(const boac_geom* g) {
    const int shape = g->n == 64 ? 1 : 2;
    return 2 * shape + (g->n_views % 4 == 0 ? 0 : 1);
}

static const FusedVariant* get_variant(const boac_geom* g, int config);

// Cluster mode for a batch too small to fill the GPU one CTA per candidate
// (images up to 128 x 128, V % 4 == 0): the cluster size G with the least
// modelled time, rounds(G) (ceil(grids / G) + 1.6) grid passes per
// iteration, where rounds(G) = ceil(B / clusters of G resident at once) and
// 1.6 grid passes stand for the cluster's per-iteration exchange; the
// smaller G on a tie; and only if that beats one CTA per candidate, whose
// even split of the batch's iterations costs grids B / min(B, SMs) passes
// per iteration.  Returns the configuration id, or -1.  (1.6 was fitted to
// earlier kernels and is high: an iteration at 128 x 128 and 120 views takes
// 295 us on one CTA, 151 / 81 / 44 / 28 us on G = 2 / 4 / 8 / 16, that is 9.8 us
// per grid pass and 0.2 to 0.8 passes of exchange.)
static int split_config(const boac_geom* g, int B) {
    if (g->n > 128 || g->n_views % 4 != 0 || B < 1) return -1;
    const int sms = sm_count();
    if (sms <= 0) return -1;
    const int ngrid = g->n_views / 4;
    int best = -1;
    double best_t = (double)ngrid * B / (B < sms ? B : sms);  // one CTA per candidate
    for (int i = 0; i < kSplitConfigs; ++i) {
        const int cfg = 2 * kShapes + kBandConfigs + i;
        const FusedVariant* v = get_variant(g, cfg);
        if (!v) continue;
        const int h = v->max_clusters();
        if (h <= 0) continue;
        const int rounds = (B + h - 1) / h;
        const double t = rounds * ((ngrid + v->g - 1) / v->g + 1.6);
        if (t < best_t - 1e-9) {
            best = cfg;
            best_t = t;
        }
    }
    return best;
}

// Default configuration for B candidates.  Batches too small to fill the
// GPU one candidate per CTA (images up to 128 x 128, V % 4 == 0) take the
// fused kernel's cluster mode (split_config).  256 x 256 images with
// V % 4 == 0 take the band kernel with the cluster size that keeps the most
// SMs busy (clusters are placed within one GPC, so the resident count
// depends on the size); the smaller cluster on a tie.  Otherwise the one-CTA
// kernel.
static int default_config(const boac_geom* g, int B) {
    const int sc = split_config(g, B);
    if (sc >= 0) return sc;
    if (g->n == 64 && B >= 1 && B <= 2 * sm_count()) {
        // at most two candidates per SM: CTAs of 8n threads (60 views, us per grid
        // of a CTA alone on its SM: 4.1, of 4n threads 5.3); beyond, three of 4n
        // threads per SM (456 candidates x 20 iterations 3.32 ms)
        return 2 * 2 + (g->n_views % 4 == 0 ? 0 : 1);
    }
    if (g->n == 256 && g->n_views % 4 == 0) {
        static const int nbs[kBandConfigs] = {5, 6, 8};
        int best = -1, best_ctas = 0;
        for (int i = 0; i < kBandConfigs; ++i) {
            const int ctas = band_max_clusters(256, nbs[i]) * nbs[i];
            if (ctas > best_ctas) {
                best = i;
                best_ctas = ctas;
            }
        }
        if (best >= 0) return 2 * kShapes + best;
    }
    return single_cta_config(g);
}

// Batches small enough that the unfused batched kernels (boac_unfused.cu:
// many CTAs per candidate) finish before the fused kernel's one CTA or one
// cluster per candidate does, for the geometries without the cluster mode
// (view counts not divisible by 4, 256 x 256 images): up to 32 candidates at
// 64 x 64 and 96 x 96, 16 at 128 x 128, 2 at 256 x 256.  Both paths scale with
// the view count, so the bound is per image size, scaled with the SM count.
// (The bounds were fitted to earlier kernels and are low: ms of 20 iterations,
// unfused against fused, 64 x 64 and 90 views 32 candidates 1.42 / 3.84, 64
// 2.62 / 3.86; 96 x 96 32 2.55 / 5.86; 128 x 128 16 2.67 / 8.87; 256 x 256 and 90
// views 4 9.5 / 190, 180 views 2 10.0 / 19.3, 4 17.8 / 21.2.)
static bool use_unfused(const boac_geom* g, int B) {
    if (split_config(g, B) >= 0) return false;
    int cap;
    switch (g->n) {
        case 64:
        case 96: cap = 32; break;
        case 128: cap = 16; break;
        case 256: cap = 2; break;
        default: return false;
    }
    const int sms = sm_count();
    return sms > 0 && (long long)B * 152 <= (long long)cap * sms;
}

static const FusedVariant* get_variant(const boac_geom* g, int config) {
    const bool split = config >= kTableConfigs;
    const FusedVariant* t = split ? split_variants(g->n) : variant_table(g->n);
    if (!t || config < 0 || config >= kConfigs) return nullptr;
    const FusedVariant* v = &t[split ? config - kTableConfigs : config];
    if (!v->launch) return nullptr;
    if (v->quad ? (g->n_views % 4 != 0) : (g->n_views % 2 != 0)) return nullptr;
    if (v->nb > 1 && !band_supported(g->n, g->n_views, v->nb)) return nullptr;
    if (v->g > 1 && (g->n_views < 4 * v->g)) return nullptr;  // at least one grid per rank
    return v;
}

// CTAs of a kernel that fit an SM by registers (given out in units of 8 per
// thread to the warps of the SM's four parts), shared memory, threads and
// columns of tensor memory; 0 after an error.  The runtime's occupancy query
// answers 1 for every kernel that allocates tensor memory, whatever its size,
// while the SM holds as many as fit: taken at its word it left 64 x 64 batches
// of more than one candidate per SM with one CTA on each (20 iterations: 456
// candidates of 60 views 5.44 -> 3.32 ms, 1000 12.13 -> 7.37, 456 of 90 views
// 17.7 -> 8.9).
static int resident_ctas(const FusedVariant* v, int dev) {
    cudaFuncAttributes fa;
    int regs = 0, smem = 0, reserved = 0, threads = 0;
    if (cudaFuncGetAttributes(&fa, v->func) != cudaSuccess ||
        cudaDeviceGetAttribute(&regs, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&threads, cudaDevAttrMaxThreadsPerMultiProcessor, dev) != cudaSuccess)
        return 0;
    const int warps = (v->nt + 31) / 32, per_warp = (fa.numRegs + 7) / 8 * 8 * 32;
    const int by_regs = 4 * (regs / 4 / per_warp) / warps;
    const int by_smem = (int)(smem / (v->smem(kMaxViews) + fa.sharedSizeBytes + reserved));
    return std::min({by_regs, by_smem, threads / v->nt, kTmemColumns / v->tmem_cols});
}

// Resident CTAs per SM of a variant, computed for the largest view table it
// may be launched with (the per-view table is a few KB, so this equals the
// occupancy at every view count); cached per device.
static int variant_occupancy(const FusedVariant* v, int V) {
    constexpr int kDev = 64;
    static int cached[kDev][4][kTableConfigs];  // 0 = not yet computed
    int dev = 0;
    if (V < 0 || V > kMaxViews) return 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
        cudaGetLastError();
        return 0;
    }
    const int ni = v->n == 64 ? 0 : (v->n == 96 ? 1 : (v->n == 128 ? 2 : 3));
    const int ci = (int)(v - variant_table(v->n));
    if (dev < kDev && cached[dev][ni][ci]) return cached[dev][ni][ci];
    if (cudaFuncSetAttribute(v->func, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)v->smem(kMaxViews)) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (v->tmem_cols > 0) nb = resident_ctas(v, dev);
    else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, v->func, v->nt, v->smem(kMaxViews)) != cudaSuccess)
        nb = 0;
    if (nb <= 0) {
        cudaGetLastError();
        return 0;
    }
    if (dev < kDev) cached[dev][ni][ci] = nb;
    return nb;
}

// Workspace of the fused kernels for `holders` CTAs (or clusters) and B
// candidates:
//   [0, 256)   status word (BOAC_OK, or BOAC_ETIMEOUT from a bounded wait)
//   tables     attenuation exponents, one region per CTA
//   sens       sensitivity image (cluster kernel: band rows) per CTA
//   images     one-CTA kernel, n > 128: padded F / accumulator / sample
//              buffer per CTA; cluster kernel: the record kernel's flag and
//              the ray-run records of every (band, grid)
//   ready      one flag per candidate (the work split's hand-over), then the
//              count of finished CTAs (ragged batches)
//   sched      one-CTA kernel, n <= 128: the scatter schedule (geometry only)
struct FusedLayout {
    size_t status, tab, sens, img, geo, ready, sched, total;
};

static FusedLayout fused_layout(const boac_geom* g, const FusedVariant* v, int holders, int B) {
    FusedLayout l;
    const size_t ctas = (size_t)holders * v->nb * v->g;
    l.status = 0;
    l.tab = 256;
    if (v->nb > 1) {
        l.sens = l.tab + align256(sizeof(float) * ctas * band_tab_floats(g->n, v->nb, g->n_views));
        l.img = l.sens + align256(sizeof(float) * ctas * band_sens_floats(g->n, v->nb));
        l.geo = l.img + 256;
        l.ready = l.geo + align256(band_geo_bytes(g->n, v->nb, g->n_views));
    } else {
        l.sens = l.tab + align256(sizeof(float) * ctas * fused_tab_floats(g->n, g->n_views, v->quad, v->g));
        l.img = l.sens + align256(sizeof(float) * ctas * g->n * g->n);
        // the images and sample buffer of sides held in global memory
        l.geo = l.img + align256(fused_global_images(g->n) ? sizeof(float) * ctas * v->image_floats : 0);
        l.ready = l.geo;
    }
    l.sched = l.total = l.ready + align256(sizeof(int) * ((size_t)B + 1));
    if (v->nb == 1 && g->n <= 128) l.total = l.sched + sched_bytes(g->n, v->quad ? g->n_views / 4 : g->n_views / 2);
    return l;
}

// CTAs (one-CTA kernel) or clusters that run at once, at most B.
static int variant_holders(const boac_geom* g, const FusedVariant* v, int B) {
    long long h;
    if (v->nb > 1) {
        h = band_max_clusters(g->n, v->nb);
    } else if (v->g > 1) {
        h = v->max_clusters();
    } else {
        const int per_sm = variant_occupancy(v, g->n_views);
        h = (long long)per_sm * sm_count();
    }
    if (h <= 0) return 0;
    return (int)(h < B ? h : B);
}

// Of them, those that a batch of B candidates with K iterations each is split
// over.  Where several 64 x 64 CTAs fit an SM, a second one takes the two r = 1.6
// times the time of one (two views per grid r = 1.4), so a whole candidate per
// CTA takes r (K + s), s iterations' time for set-up and score; one CTA per SM
// with an even split takes K B / SMs, and 2.5 iterations more than r s for its
// second and third candidates: the shorter of the two.  (60 views, 160 and 200
// candidates: 20 iterations 1.66 and 2.06 against 2.24 and 2.25 ms, one
// iteration 0.46 and 0.46 against 0.36 and 0.37.)
static int split_holders(const boac_geom* g, const FusedVariant* v, int B, long long K) {
    const int h = variant_holders(g, v, B), sms = sm_count();
    if (v->nb > 1 || v->g > 1 || sms <= 0 || h <= sms) return h;
    return ((v->quad ? 1.6 : 1.4) - (double)B / sms) * K > 2.5 ? sms : h;
}

size_t fused_workspace_bytes(const boac_geom* g, int B) {
    if (use_unfused(g, B)) return unfused_workspace_bytes(g, B);
    const FusedVariant* v = get_variant(g, default_config(g, B));
    const int h = v ? variant_holders(g, v, B) : 0;
    return h > 0 ? fused_layout(g, v, h, B).total : 0;
}

// Units per CTA of the work split: the larger of an even share and the
// longest candidate (so that a candidate is never cut into three parts).
static long long split_cap(long long units, long long longest, int slots) {
    const long long share = (units + slots - 1) / slots;
    return share > longest ? share : longest;
}

static FusedArgs base_args(const boac_geom* g, const float* mu, const float* S, long long s_stride,
                           float* F, int K, int B, double* L, int include_lgamma, char* ws,
                           const FusedLayout& l) {
    FusedArgs a;
    a.mu = mu;
    a.S = S;
    a.s_stride = s_stride;
    a.F = F;
    a.L = L;
    a.include_lgamma = include_lgamma;
    a.lgS = nullptr;
    a.B = B;
    a.V = g->n_views;
    a.K = K;
    a.dx = g->pixel_cm;
    a.tab = reinterpret_cast<float*>(ws + l.tab);
    a.sens = reinterpret_cast<float*>(ws + l.sens);
    a.img = reinterpret_cast<float*>(ws + l.img);
    a.desc = nullptr;
    a.job_start = nullptr;
    a.cap = 0;
    a.ready = reinterpret_cast<int*>(ws + l.ready);
    a.status = reinterpret_cast<int*>(ws + l.status);
    a.geo = reinterpret_cast<const int*>(ws + l.geo);
    a.geo_bad = reinterpret_cast<int*>(ws + l.img);
    a.wait_cycles = wait_cycles();
    a.withhold = -1;
    a.sched = l.total > l.sched ? reinterpret_cast<const unsigned short*>(ws + l.sched) : nullptr;
    a.overlap = 0;
    a.done = a.ready + B;
    return a;
}

static std::atomic<long long> g_wait_cycles{kWaitCycles};
long long wait_cycles() { return g_wait_cycles.load(std::memory_order_relaxed); }

// Uniform batch: zero the status and ready flags, then launch the CTAs that
// have work under the split.
static int launch_uniform(const boac_geom* g, const FusedVariant* v, int slots, const float* mu,
                          const float* S, long long s_stride, float* F, int K, int B, double* L,
                          int include_lgamma, char* ws, cudaStream_t st) {
    const FusedLayout l = fused_layout(g, v, slots, B);
    FusedArgs a = base_args(g, mu, S, s_stride, F, K, B, L, include_lgamma, ws, l);
    const long long per = K > 0 ? K : 1, units = (long long)B * per;
    a.cap = split_cap(units, per, slots);
    const int grid = (int)((units + a.cap - 1) / a.cap);
    // (cluster mode takes whole candidates: no hand-over flags)
    if (cudaMemsetAsync(ws + l.status, 0, sizeof(int), st) != cudaSuccess ||
        (v->g == 1 && cudaMemsetAsync(ws + l.ready, 0, sizeof(int) * (size_t)B, st) != cudaSuccess))
        return launch_status();
    // one shared sinogram: its ln S! sum once, in the status slot's spare bytes
    if (L && include_lgamma && s_stride == 0) {
        BOAC_RANGE("score: ln S! of the shared sinogram");
        a.lgS = lgamma_sum(g->n_views * g->n_bins, S, reinterpret_cast<double*>(ws + l.status + 8), st);
    }
    BOAC_RANGE("fused MLEM: set-up, iterations, score");
    const int s = v->prepare(&a, st);
    return s == BOAC_OK ? v->launch(a, grid, st) : s;
}

// ---------------------------------------------------------------- ragged
// Ragged workspace: [0, 256) status word; per class: the candidates'
// records, their unit offsets (job_start, B_c + 1 values) and the class's
// fused layout (without its own status word).
struct RaggedPlan {
    int cls_count[kMaxRaggedClasses];
    long long units[kMaxRaggedClasses], longest[kMaxRaggedClasses];
    double chain[kMaxRaggedClasses];  // modelled time of the class's busiest CTA
    bool shares_sm[kMaxRaggedClasses];  // several of the class's CTAs fit an SM
    bool alone[kMaxRaggedClasses];      // the class's kernel runs before the others, on the whole GPU
    int slots[kMaxRaggedClasses];
    const FusedVariant* var[kMaxRaggedClasses];
    size_t desc_off[kMaxRaggedClasses], start_off[kMaxRaggedClasses], layout_off[kMaxRaggedClasses];
    size_t total;
};

// Shares the SMs out among the classes, whose kernels run at once.  A class
// of one-CTA candidates needs at least the SMs that finish its work in the
// time T of the longest chain: T starts at the larger of the longest
// candidate's time and the even share of all work, and grows until the
// classes fit the GPU together.  Time per sample grid, modelled as that of its
// samples and of 7200 more for its barriers (0.36 to 0.42 ns each: 9.9 us at 128 x
// 128, 6.8 at 96 x 96, 4.1 at 64 x 64); two views per grid 0.85 times that (8.9,
// 6.1, 4.5 us); a second and third CTA on an SM count as 0.45 of one each.  (They
// take 0.6 and 0.75: 64 x 64, 60 views, 20 iterations of 152, 304 and 456
// candidates 1.41, 2.28 and 3.32 ms.  With 0.65, batches take longer: 600 beside
// 152 of 128 x 128 13.6 against 12.6 ms, 128 beside 128 8.8 against 7.3.)
//
// The one-CTA kernel at 256 x 256 keeps its images in global memory and slows
// down with the CTAs that share L2: 200, 320 and 525 us per grid of two views
// with 8, 64 and 152 of them, 6.6 times the time of a kernel with its images on
// chip and 0.085 more per CTA.  Up to kSharedGlobalCtas such CTAs run beside
// the other classes (32 candidates of 90 views and 16 of 180: 118 ms, one class
// after the other 129); more of them run first, alone, since they and the others
// then take each other's L2 (64 beside 152 of 128 x 128: 135 ms, one after the
// other 111).
//
// A split only decides which CTA runs which iterations, never what they compute.
constexpr int kSharedGlobalCtas = 32;
static void ragged_share(const boac_geom* classes, int n_classes, RaggedPlan* pl) {
    const int sms = sm_count();
    double cost[kMaxRaggedClasses], T = 0.0, work = 0.0;
    int per_sm[kMaxRaggedClasses], classes_in_use = 0;
    for (int c = 0; c < n_classes; ++c) {
        const FusedVariant* v = pl->var[c];
        const boac_geom& g = classes[c];
        per_sm[c] = v->nb > 1 || v->g > 1 ? 0 : variant_occupancy(v, g.n_views);
        cost[c] = (v->quad ? g.n_views / 4 : 0.85 * (g.n_views / 2)) * ((double)g.n * g.n + 7200.0) *
                  (per_sm[c] > 1 ? 1.0 + 0.45 * (per_sm[c] - 1) : 1.0);
        const bool global = per_sm[c] > 0 && fused_global_images(g.n);
        if (global) cost[c] *= 6.6 + 0.085 * pl->slots[c];
        pl->alone[c] = global && pl->slots[c] > kSharedGlobalCtas;
        pl->chain[c] = 0.0;
        pl->shares_sm[c] = per_sm[c] > 1;
        if (pl->cls_count[c] == 0 || pl->alone[c]) continue;
        ++classes_in_use;
        const int ctas = v->nb > 1 ? v->nb : v->g;
        pl->chain[c] = cost[c] / ctas * split_cap(pl->units[c], pl->longest[c], pl->slots[c]);
        if (per_sm[c] == 0) continue;  // clusters: as many as are resident, where SMs are free
        if (cost[c] * pl->longest[c] > T) T = cost[c] * pl->longest[c];
        work += cost[c] * pl->units[c] / per_sm[c];
    }
    if (classes_in_use < 2 || sms <= 0 || work <= 0.0) return;
    if (work / sms > T) T = work / sms;
    for (int step = 0; step < 200; ++step, T *= 1.01) {
        int need[kMaxRaggedClasses], used = 0;
        for (int c = 0; c < n_classes; ++c) {
            need[c] = 0;
            if (pl->cls_count[c] == 0 || per_sm[c] == 0 || pl->alone[c]) continue;
            const double n = ceil(pl->units[c] * cost[c] / T);
            need[c] = n < pl->slots[c] ? (int)n : pl->slots[c];
            used += (need[c] + per_sm[c] - 1) / per_sm[c];
        }
        if (used > sms) continue;
        for (int c = 0; c < n_classes; ++c)
            if (need[c] > 0) {
                pl->slots[c] = need[c];
                pl->chain[c] = cost[c] * split_cap(pl->units[c], pl->longest[c], need[c]);
            }
        return;
    }
}

static int ragged_plan(const boac_geom* classes, int n_classes, const boac_ragged_cand* cands, int B,
                       const int* config, RaggedPlan* pl) {
    if (!classes || n_classes < 1 || n_classes > kMaxRaggedClasses || !cands || B < 1) return BOAC_EINVAL;
    for (int c = 0; c < n_classes; ++c) {
        if (!geom_ok(&classes[c]) || classes[c].n_views % 2) return BOAC_EINVAL;
        pl->cls_count[c] = 0;
        pl->units[c] = pl->longest[c] = 0;
    }
    for (int b = 0; b < B; ++b) {
        const boac_ragged_cand& d = cands[b];
        if (d.cls < 0 || d.cls >= n_classes || d.K < 0 || d.mu_off < 0 || d.S_off < 0 || d.F_off < 0)
            return BOAC_EINVAL;
        pl->cls_count[d.cls]++;
        const long long len = d.K > 0 ? d.K : 1;
        pl->units[d.cls] += len;
        if (len > pl->longest[d.cls]) pl->longest[d.cls] = len;
    }
    size_t off = 256;
    for (int c = 0; c < n_classes; ++c) {
        if (!variant_table(classes[c].n)) return BOAC_EUNSUPPORTED;
        const int cfg = config ? config[c] : default_config(&classes[c], pl->cls_count[c]);
        pl->var[c] = get_variant(&classes[c], cfg);
        if (!pl->var[c]) return BOAC_EINVAL;
        const int cnt = pl->cls_count[c];
        pl->slots[c] = cnt ? split_holders(&classes[c], pl->var[c], cnt, pl->units[c] / cnt) : 0;
        if (cnt && pl->slots[c] <= 0) return BOAC_ECUDA;
    }
    ragged_share(classes, n_classes, pl);
    for (int c = 0; c < n_classes; ++c) {
        const int cnt = pl->cls_count[c];
        pl->desc_off[c] = off;
        off += align256(sizeof(RaggedDesc) * (size_t)cnt);
        pl->start_off[c] = off;
        off += align256(sizeof(long long) * ((size_t)cnt + 1));
        pl->layout_off[c] = off;
        off += cnt ? fused_layout(&classes[c], pl->var[c], pl->slots[c], cnt).total : 0;
    }
    pl->total = off;
    return BOAC_OK;
}

// The candidates in the order the kernels process them: by class, then by
// decreasing K.
static std::vector<int> ragged_order(const boac_ragged_cand* cands, int B) {
    std::vector<int> order((size_t)B);
    for (int b = 0; b < B; ++b) order[b] = b;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        if (cands[x].cls != cands[y].cls) return cands[x].cls < cands[y].cls;
        return cands[x].K > cands[y].K;
    });
    return order;
}

#ifdef BOAC_CHECKED
BOAC_FAULT_READER(bounds_faults_fused)
#endif

}  // namespace boac

using namespace boac;

extern "C" int boac_mlem(const boac_geom* g, const float* mu, const float* S, long long s_stride,
                         float* F, int K, int B, double* L, int include_lgamma, void* ws,
                         size_t ws_bytes, void* stream) {
    BOAC_RANGE("boac_mlem");
    if (!geom_ok(g) || !mu || !S || !F || B < 1 || K < 0 || s_stride < 0) return BOAC_EINVAL;
    if (g->n_views % 2) return BOAC_EINVAL;
    if (use_unfused(g, B))
        return mlem_unfused(g, mu, S, s_stride, F, K, B, L, include_lgamma, ws, ws_bytes, as_stream(stream));
    const FusedVariant* v = get_variant(g, default_config(g, B));
    if (!v) return BOAC_EUNSUPPORTED;
    const int slots = variant_holders(g, v, B);
    if (slots <= 0) return BOAC_ECUDA;
    if (!ws || ws_bytes < fused_layout(g, v, slots, B).total) return BOAC_EWORKSPACE;
    return launch_uniform(g, v, split_holders(g, v, B, K), mu, S, s_stride, F, K, B, L, include_lgamma,
                          static_cast<char*>(ws), as_stream(stream));
}

extern "C" long long boac_set_wait_cycles(long long cycles) {
    return g_wait_cycles.exchange(cycles > 0 ? cycles : kWaitCycles);
}

// Test hook of the bounded hand-over wait: the fused kernel of launch
// configuration `config` on exactly `holders` CTAs (or clusters), with the
// first part of candidate `withhold` keeping its flag to itself.
static int handover_plan(const boac_geom* g, int B, int K, int config, int holders, int withhold,
                         const FusedVariant** v, FusedLayout* l) {
    if (!geom_ok(g) || B < 1 || K < 0 || holders < 1 || holders > B || withhold < -1 || withhold >= B)
        return BOAC_EINVAL;
    *v = get_variant(g, config);
    if (!*v) return BOAC_EINVAL;
    if (variant_holders(g, *v, B) < holders) return BOAC_EUNSUPPORTED;  // must all be resident
    *l = fused_layout(g, *v, holders, B);
    return BOAC_OK;
}

extern "C" size_t boac_test_mlem_handover_bytes(const boac_geom* g, int B, int K, int config, int holders) {
    const FusedVariant* v;
    FusedLayout l;
    return handover_plan(g, B, K, config, holders, -1, &v, &l) == BOAC_OK ? l.total : 0;
}

extern "C" int boac_test_mlem_handover(const boac_geom* g, const float* mu, const float* S, float* F, int K,
                                       int B, double* L, int config, int holders, int withhold, void* ws,
                                       size_t ws_bytes, void* stream) {
    BOAC_RANGE("boac_test_mlem_handover");
    if (!mu || !S || !F || !L) return BOAC_EINVAL;
    const FusedVariant* v;
    FusedLayout l;
    const int s = handover_plan(g, B, K, config, holders, withhold, &v, &l);
    if (s != BOAC_OK) return s;
    if (!ws || ws_bytes < l.total) return BOAC_EWORKSPACE;
    char* base = static_cast<char*>(ws);
    cudaStream_t st = as_stream(stream);
    FusedArgs a = base_args(g, mu, S, 0, F, K, B, L, 0, base, l);
    a.withhold = withhold;
    const long long per = K > 0 ? K : 1, units = (long long)B * per;
    a.cap = split_cap(units, per, holders);
    const int grid = (int)((units + a.cap - 1) / a.cap);
    if (cudaMemsetAsync(base + l.status, 0, sizeof(int), st) != cudaSuccess ||
        cudaMemsetAsync(base + l.ready, 0, sizeof(int) * (size_t)B, st) != cudaSuccess)
        return launch_status();
    const int ps = v->prepare(&a, st);
    return ps == BOAC_OK ? v->launch(a, grid, st) : ps;
}

extern "C" int boac_workspace_status(const void* ws, size_t ws_bytes, int* status) {
    BOAC_RANGE("boac_workspace_status");
    if (!ws || ws_bytes < sizeof(int) || !status) return BOAC_EINVAL;
    if (cudaMemcpy(status, ws, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return launch_status();
    return BOAC_OK;
}

extern "C" size_t boac_mlem_ragged_workspace_bytes(const boac_geom* classes, int n_classes,
                                                   const boac_ragged_cand* cands, int B,
                                                   const int* config) {
    RaggedPlan pl;
    return ragged_plan(classes, n_classes, cands, B, config, &pl) == BOAC_OK ? pl.total : 0;
}

extern "C" int boac_mlem_ragged_prepare(const boac_geom* classes, int n_classes,
                                        const boac_ragged_cand* cands, int B, const int* config,
                                        void* ws, size_t ws_bytes, void* stream) {
    BOAC_RANGE("boac_mlem_ragged_prepare");
    RaggedPlan pl;
    int s = ragged_plan(classes, n_classes, cands, B, config, &pl);
    if (s != BOAC_OK) return s;
    if (!ws || ws_bytes < pl.total) return BOAC_EWORKSPACE;
    // Per-class records and unit offsets, copied from pageable host memory
    // (the copies are staged before this call returns).
    const std::vector<int> order = ragged_order(cands, B);
    std::vector<RaggedDesc> desc((size_t)B);
    std::vector<long long> start((size_t)B + n_classes);
    char* base = static_cast<char*>(ws);
    int first = 0;
    for (int c = 0; c < n_classes; ++c) {
        const int cnt = pl.cls_count[c];
        if (cnt == 0) continue;
        long long* js = start.data() + first + c;
        js[0] = 0;
        for (int i = 0; i < cnt; ++i) {
            const boac_ragged_cand& d = cands[order[first + i]];
            desc[first + i] = RaggedDesc{d.mu_off, d.S_off, d.F_off, d.K, order[first + i]};
            js[i + 1] = js[i] + (d.K > 0 ? d.K : 1);
        }
        if (cudaMemcpyAsync(base + pl.desc_off[c], desc.data() + first, sizeof(RaggedDesc) * cnt,
                            cudaMemcpyHostToDevice, as_stream(stream)) != cudaSuccess ||
            cudaMemcpyAsync(base + pl.start_off[c], js, sizeof(long long) * (cnt + 1),
                            cudaMemcpyHostToDevice, as_stream(stream)) != cudaSuccess)
            return launch_status();
        first += cnt;
    }
    return BOAC_OK;
}

extern "C" int boac_mlem_ragged_run(const boac_geom* classes, int n_classes,
                                    const boac_ragged_cand* cands, int B, const float* mu_pool,
                                    const float* S_pool, float* F_pool, double* L, int include_lgamma,
                                    const int* config, void* ws, size_t ws_bytes, void* stream) {
    BOAC_RANGE("boac_mlem_ragged_run");
    if (!mu_pool || !S_pool || !F_pool || !L) return BOAC_EINVAL;
    RaggedPlan pl;
    int s = ragged_plan(classes, n_classes, cands, B, config, &pl);
    if (s != BOAC_OK) return s;
    if (!ws || ws_bytes < pl.total) return BOAC_EWORKSPACE;
    char* base = static_cast<char*>(ws);
    cudaStream_t st = as_stream(stream);
    if (cudaMemsetAsync(base, 0, sizeof(int), st) != cudaSuccess) return launch_status();
    // What every class's kernel needs first, then the kernels, each free to
    // start beside the ones before it (but see RaggedPlan::alone): one after the other they take the sum
    // of the classes' longest chains (256 candidates of three sizes, 20 to 80
    // iterations: 57.0 ms, together 28.8).  The longest chain goes first, but
    // CTAs that share an SM last: on an empty GPU each would be given an SM of
    // its own and keep the larger CTAs off it.
    FusedArgs args[kMaxRaggedClasses];
    int grids[kMaxRaggedClasses], order[kMaxRaggedClasses], used = 0;
    for (int c = 0; c < n_classes; ++c) {
        const int cnt = pl.cls_count[c];
        if (cnt == 0) continue;
        int at = used++;
        auto before = [&](int x, int y) {
            if (pl.alone[x] != pl.alone[y]) return pl.alone[x];
            return pl.shares_sm[x] != pl.shares_sm[y] ? pl.shares_sm[y] : pl.chain[x] > pl.chain[y];
        };
        for (; at > 0 && before(c, order[at - 1]); --at) order[at] = order[at - 1];
        order[at] = c;
        const FusedLayout l = fused_layout(&classes[c], pl.var[c], pl.slots[c], cnt);
        char* cbase = base + pl.layout_off[c];
        FusedArgs a = base_args(&classes[c], mu_pool, S_pool, 0, F_pool, 0, cnt, L, include_lgamma, cbase, l);
        a.desc = reinterpret_cast<const RaggedDesc*>(base + pl.desc_off[c]);
        a.job_start = reinterpret_cast<const long long*>(base + pl.start_off[c]);
        a.status = reinterpret_cast<int*>(base);  // one status word for the call
        a.cap = split_cap(pl.units[c], pl.longest[c], pl.slots[c]);
        grids[c] = (int)((pl.units[c] + a.cap - 1) / a.cap);
        if (cudaMemsetAsync(cbase + l.ready, 0, sizeof(int) * ((size_t)cnt + 1), st) != cudaSuccess)
            return launch_status();
        s = pl.var[c]->prepare(&a, st);
        if (s != BOAC_OK) return s;
        args[c] = a;
    }
    for (int i = 0; i < used; ++i) {
        const int c = order[i];
        args[c].overlap = pl.alone[c] ? 0
                                      : (i + 1 < used ? FusedArgs::kTrigger : 0) |
                                            (i > 0 && !pl.alone[order[i - 1]] ? FusedArgs::kJoin : 0);
        s = pl.var[c]->launch(args[c], grids[c], st);
        if (s != BOAC_OK) return s;
    }
    return BOAC_OK;
}

extern "C" int boac_mlem_ragged(const boac_geom* classes, int n_classes, const boac_ragged_cand* cands,
                                int B, const float* mu_pool, const float* S_pool, float* F_pool,
                                double* L, int include_lgamma, const int* config, void* ws,
                                size_t ws_bytes, void* stream) {
    BOAC_RANGE("boac_mlem_ragged");
    if (!mu_pool || !S_pool || !F_pool || !L) return BOAC_EINVAL;
    int s = boac_mlem_ragged_prepare(classes, n_classes, cands, B, config, ws, ws_bytes, stream);
    if (s != BOAC_OK) return s;
    return boac_mlem_ragged_run(classes, n_classes, cands, B, mu_pool, S_pool, F_pool, L,
                                include_lgamma, config, ws, ws_bytes, stream);
}

// ---------------------------------------------------------------------------
// Allocation-free variant of boac_mlem.
//
// Some callers cannot allocate device memory at the moment they want a
// reconstruction: code running inside another framework's memory pool or
// allocator lock, a callback that must not call cudaMalloc (which can
// synchronise the device), or a host process that has no allocator of its
// own to hand the library a workspace.  boac_mlem_noalloc takes the fused
// kernel's scratch (per-CTA attenuation tables and sensitivity images) from
// a fixed array compiled into this library instead of from a caller
// workspace.  The array lives in device memory on every GPU that loads the
// library, for as long as the process runs.
namespace boac {

// Size of the built-in scratch: 64 MiB.
constexpr size_t kNoAllocScratchBytes = size_t(64) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// Device address of g_noalloc_scratch on the current device, looked up on
// every call: in host code the array's name stands for a host-side shadow,
// not device memory, so the kernel must be given the address
// cudaGetSymbolAddress returns.  Not caching it keeps the address right after
// a device reset or a re-created primary context (the module, and the array
// with it, may then sit elsewhere) and leaves no shared state between host
// threads; the lookup costs next to nothing beside an MLEM launch.
static void* noalloc_scratch_ptr() {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

// Largest number of resident CTA slots whose tables, sensitivity images and
// the candidates' hand-over flags fit the built-in scratch (0 if not even
// one slot does).
static int noalloc_slots(const boac_geom* g, const FusedVariant* v, int B) {
    int slots = variant_holders(g, v, B);
    while (slots > 0 && fused_layout(g, v, slots, B).total > kNoAllocScratchBytes) --slots;
    return slots;
}

}  // namespace boac

extern "C" int boac_mlem_noalloc(const boac_geom* g, const float* mu, const float* S,
                                 long long s_stride, float* F, int K, int B, double* L,
                                 int include_lgamma, void* stream) {
    BOAC_RANGE("boac_mlem_noalloc");
    // L is required: the status word of the bounded hand-over wait lives in
    // the built-in array, out of the caller's reach, so a candidate that gave
    // up shows only as a NaN score.
    if (!geom_ok(g) || !mu || !S || !F || !L || B < 1 || K < 0 || s_stride < 0) return BOAC_EINVAL;
    if (g->n_views % 2) return BOAC_EINVAL;
    // the one-CTA kernel: its per-CTA scratch is the smallest
    const FusedVariant* v = get_variant(g, single_cta_config(g));
    if (!v) return BOAC_EUNSUPPORTED;
    if (variant_holders(g, v, B) <= 0) return BOAC_ECUDA;
    int slots = noalloc_slots(g, v, B);
    if (slots <= 0) return BOAC_EWORKSPACE;  // one candidate's scratch exceeds 64 MiB
    slots = std::min(slots, split_holders(g, v, B, K));
    void* scratch = noalloc_scratch_ptr();
    if (!scratch) return BOAC_ECUDA;
    // The kernel writes every table entry and sensitivity pixel of a slot
    // before reading it; the status word and the candidates' hand-over flags
    // must start at zero and are cleared here, on the caller's stream.
    return launch_uniform(g, v, slots, mu, S, s_stride, F, K, B, L, include_lgamma,
                          static_cast<char*>(scratch), as_stream(stream));
}
