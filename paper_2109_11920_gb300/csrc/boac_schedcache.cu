// boac_schedcache.cu -- the scatter schedules of the geometries in use, kept
// on the device across calls.
//
// A schedule (boac_sched.cuh) depends on the image size, the view count,
// the number of sample grids and the pitch of the kernel's sample buffer
// only; building one takes about 0.2 ms at 128 x 128 / 120 views, a tenth of
// a 16-candidate call and more than the operators take.  The library keeps
// schedules in an arena of static device memory, each with a device-side tag
// naming the geometry it holds.  Static device memory is zero when the module
// is loaded, so after a device reset every tag is empty again and the next
// call rebuilds.  The host gives a geometry the next stretch of the arena, of
// its schedule's size, the first time it meets it on a device and never
// reassigns it, so no call can read a schedule that another call is
// replacing.  Every call launches the builder on its stretch, whose CTAs
// return at once when the tag already names the geometry, then a one-thread
// kernel that writes the tag (after the build, in stream order).  Two calls
// on different streams that both find the tag empty build the schedule at the
// same time and store the same bytes (scatter_schedule_kernel), so neither a
// kernel that reads it meanwhile nor a later one sees anything else.
//
// A geometry that finds no room, or whose schedule is larger than 4 MiB, has
// no kept schedule: it is built into the caller's workspace on every call, or,
// for the callers that give none because they scatter a few grids per call,
// not at all.  (Eight fixed slots of 4 MiB held a program of nine geometries
// no more: back-projections of one to eight 128 x 128 images then took 183 to
// 305 us, most of it the build.)
#include <cuda_runtime.h>

#include <mutex>

#include "boac_internal.h"
#include "boac_sched.cuh"

namespace boac {

namespace {

constexpr int kSchedCacheSlots = 256;
constexpr size_t kSchedArenaEntries = ((size_t)64 << 20) / sizeof(unsigned short);  // 60 of 1.1 MB (128 x 128, 120 views)
constexpr size_t kSchedMaxBytes = (size_t)4 << 20;  // the largest schedule kept
constexpr int kSchedCacheDevices = 64;

struct SlotGeom {
    int n, V, ngrid, wp;  // n == 0: free
    size_t at;            // its first entry in the arena
};

std::mutex g_sched_mu;
SlotGeom g_sched_geom[kSchedCacheDevices][kSchedCacheSlots];

}  // namespace

static __device__ __align__(256) unsigned short g_sched_cache[kSchedArenaEntries];
static __device__ unsigned long long g_sched_tag[kSchedCacheSlots];

__global__ void sched_tag_kernel(unsigned long long* tag, unsigned long long v) { *tag = v; }

// The slot of (n, V, ngrid, wp) on device dev, assigning the next one and the
// arena's next entries (*at); -1 if either runs out.
static int sched_slot_of(int dev, int n, int V, int ngrid, int wp, size_t* at) {
    const size_t need = sched_bytes(n, ngrid) / sizeof(unsigned short);  // a multiple of 256 bytes
    std::lock_guard<std::mutex> lock(g_sched_mu);
    size_t used = 0;
    // slots are filled in order and never freed, so no match follows a free slot
    for (int i = 0; i < kSchedCacheSlots; ++i) {
        SlotGeom& s = g_sched_geom[dev][i];
        if (s.n == 0) {
            if (need > kSchedArenaEntries - used) return -1;
            s = SlotGeom{n, V, ngrid, wp, used};
        }
        if (s.n == n && s.V == V && s.ngrid == ngrid && s.wp == wp) {
            *at = s.at;
            return i;
        }
        used = s.at + sched_bytes(s.n, s.ngrid) / sizeof(unsigned short);
    }
    return -1;
}

const unsigned short* sched_prepare(int n, int V, int ngrid, int wp, unsigned short* ws, cudaStream_t st,
                                    int* status) {
    int dev = -1, slot = -1;
    size_t at = 0;
    if (sched_bytes(n, ngrid) <= kSchedMaxBytes && cudaGetDevice(&dev) == cudaSuccess && dev >= 0 &&
        dev < kSchedCacheDevices)
        slot = sched_slot_of(dev, n, V, ngrid, wp, &at);
    void* base = nullptr;
    void* tags = nullptr;
    if (slot >= 0 && (cudaGetSymbolAddress(&base, g_sched_cache) != cudaSuccess ||
                      cudaGetSymbolAddress(&tags, g_sched_tag) != cudaSuccess || !base || !tags)) {
        cudaGetLastError();  // not a sticky error: as without a slot
        slot = -1;
    }
    if (slot < 0) {
        *status = ws ? sched_launch(n, V, ngrid, wp, ws, st) : BOAC_OK;
        return ws;
    }
    unsigned short* sched = static_cast<unsigned short*>(base) + at;
    unsigned long long* tag = static_cast<unsigned long long*>(tags) + slot;
    const unsigned long long want = sched_tag_value(n, V, ngrid, wp);
    *status = sched_launch(n, V, ngrid, wp, sched, st, tag, want);
    if (*status != BOAC_OK) return sched;
    sched_tag_kernel<<<1, 1, 0, st>>>(tag, want);
    *status = launch_status();
    return sched;
}

}  // namespace boac

using namespace boac;

// Test hook: the schedule that the library builds for g and a sample buffer of
// pitch n + pad, into the caller's memory.
extern "C" size_t boac_test_schedule_bytes(const boac_geom* g, int views_per_grid) {
    if (!geom_ok(g) || (g->n != 64 && g->n != 96 && g->n != 128)) return 0;
    if ((views_per_grid != 2 && views_per_grid != 4) || g->n_views % views_per_grid) return 0;
    return sched_bytes(g->n, g->n_views / views_per_grid);
}

extern "C" int boac_test_schedule(const boac_geom* g, int views_per_grid, int pad, void* sched, size_t bytes,
                                  void* stream) {
    const size_t need = boac_test_schedule_bytes(g, views_per_grid);
    if (need == 0 || !sched || (pad != 1 && pad != 4)) return BOAC_EINVAL;
    if (bytes < need) return BOAC_EWORKSPACE;
    return sched_launch(g->n, g->n_views, g->n_views / views_per_grid, g->n + pad, static_cast<unsigned short*>(sched),
                        as_stream(stream));
}
