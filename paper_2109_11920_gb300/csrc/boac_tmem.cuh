// boac_tmem.cuh -- tensor memory as a per-thread stash.
//
// An SM's 256 KB of tensor memory (128 lanes x 512 columns of 32 bits) is
// idle in kernels that issue no matrix instructions.  The fused kernels keep
// the attenuation factors of the grid in flight there: written by the
// forward passes, read back by the back-projection weights of the same
// thread, so neither the exponents are read from L2 a second time nor their
// exponentials taken again.  tcgen05.st / ld move 32 lanes x k columns per
// warp at full register width; a warp reaches the 32 lanes of its quarter
// (warp index mod 4), and the warps of one quarter split the columns.
#pragma once

#include <cuda_runtime.h>

namespace boac {

constexpr int kTmemColumns = 512;  // of an SM

// Columns to allocate for a CTA of `warps` warps with `per_thread` floats per
// thread: a power of two, at least 32.
__host__ __device__ constexpr int tmem_columns(int warps, int per_thread) {
    const int need = (warps + 3) / 4 * per_thread;
    int c = 32;
    while (c < need) c *= 2;
    return c;
}

// Allocates COLS columns for the CTA (one whole warp calls it; blocks while
// another CTA of the SM holds them) and leaves the address in *smem_addr.
template <int COLS>
__device__ __forceinline__ void tmem_alloc(unsigned* smem_addr) {
    static_assert(COLS >= 32 && COLS <= kTmemColumns && (COLS & (COLS - 1)) == 0, "tensor-memory columns");
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem_addr);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s), "n"(COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <int COLS>
__device__ __forceinline__ void tmem_free(unsigned addr) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "n"(COLS) : "memory");
}

// Address of this thread's columns in a CTA-wide allocation at `base`.
__device__ __forceinline__ unsigned tmem_mine(unsigned base, int tid, int per_thread) {
    const unsigned warp = (unsigned)tid >> 5;
    return base + ((warp & 3u) << 21) + (warp >> 2) * (unsigned)per_thread;  // lane 32 (warp % 4) in bits 16..
}

// Eight floats per thread to / from consecutive columns.  All lanes of the
// warp take part.  Stores are complete after tmem_wait_st, loads after
// tmem_wait_ld.
__device__ __forceinline__ void tmem_st8(unsigned addr, const float (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "f"(v[0]),
                 "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_ld8(unsigned addr, float (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(addr)
                 : "memory");
}
// Four floats, likewise.
__device__ __forceinline__ void tmem_st4(unsigned addr, float4 v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld4(unsigned addr, float (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// The loaded values are used only after the wait: they pass through it.
__device__ __forceinline__ void tmem_wait_ld(float (&a)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7])
                 :
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_ld(float (&a)[4]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3])
                 :
                 : "memory");
}

}  // namespace boac
