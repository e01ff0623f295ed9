// Shared by the kernels that sum ring pairs on tcgen05 with two-part FP16 operands
// (conv_belt_tc.cu, conv_cap_tc.cu): descriptors, the FP16 MMA, and bounded waits.
#pragma once

#include <cstdint>
#include <cuda_fp16.h>

#include "ksc_tc.cuh"

namespace ksc {
constexpr int kMaxDynSmem = 226 * 1024;  // of the split kernels, beside 1 kB of static
namespace tc {

constexpr int kXExp = 14;           // a tile's largest |m| is scaled into [2^14, 2^15)
constexpr uint32_t kRangeExp = 14;  // a block may lie this many powers of two below it

// Two FP32 values in one register pair.
__device__ __forceinline__ uint64_t pack2(uint32_t a, uint32_t b) {
    return (uint64_t)b << 32 | a;
}
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    return pack2(__float_as_uint(a), __float_as_uint(b));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// K-major, no swizzle: 8-row x 16-byte core matrices; lead = bytes between core matrices
// adjacent in K, stride = bytes between groups of eight rows.
__device__ __forceinline__ uint64_t desc(uint32_t addr, uint32_t lead, uint32_t stride) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | (uint64_t)((lead >> 4) & 0x3FFF) << 16 |
           (uint64_t)((stride >> 4) & 0x3FFF) << 32 | (uint64_t)1 << 46;
}

// FP16 operands, FP32 accumulator, both K-major.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc,
                                        uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(da), "l"(db), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t *v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t *v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
        : "memory");
}

// Waits for this thread's tensor-memory loads, the last of them into v: a use of v cannot be
// moved before the wait (the load's asm statement alone would allow it).
template <int N>
__device__ __forceinline__ void loaded(uint32_t (&v)[N]) {
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+r"(v[i]));
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}

// Bounded wait that also ends when another warp of the CTA has given up.
__device__ __forceinline__ bool wait_or_abort(uint64_t *bar, uint32_t parity,
                                              volatile int *abort) {
    for (int i = 0; i < 64; ++i) {
        if (mbar_wait(bar, parity, kMaxWait / 64)) return true;
        if (*abort) break;
    }
    *abort = 1;
    return false;
}

// One input ring as seen by a tile: Delta in [-w, w] (the whole ring where that exceeds
// it) on a grid of kChunk positions; the 16-position steps [s0, s1) are in use.  Position
// j stands for Delta = d0 + j - i, i = 0..7.  The grid is laid so that |Delta| <= 3, where a
// kernel of the map's resolution is largest, falls into one step for every i: step
// kChunk / 32 of chunk `mid`.
struct Window {
    int d0, s0, s1, mid;
};
template <int kChunk>
__host__ __device__ __forceinline__ Window tile_window(int w, int L) {
    const bool whole = 2 * w + 1 >= L;  // the whole ring, each pixel once
    const int lo = whole ? -(L / 2) : -w, hi = whole ? lo + L - 1 : w;
    Window g;
    g.mid = (unsigned)(-lo - kChunk / 2 - 3 + kChunk - 1) / kChunk;  // chunks left of it
    g.d0 = -(g.mid * kChunk + kChunk / 2 + 3);
    g.s0 = (unsigned)(lo - g.d0) / 16;          // first j of any use: Delta = lo at i = 0
    g.s1 = (unsigned)(hi - g.d0 + 7) / 16 + 1;  // last: Delta = hi at i = 7
    return g;
}
// The chunks of a window in order of work: the closest approach's last.
__host__ __device__ __forceinline__ int chunk_of(int cc, int c_hi, int mid) {
    return cc == c_hi ? mid : (cc >= mid ? cc + 1 : cc);
}

} // namespace tc
} // namespace ksc
