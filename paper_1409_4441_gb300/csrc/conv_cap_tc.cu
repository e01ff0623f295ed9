// Real-space convolution, ring pairs with a polar-cap ring, on the tcgen05 tensor cores.
//
// For output ring r (L pixels) and input ring q (L' pixels), output pixel k lies at
// s_k = n_k + f_k in units of q's pixels, n_k whole, f_k = rem_k / (2 L) in [-1/2, 1/2),
// and the weight of input pixel n_k - j is W(f_k + j), W smooth in its argument as far as
// the cut.  On each unit cell W is a polynomial of degree 8,
//
//   W(f + j) = sum_p c_p[j] f^p,      so      out_k += sum_p f_k^p y_p[n_k],
//   y_p[n] = sum_j c_p[j] m_q[n - j]:
//
// nine Toeplitz products on the input ring's own grid, whose weights no longer depend on
// the output pixel, and one short polynomial per output pixel and input ring, where the
// gather (conv_sym.cu) evaluates a weight per class and input pixel.  With l_max = 2 nside
// the degree-8 interpolant is within 2e-9 of the kernel's peak (4e-9 at l_max = 3 nside); c_p
// falls off as the derivatives do: for a beam of three pixels at l_max = 2 nside c_6 / 2^6 is
// 2^-12.7 of the peak, c_8 / 2^8 about 2e-6.  The host bounds both, and a split beyond the
// bounds (2.4 pixels with l_max = 3 nside, a kernel that peaks past its cut) has no cap stage.
//
// A CTA owns two adjacent rings and their southern mirrors (which share every weight) over
// one sector of longitude.  Per input ring:
//
//   D_h[m, (R, p, i)] = sum_x A_h[m, x] B[(R, p, i), x],   A_h[m, x] = m_q[n0 + d0 + x + 8 m],
//   D_h[m, (R, p, i)] = y_p[n0 + 8 m + i] of ring R on hemisphere h:
//
// M = 128 rows are groups of eight input positions, N = 2 rings x 9 powers x 8 offsets.
// As in the belt kernel neither operand is a full matrix: A's rows are 16 bytes apart in
// the staged ring segment, B's eight rows of one (R, p) are one sequence shifted by i.
//
// Precision as in conv_belt_tc.cu: two FP16 parts of map and weights (23 bits of the 24), w_h
// m_h in one FP32 accumulator, w_h m_l + w_l m_h in a second one, with w_l m_l and a third
// part of c_0 times m_h (near rings) in the step of the closest approach, where the weights are large; for
// p = 6, 7, 8 (coefficients below 2^-10.5 of the peak, which the host checks) w_h m_h alone; far chunks first.  The polynomial and the
// pixels of the two cells that the cut divides (at most one pixel a side, tested with the
// exact integers) are in FP32; the rounding errors of a ring's last sum and of the sum over
// input rings are carried along.  Error rms of cap pixels against 64 bits, over the output
// rms, white noise, 1e-7: gather / this kernel without the third part and with a plain Kahan
// sum / now: nside 512, 480': 0.84 / 1.01 / 0.82; 2048, 240': 0.85 / 1.08 / 0.86; 2048, 120':
// 0.87 / 0.94 / 0.78 (stage at 2048, 240': 105.8 -> 107.4 ms).
//
// The coefficients c_p[j] depend on the ring pair alone and are laid out once per split
// (cap_coef_kernel: 20 ms and 2.4 GB at nside 2048 with a 240' cut); evaluated inside
// this kernel they took half of its instructions, for every sector again.
//
// Ring pairs near the poles whose window is the whole ring or close to it, and input rings of
// fewer than 32 pixels, go through cap_direct_kernel: every weight from the chord, each for
// the four quarter turns and the two hemispheres.
//
// A pair of rings whose input rings span more than 2^14 in largest magnitudes (all-zero
// blocks aside) or hold an infinity or NaN is flagged and left to conv_sym_kernel.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "ksc_device.cuh"
#include "ksc_internal.h"
#include "ksc_tc_split.cuh"

namespace ksc {
namespace {

constexpr int kEpi = 256;          // threads that sum up: a warp per ring and 256 positions
constexpr int kBuild = 256;        // threads that stage and lay out the operands
constexpr int kT = kEpi + kBuild;
constexpr int kThreads = kT + 128; // and four warps that issue the MMAs
constexpr int kP = 9;              // polynomial coefficients
constexpr int kP3 = 6;             // of which three-product ones
constexpr int kG = 2 * kP;         // (ring, power) groups of eight B rows
constexpr int kG3 = 2 * kP3;
constexpr int kN = 8 * kG;         // columns of an accumulator (144)
constexpr int kN3 = 8 * kG3;       // columns of the three-product groups (96)
constexpr int kHemi = kN + kN3;    // columns of a hemisphere: leading and small products
constexpr int kChunk = 32;         // window positions per B stage
constexpr int kSteps = kChunk / 16;
// K-adjacent core matrices of B lie 144 bytes apart, so that eight lanes that each write a
// row of their own core matrix reach all banks (at 128 bytes they share four)
constexpr int kLead = 144;
constexpr int kGroupBytes = kChunk / 8 * kLead;
constexpr int kStageBytes = (kG + kG3) * kGroupBytes;  // high parts, then low parts
constexpr int kStages = 3;
constexpr int kSpan = 1024;        // positions of a tile (128 rows of eight)
constexpr int kOut = 9;            // outputs a lane carries at a time
constexpr int kTurn = 32 * 10;     // float2 of a warp's turning buffer (10 per 8 positions)
// Third parts of c_0: the cells that the closest approach's step reaches (|Delta| <= 12), as
// two groups of two core matrices a ring pair
constexpr int kE = 13;
constexpr int kEBytes = 2 * 2 * kLead;
constexpr int kNear = 12;  // input rings this near the output rings have them
constexpr int kXr = 7;             // staged elements of a builder thread and hemisphere

using tc::Window;
using tc::add2;
using tc::fma2;
using tc::pack2;
__host__ __device__ __forceinline__ Window window_of(int w, int L) {
    return tc::tile_window<kChunk>(w, L);
}

// Interpolation nodes: 0 and the other Chebyshev nodes of [-1/2, 1/2] at nine points, to 2^-10 (so
// that j + g is exact in FP32).
__host__ __device__ constexpr float node(int s) {
    return s == 0 ? 0.0f : s == 1 ? 175.0f / 1024 : s == 2 ? 329.0f / 1024
           : s == 3 ? 443.0f / 1024 : 504.0f / 1024;
}


// a + b and its rounding error.
__device__ __forceinline__ uint64_t two_sum2(uint64_t a, uint64_t b, uint64_t *err) {
    const uint64_t m1 = pack2(-1.0f, -1.0f);
    const uint64_t s = add2(a, b), bb = fma2(a, m1, s);
    *err = add2(fma2(fma2(bb, m1, s), m1, a), fma2(bb, m1, b));
    return s;
}

// Group of (ring R, power p): three-product groups first, the
// two rings' c_0 side by side.
__device__ __forceinline__ int group_of(int R, int p) { return 2 * p + R; }

// Wait that gives up at once when the CTA has (builder warps meet at barriers: none of
// them may leave the loop).
__device__ __forceinline__ void wait_all(uint64_t *bar, uint32_t parity, volatile int *abort) {
    if (!*abort) tc::wait_or_abort(bar, parity, abort);
    __syncwarp();
}

__device__ __forceinline__ void copy16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::saddr(dst)), "l"(src) : "memory");
}

struct QInfo {      // an input ring as the tile sees it (shorts: the cut's width is bound by their memory)
    uint32_t off[2];  // first coefficient word of each ring, in units of four
    int start;      // first pixel of the ring
    short n0;       // first position (input pixel) of row 0
    short eR[2];    // rem <= eR: the right edge cell's pixel lies within the cut
    short a;        // ring pixel of element 0 of the staged segments
    short len, phase;  // of the input ring
    short n_e;      // elements staged
    short base;     // d0 + 16 s0: Delta of element 0 at offset i = 0
    short jE[2];    // edge cell of each ring (-1: no pixel within the cut)
    short s0, s1, mid;  // window steps and the chunk of the closest approach
    unsigned short c[2];  // constants taken off the ring and its mirror, BF16 numbers
};

// Words of a ring pair's coefficients: [cell][power] in two parts, then the third parts of c_0
// in the first kE cells; rounded up to 16 bytes.
__host__ __device__ __forceinline__ int coef_words(int jE) {
    return (kP * (jE + 1) + (kE + 1) / 2 + 3) & ~3;
}
__device__ __forceinline__ const __half *third_parts(const uint32_t *coef, int jE) {
    return reinterpret_cast<const __half *>(coef + kP * (jE + 1));
}

// grid.x runs over tiles {rings - 1 << 16 | first ring, sectors << 16 | sector}, grid.y over
// maps.  Eight builder warps
// stage ring n + 1 while the tensor cores work on ring n and eight summing warps on ring
// n - 1 (their accumulators are the same: a summing warp reads them power by power and
// gives them back with d_free before it adds up).
//
// A summing warp owns ring R and 256 positions.  Its lanes take consecutive outputs; the
// accumulators come in rows of eight positions a lane, so each power of both hemispheres
// is turned in shared memory (as (north, south) pairs, which the polynomial, the edge
// pixels and the sums keep as FP32 pairs).
__global__ void __launch_bounds__(kThreads, 1)
conv_cap_tc_kernel(const ConvPlan P, const CapTc C, const int2 *__restrict__ tiles,
                   const MapSet maps,
                   int belt_split, int band_lo, int band_hi, const uint2 *__restrict__ ring_range,
                   int *__restrict__ flags, int back, int *__restrict__ err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    // B stages | third parts of c_0 [buffer] | map segments [h][buffer][part] | turning buffers | totals (north, south:
    // sums, compensations) [ring] | the segments as they are, (north, south) [buffer] |
    // coefficients as stored [buffer] | coefficient sequences | input rings
    const int xc = C.span + C.wpos;
    // words of one coefficient sequence, two FP16 elements each; 16-byte rows, and 20 words
    // more than a multiple of 32 so that the groups start in different banks
    const int w_cap = ((C.wpos / 2 + 8 + 11) & ~31) + 20;
    const int k_cap = 2 * coef_words(C.jcap - 1);
    unsigned char *sB = smem;
    unsigned char *sE = smem + kStages * kStageBytes;
    __half *sX = reinterpret_cast<__half *>(sE + 2 * kEBytes);
    float2 *sY = reinterpret_cast<float2 *>(sX + 8 * xc);
    float4 *sT = reinterpret_cast<float4 *>(sY + kEpi / 32 * kTurn);
    float2 *sF = reinterpret_cast<float2 *>(sT + 2 * C.tcap);
    uint32_t *sK = reinterpret_cast<uint32_t *>(sF + 2 * xc);
    uint32_t *sC = sK + 2 * k_cap;
    QInfo *sQ = reinterpret_cast<QInfo *>(sC + 2 * (kG + kG3) * w_cap);
    __shared__ __align__(8) uint64_t b_full[kStages], b_free[kStages], d_done, d_free[2], e_ready[2],
        s_drain[4];
    __shared__ uint32_t tmem_base, s_max, s_min;
    __shared__ int s_abort, s_lo, s_hi, s_bad, s_shift;
    __shared__ float s_edge[2][2][kP + 3], s_sum[2][2][kP];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int2 tile = tiles[back ? gridDim.x - 1 - blockIdx.x : blockIdx.x];
    const int r0 = tile.x & 0xffff, n_r = (tile.x >> 16) + 1;
    const int sector = tile.y & 0xffff, n_sec = tile.y >> 16;
    const bool add = belt_split && r0 >= P.belt_lo;
    const float *__restrict__ m = maps.input(blockIdx.y);
    float *__restrict__ o = maps.output(blockIdx.y);
    const uint2 *rr = ring_range + (long long)blockIdx.y * P.nrings;
    const DevRing Ra = P.d_rings[r0], Rb = P.d_rings[r0 + n_r - 1];
    const int L0 = Ra.len, L1 = Rb.len;
    auto sec_lo = [&](int L, int s) { return (int)(((long long)s * L + n_sec - 1) / n_sec); };
    const int k_lo0 = sec_lo(L0, sector), k_hi0 = sec_lo(L0, sector + 1) - 1;
    const int k_lo1 = sec_lo(L1, sector), k_hi1 = n_r == 2 ? sec_lo(L1, sector + 1) - 1 : k_lo1 - 1;

    if (tid == 0) {
        s_max = 0u;
        s_min = 0xffffffffu;
        s_abort = s_bad = s_shift = 0;
        s_lo = min(P.d_range[r0].x, P.d_range[r0 + n_r - 1].x);
        s_hi = max(P.d_range[r0].y, P.d_range[r0 + n_r - 1].y);
        for (int b = 0; b < kStages; ++b) {
            tc::mbar_init(&b_full[b], kBuild / 32);
            tc::mbar_init(&b_free[b], 4);
        }
        tc::mbar_init(&d_done, 4);
        for (int b = 0; b < 4; ++b) tc::mbar_init(&s_drain[b], 1);
        for (int b = 0; b < 2; ++b) {  // ring n uses the one of its parity
            tc::mbar_init(&d_free[b], kEpi / 32);
            tc::mbar_init(&e_ready[b], kBuild / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int q_lo = s_lo, nq = s_hi - s_lo + 1;
    // ---- the input rings as the tile sees them, and the range of their values
    uint32_t vmax = 0u, vmin = 0xffffffffu;
    for (int qi = tid; qi < nq; qi += kThreads) {
        const int q = q_lo + qi;
        const DevRing Q = P.d_rings[q];
        QInfo g;
        g.jE[0] = g.jE[1] = -1;
        g.eR[0] = g.eR[1] = 0;
        g.off[0] = g.off[1] = 0u;
        g.c[0] = g.c[1] = 0;
        const bool skip = add && q >= P.belt_lo && q <= P.belt_hi;
        for (int R = 0; R < n_r && !skip; ++R) {
            const int2 rg = P.d_range[r0 + R];
            if (q < rg.x || q > rg.y) continue;
            const int ip = P.d_pair_base[r0 + R] + q - rg.x;
            const int ncut = C.d_ncut[ip], L = R ? L1 : L0;
            if (ncut < 0) continue;
            g.jE[R] = ncut >= L ? (short)((ncut - L) / (2 * L) + 1) : 0;
            g.eR[R] = (short)(ncut - 2 * L * g.jE[R]);
            g.off[R] = C.d_coef_off[ip];
        }
        const int w = max((int)g.jE[0], (int)g.jE[1]);
        // positions of the sector's first and last outputs
        auto pos = [&](int k, int t, int L) {
            return (int)((unsigned)((2 * k + t) * Q.len + (1 - Q.phase) * L) / (unsigned)(2 * L));
        };
        int lo = 0x7fffffff, hi = -1;
        if (k_hi0 >= k_lo0) {
            lo = pos(k_lo0, Ra.phase, L0);
            hi = pos(k_hi0, Ra.phase, L0);
        }
        if (k_hi1 >= k_lo1) {
            lo = min(lo, pos(k_lo1, Rb.phase, L1));
            hi = max(hi, pos(k_hi1, Rb.phase, L1));
        }
        g.n0 = (short)lo;
        g.len = (short)Q.len;
        g.phase = (short)Q.phase;
        g.start = Q.start;
        if (w >= 0) {
            const Window v = window_of(w, Q.len);
            g.s0 = (short)v.s0;
            g.s1 = (short)v.s1;
            g.mid = (short)v.mid;
            g.base = (short)(v.d0 + 16 * v.s0);
            g.n_e = (short)(((hi - lo + 8) & ~7) + 16 * (v.s1 - v.s0));
            const int a = (lo + g.base) % Q.len;
            g.a = (short)(a < 0 ? a + Q.len : a);
            // sized by the host for every tile: never expected
            if (16 * (v.s1 - v.s0) > C.wpos || w + 1 > C.jcap || hi - lo + 1 > C.span ||
                g.n_e > kXr * kBuild || hi < lo || 2 * w + 1 > Q.len)
                s_bad = 1;
            for (int h = 0; h < 2; ++h) {
                const uint2 e = rr[h ? P.nrings - 1 - q : q];
                vmax = max(vmax, e.x);
                vmin = min(vmin, e.y);
                // blocks all within a factor of four of the largest: a constant may be taken off
                g.c[h] = e.x != 0u && (e.x >> 23) - (e.y >> 23) <= 1u;
            }
        }
        if (qi < C.nq) sQ[qi] = g;
        else s_bad = 1;
    }
    vmax = __reduce_max_sync(~0u, vmax);
    vmin = __reduce_min_sync(~0u, vmin);
    if (lane == 0) {
        atomicMax(&s_max, vmax);
        atomicMin(&s_min, vmin);
    }
    if (tid == 0 && max(k_hi0 - k_lo0, k_hi1 - k_lo1) + 1 > C.tcap) s_bad = 1;
    for (int e = tid; e < 2 * C.tcap; e += kThreads) sT[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (warp == kT / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         tc::saddr(&tmem_base)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_base;
    const uint32_t emax = s_max >> 23, emin = s_min >> 23;  // biased exponents
    const bool zero = s_max == 0u;
    const bool flag = !zero && (emax >= 255u || emax < 48u || emax > 206u || emin == 0u ||
                                emax - emin > tc::kRangeExp);
    if (tid == 0) {
        if (flag) {
            int *f = flags + (long long)blockIdx.y * (P.nrings + 1);
            f[r0] = 1;
            f[r0 + n_r - 1] = 1;
            f[P.nrings] = 1;
        }
        if (s_bad) atomicExch(err, KSC_ERR_DEVICE_BOUNDS);
    }
    // A constant taken off an input ring whose blocks are all within a factor of four of its
    // largest: near the mean of 128 of its pixels, a multiple of 2^-3 of the largest value's
    // power of two, where it is at least two of them (not for maps about zero).  The MMAs' cuts are toward zero and add up
    // where all products have one sign; the sums of the weights put the constant back.
    if (!zero && !flag && !s_bad) {
        for (int i = warp; i < 2 * nq; i += kThreads / 32) {
            QInfo &g = sQ[i >> 1];
            const int h = i & 1;
            if (!g.c[h]) continue;
            const uint32_t top = rr[h ? P.nrings - 1 - (q_lo + (i >> 1)) : q_lo + (i >> 1)].x;
            float v = 0.0f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                int k = g.a + (4 * lane + j) * g.n_e / 128;
                while (k >= g.len) k -= g.len;
                v += __ldg(m + (h ? P.npix - g.start - g.len : g.start) + k);
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(~0u, v, s);
            const float quantum = __uint_as_float(((top >> 23) - 3u) << 23);
            v = rintf(v * (1.0f / 128.0f) / quantum) * quantum;
            if (fabsf(v) < 2.0f * quantum) v = 0.0f;
            if (lane == 0) {
                g.c[h] = (unsigned short)(__float_as_uint(v + 0.0f) >> 16);  // (five digits: exact)
                if (v != 0.0f) s_shift = 1;
            }
        }
    }
    __syncthreads();
    const uint32_t ex = emax + (s_shift ? 1u : 0u);  // |m - c| may reach twice the largest |m|
    const float xscale = zero || flag ? 1.0f : __uint_as_float((127u + tc::kXExp + 127u - ex) << 23);
    const float xunscale = zero || flag ? 1.0f : __uint_as_float((ex - tc::kXExp) << 23);
    auto shift_of = [&](const QInfo &g, int h) {  // scaled
        return __uint_as_float((uint32_t)g.c[h] << 16) * xscale;
    };
    bool drained = true;
    // hemispheres with an output ring in the band; the other one's products are left out (its
    // accumulators hold anything, and nothing of them is written; the 1023 rings of the
    // northern cap at nside 2048, 120': 25.0 -> 23.4 ms)
    const bool band_n = r0 <= band_hi && r0 + n_r - 1 >= band_lo;
    const bool band_s = P.nrings - r0 - n_r <= band_hi && P.nrings - 1 - r0 >= band_lo;

    if (flag || s_bad) {
        // left to the gather (or never expected)
    } else if (warp >= kT / 32) {
        // ---- the issuing warps: one per hemisphere and accumulator (an MMA takes its
        // thread about as long to issue as 80 columns take to compute)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
        if (lane == 0) {
            const int h = warp & 1;
            const bool small = warp & 2;  // the small products' accumulator, else the leading ones'
            const uint32_t idesc = small ? tc::idesc_f16(128, kN3) : tc::idesc_f16(128, kN);
            const uint32_t d = tmem + h * kHemi + (small ? kN : 0);
            const uint64_t b_base = tc::desc(tc::saddr(sB), kLead, kGroupBytes);
            const uint64_t a_base = tc::desc(tc::saddr(sX) + h * 8 * xc, 16, 128);
            const uint64_t e_base = tc::desc(tc::saddr(sE), kLead, 2 * kLead);
            const uint32_t a_l = (uint32_t)(2 * xc) >> 4, b_l = (kG * kGroupBytes) >> 4;
            uint32_t n = 0, n_chunks = 0, st = 0, ph = 0;
            bool ok = true;
            for (int qi = 0; qi < nq && ok; ++qi) {
                const QInfo &g = sQ[qi];
                if (max((int)g.jE[0], (int)g.jE[1]) < 0) continue;
                const int s0 = g.s0, s1 = g.s1, mid = g.mid;
                const int c_lo = s0 / kSteps, c_hi = (s1 - 1) / kSteps;
                const uint64_t da0 = a_base + (n & 1u) * ((4 * xc) >> 4);
                if (n > 0 && !tc::wait_or_abort(&d_free[(n - 1u) & 1u], ((n - 1u) >> 1) & 1u, &s_abort))
                    break;
                uint32_t acc = 0u;
                for (int cc = c_lo; cc <= c_hi; ++cc, ++n_chunks) {
                    const int c = tc::chunk_of(cc, c_hi, mid);
                    if (!tc::wait_or_abort(&b_full[st], ph, &s_abort)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    const int t0 = max(s0, kSteps * c), t1 = min(s1, kSteps * c + kSteps);
                    // descriptors of step t0; a step is 32 bytes of the segment, two core
                    // matrices of B
                    uint64_t da = da0 + (uint32_t)((t0 - s0) * 2);
                    uint64_t db = b_base + (uint32_t)((st * kStageBytes) >> 4) +
                                  (uint32_t)((t0 - kSteps * c) * (2 * kLead / 16));
                    if (!(h ? band_s : band_n)) {
                        // (this warp only keeps the barriers' counts)
                    } else if (small) {
                        const int s_c = kSteps * c + kSteps / 2 - t0;  // the closest approach's step
                        if (c == mid && s_c >= 0 && s_c < t1 - t0) {
                            tc::mma_f16(d, da + (uint32_t)(2 * s_c) + a_l,
                                        db + (uint32_t)(s_c * (2 * kLead / 16)) + b_l, idesc, acc);
                            if (abs(q_lo + qi - r0) <= kNear)
                                tc::mma_f16(d, da + (uint32_t)(2 * s_c), e_base + (n & 1u) * (kEBytes >> 4),
                                            tc::idesc_f16(128, 16), 1u);
                            acc = 1u;
                        }
#pragma unroll
                        for (int s = 0; s < kSteps; ++s) {
                            if (s >= t1 - t0) break;
                            tc::mma_f16(d, da + (uint32_t)(2 * s), db + (uint32_t)(s * (2 * kLead / 16)) + b_l,
                                        idesc, acc);
                            tc::mma_f16(d, da + (uint32_t)(2 * s) + a_l,
                                        db + (uint32_t)(s * (2 * kLead / 16)), idesc, 1u);
                            acc = 1u;
                        }
                    } else {
#pragma unroll
                        for (int s = 0; s < kSteps; ++s) {  // (the closest approach's is the last)
                            if (s >= t1 - t0) break;
                            tc::mma_f16(d, da + (uint32_t)(2 * s), db + (uint32_t)(s * (2 * kLead / 16)),
                                        idesc, acc);
                            acc = 1u;
                        }
                    }
                    tc::mma_commit(&b_free[st]);
                    if (++st == kStages) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (!ok) break;
                tc::mma_commit(&d_done);
                ++n;
            }
            // (after an abort: nothing of this thread is in flight when its last commit is done)
            if (n_chunks > 0 && s_abort) {
                tc::mma_commit(&s_drain[warp & 3]);
                drained = tc::mbar_wait(&s_drain[warp & 3], 0u);
            }
        }
        __syncwarp();
    } else {
        // 640 x 96 registers at launch = 512 x 112 + 128 x 32
        asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        if (warp < kEpi / 32) {
            // ---- summing warps
            const int R = warp >> 2, quarter = warp & 3;
            const int L = R ? L1 : L0, t = R ? Rb.phase : Ra.phase;
            const int k_lo = R ? k_lo1 : k_lo0, k_hi = R ? k_hi1 : k_hi0;
            const int two_l = 2 * L;
            const float inv2L = 1.0f / (float)two_l;
            float4 *tot = sT + R * C.tcap;
            float2 *turn = sY + warp * kTurn;
            const uint32_t td = tmem + ((uint32_t)(quarter * 32) << 16);
            const uint64_t m1 = pack2(-1.0f, -1.0f), cut = pack2(-0x1p-24f, -0x1p-24f);
            uint32_t n = 0;
            for (int qi = 0; qi < nq; ++qi) {
                const QInfo g = sQ[qi];
                if (max((int)g.jE[0], (int)g.jE[1]) < 0) continue;
                const uint32_t buf = n & 1u;
                wait_all(&e_ready[buf], (n >> 1) & 1u, &s_abort);
                // the ring's other warps have added ring n - 1: outputs change hands
                asm volatile("bar.sync %0, 128;" ::"r"(2 + R) : "memory");
                const int jE = g.jE[R], Lq = g.len, step = 2 * Lq;
                const bool shifted = g.c[0] | g.c[1];
                // outputs at positions n0 + 256 quarter .. + 255: k in [kA, kB]
                auto first = [&](int pos) {  // ceil(num / step)
                    const int num = (2 * pos + g.phase - 1) * L - t * Lq;
                    int k = (int)((float)num / (float)step);
                    k += k * step < num ? 1 : 0;
                    k -= (k - 1) * step >= num ? 1 : 0;
                    return k;
                };
                const int p0 = g.n0 + 256 * quarter;
                const int kA = max(first(p0), k_lo);
                const int kB = jE < 0 ? kA - 1 : min(first(p0 + 256) - 1, k_hi);
                bool waited = false;
                for (int kb = kA; kb <= kB; kb += 32 * kOut) {
                    float f[kOut];
                    uint64_t e2[kOut], v[kOut];
                    int at[kOut];
                    float ec[kP];  // the edge cell's polynomial, for the map as stored
#pragma unroll
                    for (int p = 0; p < kP; ++p) ec[p] = s_edge[buf][R][p] * xscale;
                    const int eR = g.eR[R];
                    const float2 *x = sF + buf * xc;
#pragma unroll
                    for (int o = 0; o < kOut; ++o) {
                        // position and offset of output k (clamped: the last ones are not kept)
                        const int k = min(kb + 32 * o + lane, kB);
                        const int u = (2 * k + t) * Lq + (1 - g.phase) * L - two_l * p0;
                        int i = (int)((float)u * inv2L);
                        int rem = u - i * two_l;
                        if (rem < 0) {
                            --i;
                            rem += two_l;
                        } else if (rem >= two_l) {
                            ++i;
                            rem -= two_l;
                        }
                        rem -= L;
                        f[o] = (float)rem * inv2L;
                        at[o] = i + (i >> 3) * 2;
                        const float fo = f[o], f2 = fo * fo;
                        // the edge cells' weights: even and odd parts
                        const float we = fmaf(f2, fmaf(f2, fmaf(f2, fmaf(f2, ec[8], ec[6]), ec[4]), ec[2]), ec[0]);
                        const float wo = fo * fmaf(f2, fmaf(f2, fmaf(f2, ec[7], ec[5]), ec[3]), ec[1]);
                        const bool in_r = rem <= eR, in_l = rem >= -eR;
                        const float wr = jE > 0 ? (in_r ? we + wo : 0.0f) : (in_r && in_l ? we : 0.0f);
                        const float wl = jE > 0 && in_l ? we - wo : 0.0f;
                        // elements of positions n - jE and n + jE
                        const int er = 256 * quarter + i - jE - g.base;
                        const float2 xr = x[er], xl = x[er + 2 * jE];
                        e2[o] = fma2(pack2(wl, wl), pack2(xl.x, xl.y),
                                     fma2(pack2(wr, wr), pack2(xr.x, xr.y), 0ull));
                        v[o] = 0ull;
                    }
                    if (!waited) {  // the accumulators (the edge pixels came from the map)
                        wait_all(&d_done, n & 1u, &s_abort);
                        tc::fence_after_sync();
                        waited = true;
                    }
#pragma unroll 1
                    for (int p = kP - 1;; --p) {
                        const uint32_t c = td + (uint32_t)(8 * group_of(R, p));
                        uint32_t a[8], b[8];
                        tc::tmem_ld8(c, a);
                        tc::tmem_ld8(c + kHemi, b);
                        uint64_t w[8];
                        if (p < kP3) {
                            uint32_t xa[8], xb[8];
                            tc::tmem_ld8(c + kN, xa);
                            tc::tmem_ld8(c + kN + kHemi, xb);
                            tc::loaded(a);
                            tc::loaded(b);
                            tc::loaded(xa);
                            tc::loaded(xb);
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                w[i] = add2((uint64_t)b[i] << 32 | a[i], (uint64_t)xb[i] << 32 | xa[i]);
                        } else {
                            tc::loaded(a);
                            tc::loaded(b);
#pragma unroll
                            for (int i = 0; i < 8; ++i) w[i] = (uint64_t)b[i] << 32 | a[i];
                        }
                        __syncwarp();
                        ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(turn + 10 * lane);
#pragma unroll
                        for (int i = 0; i < 8; i += 2) dst[i / 2] = make_ulonglong2(w[i], w[i + 1]);
                        __syncwarp();
                        if (p == 0) break;  // y_0 waits in the buffer
#pragma unroll
                        for (int o = 0; o < kOut; ++o)
                            v[o] = fma2(v[o], pack2(f[o], f[o]),
                                        *reinterpret_cast<const uint64_t *>(turn + at[o]));
                    }
                    const bool last = kb + 32 * kOut > kB;
                    if (last && !shifted) {  // the accumulators are no longer needed
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&d_free[buf]);
                    }
#pragma unroll
                    for (int o = 0; o < kOut; ++o) {
                        const int k = kb + 32 * o + lane;
                        if (k > kB) break;
                        // z, the ring's sum, and total + z with the rounding errors of both, and
                        // with the 2^-24 of z that the MMAs' cuts cost on average, kept apart
                        ulonglong2 *q = reinterpret_cast<ulonglong2 *>(tot + k - k_lo);
                        ulonglong2 s = *q;
                        uint64_t e0, e1;
                        const uint64_t z =
                            two_sum2(*reinterpret_cast<const uint64_t *>(turn + at[o]),
                                     fma2(v[o], pack2(f[o], f[o]), e2[o]), &e0);
                        s.x = two_sum2(s.x, z, &e1);
                        s.y = fma2(z, cut, fma2(add2(e0, e1), m1, s.y));
                        *q = s;
                    }
                    if (shifted) {  // the constants' share
                        const float *S = s_sum[buf][R];
                        const float ms_n = shift_of(g, 0), ms_s = shift_of(g, 1);
#pragma unroll 1
                        for (int k = kb + lane; k <= min(kB, kb + 32 * kOut - 1); k += 32) {
                            const int u = (2 * k + t) * Lq + (1 - g.phase) * L - two_l * p0;
                            const float f = (float)(u % two_l - L) * inv2L, f2 = f * f;
                            const float c = fmaf(f2, fmaf(f2, fmaf(f2, fmaf(f2, S[8], S[6]), S[4]), S[2]), S[0]);
                            ulonglong2 *q = reinterpret_cast<ulonglong2 *>(tot + k - k_lo);
                            ulonglong2 s = *q;
                            uint64_t e;
                            s.x = two_sum2(s.x, pack2(ms_n * c, ms_s * c), &e);
                            s.y = fma2(e, m1, s.y);
                            *q = s;
                        }
                    }
                    if (last && shifted) {  // (nor the sums of the weights)
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&d_free[buf]);
                    }
                }
                if (!waited) {  // no outputs here: keep step
                    wait_all(&d_done, n & 1u, &s_abort);
                    if (lane == 0) tc::mbar_arrive(&d_free[buf]);
                }
                ++n;
            }
            asm volatile("bar.sync 4, %0;" ::"r"(kEpi) : "memory");
            // ---- outputs: four warps per (ring, hemisphere) in turn
            for (int h = 0; h < 2; ++h) {
                const int ring = h ? P.nrings - 1 - (r0 + R) : r0 + R;
                if (R >= n_r || ring < band_lo || ring > band_hi || (h && ring == r0 + R) || s_abort)
                    continue;
                float *dst = o + P.d_rings[ring].start;
                const float unscale = xunscale * C.wunscale;
                for (int k = k_lo + quarter * 32 + lane; k <= k_hi; k += 128) {
                    const float4 s = tot[k - k_lo];
                    const float hi = (h ? s.y : s.x) * unscale, lo = -(h ? s.w : s.z) * unscale;
                    const float v = fmaf(hi, P.domega, fmaf(hi, C.domega_lo, lo * P.domega));
                    if (add) dst[k] += v;
                    else dst[k] = v;
                }
            }
        } else {
            // ---- builder warps
            const int bt = tid - kEpi, bw = warp - kEpi / 32;
            uint32_t n = 0, n_chunks = 0;
            float xn[kXr], xs[kXr];
            // loads of an input ring: segments into registers, coefficients by async copies
            auto fetch = [&](int qi, uint32_t m_) {
                const QInfo g = sQ[qi];
                const float *rn = m + g.start, *rs = m + (P.npix - g.start - g.len);
#pragma unroll
                for (int e = 0; e < kXr; ++e) {
                    if (bt + e * kBuild >= g.n_e) break;
                    int i = g.a + bt + e * kBuild;
                    while (i >= g.len) i -= g.len;
                    xn[e] = __ldg(rn + i);
                    xs[e] = __ldg(rs + i);
                }
                uint32_t *dst = sK + (m_ & 1u) * k_cap;
                const int w0 = g.jE[0] >= 0 ? coef_words(g.jE[0]) / 4 : 0;
                const int w1 = g.jE[1] >= 0 ? coef_words(g.jE[1]) / 4 : 0;
                for (int e = bt; e < w0 + w1; e += kBuild)
                    copy16(dst + 4 * e, C.d_coef + 4ull * (e < w0 ? g.off[0] + e : g.off[1] + (e - w0)));
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            auto next = [&](int qi) {  // the next input ring with pixels within the cut
                while (qi < nq && max(sQ[qi].jE[0], sQ[qi].jE[1]) < 0) ++qi;
                return qi;
            };
            int qi = next(0);
            if (qi < nq) fetch(qi, 0u);
            while (qi < nq) {
                const QInfo g = sQ[qi];
                const uint32_t buf = n & 1u;
                const int n_pos = 16 * (g.s1 - g.s0);
                const float ms_n = shift_of(g, 0), ms_s = shift_of(g, 1);
                // ring n - 2 has left these buffers
                if (n >= 2) wait_all(&d_free[buf], ((n >> 1) - 1u) & 1u, &s_abort);
                // ---- the segments, as they are and scaled and split
#pragma unroll
                for (int e = 0; e < kXr; ++e) {
                    const int i = bt + e * kBuild;
                    if (i >= g.n_e) break;
                    sF[buf * xc + i] = make_float2(xn[e], xs[e]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (!(h ? band_s : band_n)) continue;
                        __half *xh = sX + (h * 2 + buf) * 2 * xc;
                        const float y = fmaf(h ? xs[e] : xn[e], xscale, h ? -ms_s : -ms_n);
                        const __half hh = __float2half_rn(y);
                        xh[i] = hh;
                        xh[xc + i] = __float2half_rn(y - __half2float(hh));
                    }
                }
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                asm volatile("bar.sync 1, %0;" ::"r"(kBuild) : "memory");
                // ---- the coefficient sequences of each group (R, p): element x is
                // c_p[-Delta] at Delta = x + base - 8, c_p[-j] = (-1)^p c_p[j], zero beyond
                // the interior cells.  Word k of the even sequence holds elements 2k and
                // 2k + 1, of the odd one 2k - 1 and 2k; high parts of all groups, then low
                // parts of the first kG3.
                const uint32_t *raw = sK + buf * k_cap;
                const int raw1 = g.jE[0] >= 0 ? coef_words(g.jE[0]) : 0;
                {
                    const int n_w = n_pos / 2 + 8, n_blk = (n_w + 31) / 32;
                    for (int task = bw; task < kG * n_blk; task += kBuild / 32) {
                        const int grp = task % kG, k = task / kG * 32 + lane;
                        // (ring, power) of the group
                        const int R = grp & 1, p = grp >> 1;
                        const int jE = g.jE[R];
                        if (k >= n_w) continue;
                        const uint32_t flip = p & 1 ? 0x80008000u : 0u;
                        const uint32_t *src = raw + (R ? raw1 : 0) + p;
                        uint32_t c[3];
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            const int dl = 2 * k - 9 + i + g.base, j = dl < 0 ? -dl : dl;
                            c[i] = j < jE ? src[j * kP] ^ (dl > 0 ? flip : 0u) : 0u;
                        }
                        uint32_t *d = sC + 2 * grp * w_cap + k;
                        d[0] = __byte_perm(c[1], c[2], 0x5410);
                        d[w_cap] = __byte_perm(c[0], c[1], 0x5410);
                        if (p < kP3) {
                            d += 2 * kG * w_cap;
                            d[0] = __byte_perm(c[1], c[2], 0x7632);
                            d[w_cap] = __byte_perm(c[0], c[1], 0x7632);
                        }
                    }
                    // third parts of c_0 in the closest approach's step: a thread's element e of
                    // row i in core matrix kg of ring R (base counts Delta from step s0)
                    if (abs(q_lo + qi - r0) <= kNear) {
                        const int e = bt & 7, i = (bt >> 3) & 7, kg = (bt >> 6) & 1, R = bt >> 7;
                        const int dl = g.base + 16 * (kSteps * g.mid + kSteps / 2 - g.s0) + 8 * kg + e - i;
                        const int j = dl < 0 ? -dl : dl, jE = g.jE[R];
                        const __half *src = third_parts(raw + (R ? raw1 : 0), jE);
                        reinterpret_cast<__half *>(sE + buf * kEBytes + R * 2 * kLead + kg * kLead)[8 * i + e] =
                            j < min(jE, kE) ? src[j] : __half(0.0f);
                    }
                    // the edge cells: in FP32, not in the products
                    if (bt < 2 * kP) {
                        const int R = bt >= kP, p = bt - R * kP, jE = g.jE[R];
                        if (jE >= 0) {
                            const uint32_t hl = raw[(R ? raw1 : 0) + jE * kP + p];
                            s_edge[buf][R][p] = __half2float(__ushort_as_half((unsigned short)hl)) +
                                                __half2float(__ushort_as_half((unsigned short)(hl >> 16)));
                        }
                    }
                    if (g.c[0] | g.c[1]) {  // sums of the even coefficients over a window
                        for (int task = bw; task < 10; task += kBuild / 32) {
                            const int R = task / 5, p = 2 * (task % 5);
                            const uint32_t *src = raw + (R ? raw1 : 0) + p;
                            float s = 0.0f, comp = 0.0f;
                            for (int j = lane; j < g.jE[R]; j += 32) {
                                const uint32_t hl = src[j * kP];
                                float c = __half2float(__ushort_as_half((unsigned short)(hl >> 16)));
                                if (p == 0 && j < kE) c += __half2float(third_parts(src, g.jE[R])[j]);
                                c += __half2float(__ushort_as_half((unsigned short)hl));
                                const float z = (j ? 2.0f : 1.0f) * c - comp;
                                const float w = s + z;
                                comp = (w - s) - z;
                                s = w;
                            }
                            s -= comp;
#pragma unroll
                            for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(~0u, s, k);
                            if (lane == 0) s_sum[buf][R][p] = s;
                        }
                    }
                }
                const int qn = next(qi + 1);
                if (qn < nq) fetch(qn, n + 1u);
                asm volatile("bar.sync 1, %0;" ::"r"(kBuild) : "memory");
                if (lane == 0) tc::mbar_arrive(&e_ready[buf]);
                // ---- B, chunk by chunk
                const int c_lo = g.s0 / kSteps, c_hi = (g.s1 - 1) / kSteps;
                for (int cc = c_lo; cc <= c_hi; ++cc, ++n_chunks) {
                    const int c = tc::chunk_of(cc, c_hi, g.mid);
                    const uint32_t st = n_chunks % kStages;
                    if (n_chunks >= kStages)
                        wait_all(&b_free[st], (n_chunks / kStages - 1u) & 1u, &s_abort);
                    const int t0 = max((int)g.s0, kSteps * c), t1 = min((int)g.s1, kSteps * c + kSteps);
                    unsigned char *sb = sB + st * kStageBytes + (t0 - kSteps * c) * 2 * kLead;
                    // a thread lays out one core matrix (eight rows) of one group: rows of even
                    // i from the words of the even sequence, of odd i from the odd one, four
                    // words a row, row i two elements before row i - 2
                    const int cols = 2 * (t1 - t0);  // core matrices of a group: 2 or 4
                    const int w0 = 4 + 8 * (t0 - g.s0);  // word of the step's first element
                    for (int e = bt; e < (kG + kG3) * cols; e += kBuild) {
                        const int grp = cols == 4 ? e >> 2 : e >> 1, kg = e - grp * cols;
                        const uint32_t *p = sC + 2 * grp * w_cap + w0 + 4 * kg;
                        unsigned char *dst = sb + grp * kGroupBytes + kg * kLead;
#pragma unroll
                        for (int odd = 0; odd < 2; ++odd) {
                            const uint4 lo = *reinterpret_cast<const uint4 *>(p + odd * w_cap - 4);
                            const uint4 hi = *reinterpret_cast<const uint4 *>(p + odd * w_cap);
                            uint4 *d = reinterpret_cast<uint4 *>(dst) + odd;
                            d[0] = hi;
                            d[2] = make_uint4(lo.w, hi.x, hi.y, hi.z);
                            d[4] = make_uint4(lo.z, lo.w, hi.x, hi.y);
                            d[6] = make_uint4(lo.y, lo.z, lo.w, hi.x);
                        }
                    }
                    tc::fence_async_smem();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&b_full[st]);
                }
                qi = qn;
                ++n;
            }
        }
    }
    tc::fence_before_sync();
    const bool all_drained = __syncthreads_and(drained);
    if (s_abort && tid == 0) atomicExch(err, all_drained ? KSC_ERR_TIMEOUT : KSC_ERR_TIMEOUT_UNDRAINED);
    // tensor memory that an MMA may still write is not freed
    if (warp == kT / 32 && all_drained)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// Coefficients of the regular ring pairs of output ring r, one warp per pair, one
// lane per cell: the kernel at nine nodes of the cell, its value at a table node as an FP32
// pair, then the interpolating polynomial in FP64 (even and odd parts apart), each
// coefficient scaled and split into two FP16 parts.
__global__ void __launch_bounds__(256)
cap_coef_kernel(const ConvPlan P, const CapTc C, const CapCoef K, int ring_lo, int ring_hi) {
    const int r = ring_lo + blockIdx.x;
    if (r > ring_hi) return;
    const int2 rg = P.d_range[r];
    const int L = P.d_rings[r].len, lane = threadIdx.x & 31;
    for (int q = rg.x + (threadIdx.x >> 5); q <= rg.y; q += 8) {
        const int ip = P.d_pair_base[r] + q - rg.x;
        const int ncut = C.d_ncut[ip];
        if (ncut < 0) continue;
        const int jE = ncut >= L ? (ncut - L) / (2 * L) + 1 : 0;
        const PairInfo pi = P.d_pairs[ip];
        const DF A{pi.Ah, pi.Al}, B{pi.Bh, pi.Bl};
        const float2 cq = K.d_ringc[q];  // pi / L' as a double-float pair
        uint32_t *dst = K.d_coef + 4ull * C.d_coef_off[ip];
        for (int j = lane; j <= jE; j += 32) {
            auto value = [&](float x) {
                const float xh = x * cq.x;
                const float xl = fmaf(x, cq.x, -xh) + x * cq.y;
                int ti;
                float f;
                chord_to_table_sel(A, B, sin_df(xh, xl), K.next2, &ti, &f);
                ti = min(ti, K.n_ext - 1);
                const float4 c = __ldg(&K.d_tab[ti]);
                return (double)c.x + ((double)__ldg(&K.d_tab_lo[ti]) +
                                      (double)(f * fmaf(f, fmaf(f, c.w, c.z), c.y)));
            };
            const double w0 = value((float)j);
            double e4[4], o4[4], c[kP];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const float gs = s == 0 ? node(1) : s == 1 ? node(2) : s == 2 ? node(3) : node(4);
                const double a = value((float)j + gs), b = value((float)j - gs);
                e4[s] = 0.5 * (a + b) - w0;
                o4[s] = 0.5 * (a - b);
            }
            c[0] = w0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                double e = 0.0, d = 0.0;
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    e = fma(K.me[4 * k + s], e4[s], e);
                    d = fma(K.mo[4 * k + s], o4[s], d);
                }
                c[2 * k + 2] = e;
                c[2 * k + 1] = j == 0 ? 0.0 : d;  // even about cell 0
            }
#pragma unroll
            for (int p = 0; p < kP; ++p) {
                const double v = c[p] * (double)C.wscale;
                if (!(fabs(v) <= 65504.0)) *K.d_too_large = 1;
                const __half h = __float2half_rn((float)v);
                const __half l = __float2half_rn((float)(v - (double)__half2float(h)));
                dst[j * kP + p] = (uint32_t)__half_as_ushort(l) << 16 | __half_as_ushort(h);
                if (p == 0 && j < kE)
                    reinterpret_cast<__half *>(dst + kP * (jE + 1))[j] =
                        __float2half_rn((float)(v - (double)__half2float(h) - (double)__half2float(l)));
            }
        }
    }
}

// The irregular ring pairs of output ring r (and its mirror), added to the output.  A block
// takes 32 first-quarter positions of r, a lane each; its sixteen warps share the ring's list
// of input rings (99 blocks for 152 SMs at nside 1024, 160': 330 us with eight warps, 281 us
// with sixteen; 612 blocks at 2048, 240': 6.47 ms, and 5.0 with weights and products inside the
// cut only; two blocks per SM, at 64 registers: slower).  For one input pixel all lanes
// read the same values, eight (four quarter turns, two hemispheres) per weight.
constexpr int kDirect = 512;
// input pixels between folds into the compensated sums: nside 256, 1800': error rms 9.2e-8 of
// the output's with 64 (near a centre a few large products share a chunk with many small
// ones), 7.4e-8 with 16 (gather 8.3e-8); nside 1024, 128 pixels: 35.3 and 36.0 ms a call
constexpr int kFold = 16;
__global__ void __launch_bounds__(kDirect)
cap_direct_kernel(const ConvPlan P, const int2 *__restrict__ items,
                  const int *__restrict__ list_first, const int *__restrict__ list,
                  const MapSet maps, int band_lo, int band_hi, const int *__restrict__ flags) {
    constexpr int kW = kDirect / 32;
    __shared__ float part[kW][8][32];
    const int2 it = items[blockIdx.x];
    const int r = it.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (flags[(long long)blockIdx.y * (P.nrings + 1) + r]) return;
    const float *__restrict__ m = maps.input(blockIdx.y);
    float *__restrict__ o = maps.output(blockIdx.y);
    const DevRing R = P.d_rings[r];
    const int L = R.len, Q = L / 4, k = min(it.y + lane, Q - 1);
    const int base = P.d_pair_base[r] - P.d_range[r].x;
    float sum[8], comp[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) sum[i] = comp[i] = 0.0f;
    for (int e = list_first[r] + warp; e < list_first[r + 1]; e += kW) {
        const int q = list[e];
        const DevRing G = P.d_rings[q];
        const int Lq = G.len, Qq = Lq / 4;
        const PairInfo pi = P.d_pairs[base + q];
        const DF A{pi.Ah, pi.Al}, B{pi.Bh, pi.Bl};
        const float *xn = m + G.start, *xs = m + P.d_rings[P.nrings - 1 - q].start;
        const int full = 2 * L * Lq;
        int n0 = (2 * k + R.phase) * Lq - G.phase * L;  // N of input pixel 0
        for (int j0 = 0; j0 < Lq; j0 += kFold) {
            float acc[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
            const int j1 = min(j0 + kFold, Lq);
#pragma unroll 4
            for (int j = j0; j < j1; ++j) {
                int n = n0 - 2 * j * L;  // folded to half a turn
                n += n < -(full / 2) ? full : 0;
                n -= n > full / 2 ? full : 0;
                const float nf = (float)n;
                const float xh = nf * pi.ch, xl = fmaf(nf, pi.ch, -xh) + nf * pi.cl;
                int ti;
                float f;
                // (a pixel past the cut adds nothing, whatever its value)
                if (!chord_to_table_sel(A, B, sin_df(xh, xl), P.nint2, &ti, &f)) continue;
                const float w = hermite(__ldg(&P.d_tab[min(ti, P.n_int)]), f);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    int i = j + a * Qq;
                    i -= i >= Lq ? Lq : 0;
                    acc[a] = fmaf(w, __ldg(xn + i), acc[a]);
                    acc[4 + a] = fmaf(w, __ldg(xs + i), acc[4 + a]);
                }
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float y = acc[i] - comp[i], t = sum[i] + y;
                comp[i] = (t - sum[i]) - y;
                sum[i] = t;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) part[warp][i][lane] = sum[i] - comp[i];
    __syncthreads();
    if (warp >= 8) return;
    // image `warp` of every position: the warps' sums in order
    const int a = warp & 3, south = warp >> 2;
    const int rs = P.nrings - 1 - r, ring = south ? rs : r;
    if (it.y + lane < Q && ring >= band_lo && ring <= band_hi && !(south && rs == r)) {
        float s = 0.0f, c = 0.0f;
#pragma unroll
        for (int i = 0; i < kW; ++i) {
            const float y = part[i][warp][lane] - c, t = s + y;
            c = (t - s) - y;
            s = t;
        }
        float *dst = o + P.d_rings[ring].start + it.y + lane + a * Q;
        *dst = fmaf(s, P.domega, *dst);
    }
}

// ring_range[map][ring] = the largest and the smallest nonzero block maximum (bits) over
// the 64-pixel blocks that the ring touches; one warp per ring of the reach.
__global__ void __launch_bounds__(256)
ring_range_kernel(const ConvPlan P, const uint32_t *__restrict__ blockmax, long long block_stride,
                  const InputReach in, uint2 *__restrict__ ring_range) {
    const uint32_t *bm = blockmax + (long long)blockIdx.y * block_stride;
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int n0 = in.q1 - in.q0 + 1, n = n0 + max(in.q3 - in.q2 + 1, 0);
    if (i >= n) return;
    const int r = i < n0 ? in.q0 + i : in.q2 + (i - n0);
    const DevRing R = P.d_rings[r];
    uint32_t mx = 0u, mn = 0xffffffffu;
    for (int b = (R.start >> 6) + lane; b <= (R.start + R.len - 1) >> 6; b += 32) {
        const uint32_t v = __ldg(bm + b);
        mx = max(mx, v);
        if (v) mn = min(mn, v);
    }
    mx = __reduce_max_sync(~0u, mx);
    mn = __reduce_min_sync(~0u, mn);
    if (lane == 0) ring_range[(long long)blockIdx.y * P.nrings + r] = make_uint2(mx, mn);
}

size_t cap_smem(const CapTc &c) {
    const size_t xc = c.span + c.wpos, w_cap = ((c.wpos / 2 + 8 + 11) & ~31) + 20;
    const size_t body = 2 * 8 * xc + 8 * (size_t)(kEpi / 32) * kTurn + 16 * 2 * (size_t)c.tcap +
                        8 * 2 * xc + 4 * 4 * (size_t)coef_words(c.jcap - 1) +
                        4 * 2 * (kG + kG3) * w_cap + sizeof(QInfo) * (size_t)c.nq;
    // (the rows past a tile's last position read up to 1024 + wpos elements of a segment)
    return (size_t)kStages * kStageBytes + 2 * kEBytes + std::max(body, (size_t)2 * (6 * xc + kSpan + c.wpos + xc));
}

// Inverse of a 4 x 4 matrix (Gauss-Jordan with row pivots).
void invert4(double a[4][4], double inv[4][4]) {
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) inv[i][j] = i == j;
    for (int c = 0; c < 4; ++c) {
        int p = c;
        for (int i = c + 1; i < 4; ++i)
            if (std::fabs(a[i][c]) > std::fabs(a[p][c])) p = i;
        for (int j = 0; j < 4; ++j) {
            std::swap(a[c][j], a[p][j]);
            std::swap(inv[c][j], inv[p][j]);
        }
        const double d = a[c][c];
        for (int j = 0; j < 4; ++j) {
            a[c][j] /= d;
            inv[c][j] /= d;
        }
        for (int i = 0; i < 4; ++i) {
            if (i == c) continue;
            const double f = a[i][c];
            for (int j = 0; j < 4; ++j) {
                a[i][j] -= f * a[c][j];
                inv[i][j] -= f * inv[c][j];
            }
        }
    }
}

} // namespace

int cap_tc_span() { return kSpan; }
int cap_tc_degree() { return kP - 1; }
int cap_tc_split_powers() { return kP3; }
int cap_tc_positions(int w, int L) {
    const Window v = window_of(w, L);
    return 16 * (v.s1 - v.s0);
}

bool cap_tc_fits(const CapTc &c) {
    return cap_smem(c) <= (size_t)kMaxDynSmem && c.span + c.wpos <= kXr * kBuild;
}

int cap_tc_words(int jE) { return coef_words(jE); }

cudaError_t launch_cap_coef(const ConvPlan &p, const CapTc &c, const CapCoef &k, cudaStream_t st) {
    CapCoef kk = k;
    double a[4][4], inv[4][4];
    for (int s = 0; s < 4; ++s)
        for (int i = 0; i < 4; ++i) a[s][i] = std::pow((double)node(s + 1), 2 * (i + 1));
    invert4(a, inv);
    for (int i = 0; i < 4; ++i)
        for (int s = 0; s < 4; ++s) kk.me[4 * i + s] = inv[i][s];
    for (int s = 0; s < 4; ++s)
        for (int i = 0; i < 4; ++i) a[s][i] = std::pow((double)node(s + 1), 2 * i + 1);
    invert4(a, inv);
    for (int i = 0; i < 4; ++i)
        for (int s = 0; s < 4; ++s) kk.mo[4 * i + s] = inv[i][s];
    cap_coef_kernel<<<c.ring_end - c.ring_first + 1, 256, 0, st>>>(p, c, kk, c.ring_first, c.ring_end);
    return cudaGetLastError();
}

cudaError_t launch_ring_range(const ConvPlan &p, const unsigned *bm, int n_maps,
                              const InputReach &in, uint2 *rr, cudaStream_t st) {
    const int n = in.q1 - in.q0 + 1 + std::max(in.q3 - in.q2 + 1, 0);
    dim3 grid((n + 7) / 8, n_maps);
    ring_range_kernel<<<grid, 256, 0, st>>>(p, bm, map_blocks(p), in, rr);
    return cudaGetLastError();
}

cudaError_t launch_cap_direct(const ConvPlan &p, const int2 *d_items, int n_items,
                              const int *d_first, const int *d_list, const MapSet &maps,
                              int n_maps, int band_lo, int band_hi, const int *flags,
                              cudaStream_t st) {
    if (n_items <= 0) return cudaSuccess;
    dim3 grid(n_items, n_maps);
    cap_direct_kernel<<<grid, kDirect, 0, st>>>(p, d_items, d_first, d_list, maps, band_lo, band_hi,
                                            flags);
    return cudaGetLastError();
}

cudaError_t launch_conv_cap_tc(const ConvPlan &p, const CapTc &c, const int2 *d_tiles, int n_tiles,
                               const MapSet &maps, int n_maps, int belt_split, int band_lo,
                               int band_hi, const uint2 *rr, int *flags, bool back,
                               int *d_err, cudaStream_t st) {
    if (n_tiles <= 0) return cudaSuccess;
    const size_t smem = cap_smem(c);
    cudaError_t e = cudaFuncSetAttribute(conv_cap_tc_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kMaxDynSmem);  // (one value: calls may race)
    if (e != cudaSuccess) return e;
    dim3 grid(n_tiles, n_maps);
    conv_cap_tc_kernel<<<grid, kThreads, smem, st>>>(p, c, d_tiles, maps, belt_split, band_lo,
                                                     band_hi, rr, flags, back, d_err);
    return cudaGetLastError();
}

} // namespace ksc
