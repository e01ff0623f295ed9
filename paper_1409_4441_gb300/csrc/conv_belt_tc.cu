// Real-space convolution, equatorial-belt ring pairs, on the tcgen05 tensor cores.
//
// For an output ring r and an input ring q of the belt the kernel weight depends on
// Delta = k' - k only (conv_belt.cu), so the ring pair is a Toeplitz product.  A CTA
// owns 16 consecutive output rings and 8 N consecutive pixels of each, and for every
// input ring q in reach of one of them adds
//
//   D[(R, i), n] += sum_j A[(R, i), j] B[j, n],   A[(R, i), j] = w_R[d0 + j - i],
//                                                 B[j, n] = m_q[k0 + d0 + j + 8 n],
//
// D[(R, i), n] being pixel k0 + 8 n + i of ring R: M = 128 rows are 16 rings x 8 offsets,
// N columns are groups of eight pixels, K is the window.  Neither operand is copied out
// to a full matrix.  B's core matrices (8 columns x 16 bytes) are read straight from the
// input segment as it lies in shared memory: columns 8 elements (16 bytes) apart, so
// K-adjacent core matrices overlap at a stride of 16 bytes.  A's eight rows of a ring are
// the same weights shifted by one element each.  The padding of a window is 7 positions
// plus the rounding to K = 16, against 13 to 25 of the FFMA form.
//
// Precision.  With the map scaled per tile and the weights per split so that their
// largest magnitudes lie near 2^15 and 2^13, each value is the sum of two FP16 numbers,
// v = h + l, l the rounding error of h, for |v| >= 2^-1 to 23 of FP32's 24 bits (two parts of 11
// and a sign: a quarter of the values lose their last one, 4.4e-8 rms), within 2^-25
// otherwise, i.e. within 2^-40 of the largest.  Three MMAs
// per 16 positions sum w_h m_l, w_l m_h and w_h m_h in FP32; w_l m_l (below 2^-24 of the
// product) is summed too where the weights are large, in the step of the closest
// approach.  An MMA cuts every addend, the accumulator too, at 2^-25 of the largest one and
// rounds the sum toward zero to 24 bits (found with known operands), so the order matters:
// within 128 positions the small products first, the 128 positions that hold the closest
// approach last, and its own step at the very end.  After each input ring the
// accumulator is folded into FP32 totals with the rounding error of the sum (two-sum),
// plus the 2^-24 of the partial that the cuts take from it on average, written back to
// tensor memory as the start of a later partial.  The weights keep the rounding error of
// their last addition in w_l.  The cuts are toward zero and add up where all products have
// one sign: where the blocks of an input ring are of one size, a constant near their mean is
// taken off the ring and put back through the sum of the weights (signed mean error of belt
// pixels, a positive map with a gradient from pole to pole, nside 1024, 10' beam, l_cut 512,
// 400': 2.9e-7 of the output with one constant a tile, 7e-9 so).
//
// A tile where some block of 64 input pixels is more than 2^14 below the tile's largest
// value (all-zero blocks aside), or that holds an infinity or NaN, is left to
// conv_belt_kernel (belt_tc_flags): the scaled split would not carry its values to 26
// bits of their neighbourhood, or would spread a NaN further than the window.
//
// Every mbarrier wait is bounded; a wait that runs out raises the device error flag.
#include <algorithm>
#include <cstdint>

#include "ksc_device.cuh"
#include "ksc_internal.h"
#include "ksc_tc_split.cuh"

namespace ksc {
namespace {

constexpr int kT = 512;        // builder threads: warp R builds ring R's weights
constexpr int kThreads = kT + 128;  // and a warpgroup whose first warp issues the MMAs
constexpr int kRings = 16;     // output rings of a tile
constexpr int kChunk = 128;    // window positions per A stage
constexpr int kSteps = kChunk / 16;
constexpr int kPartBytes = kRings * kChunk * 16;  // one FP16 part of an A stage (32 kB)
constexpr int kStageBytes = 2 * kPartBytes;
constexpr int kStages = 2;

using tc::Window;
using tc::add2;
using tc::chunk_of;
using tc::fma2;
using tc::pack2;
using tc::idesc_f16;
using tc::kRangeExp;
using tc::kXExp;
using tc::mma_f16;
using tc::tmem_ld8;
using tc::tmem_st8;
using tc::wait_or_abort;

__host__ __device__ __forceinline__ Window tile_window(int w, int L) {
    return tc::tile_window<kChunk>(w, L);
}

// N columns: 8 N pixels per ring.  grid.x runs over tiles (16-ring block, pixel tile),
// grid.y over maps.  A tile belongs to one of the split's (of plan_cols >= N columns), from
// which its scale, its constants and its flag come: a band of few rings takes narrower tiles, more
// of them, for the same bits.  Sixteen builder warps stage the map, evaluate the weights, lay out A
// and fold the accumulators; a seventeenth issues the MMAs (the
// rest of its warpgroup only gives its registers to the builders).  A builder warp hands a stage
// over by arriving on a_full; that arrival also says that its part of the ring's input
// segment is staged and that it has folded the accumulator the ring's MMAs will write
// (each warp folds ring n - 2 before it arrives for ring n).
template <int N>
__global__ void __launch_bounds__(kThreads, 1)
conv_belt_tc_kernel(const ConvPlan P, int block_lo, int n_tiles_k, int ring_lo, int ring_hi,
                    const MapSet maps,
                    const uint32_t *__restrict__ blockmax, long long block_stride,
                    unsigned char *__restrict__ flags, int n_tiles, int plan_cols, int wpos_cap,
                    int nq_cap,
                    float wscale, float wunscale, float domega_lo, int *__restrict__ err) {
    constexpr int kCols = N / 4;  // columns per thread (four warps share a lane quarter)
    constexpr int kStep = kCols < 16 ? 8 : 16;
    constexpr uint32_t kTmem = 2 * N;
    extern __shared__ __align__(1024) unsigned char smem[];
    // A stages | two input segments (two FP16 parts each) | weights (h, l pairs) | windows |
    // constants taken off the input rings (BF16 numbers)
    const int seg_cap = 8 * N + wpos_cap;  // elements
    const int w_cap = wpos_cap + 16;
    unsigned char *sA = smem;
    __half *sB = reinterpret_cast<__half *>(smem + kStages * kStageBytes);
    uint32_t *sW = reinterpret_cast<uint32_t *>(sB + 4 * seg_cap);
    short *sQ = reinterpret_cast<short *>(sW + kRings * w_cap);
    unsigned short *sC = reinterpret_cast<unsigned short *>(sQ + ((nq_cap + 1) & ~1));
    __shared__ __align__(8) uint64_t a_full[kStages], a_free[kStages], d_done[2];
    __shared__ uint32_t tmem_base;
    __shared__ uint32_t s_max, s_min;
    __shared__ int s_abort, s_lo, s_hi, s_bad, s_shift, s_band_lo, s_band_hi, s_tail;
    __shared__ float s_wsum[kRings];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rb = block_lo + blockIdx.x / n_tiles_k, ct = blockIdx.x % n_tiles_k;
    const int r_first = P.belt_lo + rb * kRings;
    const int n_rows = min(kRings, P.belt_hi - r_first + 1);
    const int L = 4 * P.nside, k0 = ct * 8 * N;
    const int plan_tile = k0 / (8 * plan_cols), plan_k0 = plan_tile * 8 * plan_cols;
    const float *__restrict__ m = maps.input(blockIdx.y);
    float *__restrict__ o = maps.output(blockIdx.y);
    const uint32_t *bm = blockmax + (long long)blockIdx.y * block_stride;
    const int start0 = P.d_rings[r_first].start;

    // ---- the tile's input rings and windows, and the range of the values in them
    if (tid == 0) {
        s_max = 0u;
        s_min = 0xffffffffu;
        s_abort = s_bad = s_shift = s_tail = 0;
        s_lo = P.belt_hi;
        s_hi = P.belt_lo;
        s_band_lo = P.belt_hi;
        s_band_hi = P.belt_lo;
        for (int b = 0; b < kStages; ++b) {
            tc::mbar_init(&a_full[b], kRings);
            tc::mbar_init(&a_free[b], 1);
        }
        for (int b = 0; b < 2; ++b) tc::mbar_init(&d_done[b], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (warp == 0 && lane < n_rows) {
        const int2 g = P.d_range[r_first + lane];
        atomicMin(&s_lo, max(g.x, P.belt_lo));
        atomicMax(&s_hi, min(g.y, P.belt_hi));
        if (r_first + lane >= ring_lo && r_first + lane <= ring_hi) {
            atomicMin(&s_band_lo, max(g.x, P.belt_lo));
            atomicMax(&s_band_hi, min(g.y, P.belt_hi));
        }
    }
    __syncthreads();
    const int q_lo = s_lo, nq = s_hi - s_lo + 1;
    // Input rings [s_band_lo, s_band_hi] reach an output ring of the band.  Those before add
    // nothing to its sums, whose folds are then all zero; of the s_tail rings after, only the folds
    // are carried out.  (Narrow tiles, which bands of few rings take: nine rings of nside 2048, 16
    // pixels: 0.165 -> 0.133 ms; wide ones have no registers for a second kind of fold.)
    constexpr bool kTrim = N <= 64;
    uint32_t vmax = 0u, vmin = 0xffffffffu;
    for (int q = q_lo + warp; q < q_lo + nq; q += kThreads / 32) {
        int w = -1;
        if (lane < n_rows) {
            const int2 g = P.d_range[r_first + lane];
            if (q >= g.x && q <= g.y) w = P.d_pairs[P.d_pair_base[r_first + lane] + q - g.x].w;
        }
        w = __reduce_max_sync(~0u, w);
        w = min(w, L / 2);
        if (w < 0) {
            if (lane == 0 && q - q_lo < nq_cap) sQ[q - q_lo] = -1;
            continue;
        }
        const Window g = tile_window(w, L);
        if (lane == 0) {  // the host sized both for every tile: never expected
            if (q - q_lo < nq_cap && 16 * (g.s1 - g.s0) <= wpos_cap)
                sQ[q - q_lo] = (short)(kTrim && (q < s_band_lo || q > s_band_hi) ? -1 : w);
            else s_bad = 1;
            if (kTrim && q > s_band_hi) atomicAdd(&s_tail, 1);
        }
        const int start = P.d_rings[q].start;
        // pixels [a, a + len) of the ring, wrapped; every block of 64 map pixels in them
        const int len = min(8 * plan_cols + 16 * (g.s1 - g.s0), L);
        int a = (plan_k0 + g.d0 + 16 * g.s0) % L;
        a += a < 0 ? L : 0;
        const int head = min(len, L - a);
        uint32_t qmax = 0u, qmin = 0xffffffffu;
        for (int part = 0; part < 2; ++part) {
            const int p0 = start + (part ? 0 : a), p1 = start + (part ? len - head : a + head);
            if (p1 <= p0) continue;
            for (int b = (p0 >> 6) + lane; b <= (p1 - 1) >> 6; b += 32) {
                const uint32_t v = __ldg(bm + b);
                qmax = max(qmax, v);
                if (v) qmin = min(qmin, v);
            }
        }
        qmax = __reduce_max_sync(~0u, qmax);
        qmin = __reduce_min_sync(~0u, qmin);
        vmax = max(vmax, qmax);
        vmin = min(vmin, qmin);
        // A constant taken off the ring where its blocks are all within a factor of four of the
        // largest: near the mean of 128 of its pixels, a multiple of 2^-3 of the largest value's
        // power of two, where it is at least two of them (not for maps about zero).
        unsigned short shift = 0;
        if (qmax != 0u && qmax < 0x7f800000u && qmax >= 0x02000000u && (qmax >> 23) - (qmin >> 23) <= 1u) {
            float v = 0.0f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                int i = a + (int)((4u * lane + j) * (unsigned)len / 128u);
                i -= i >= L ? L : 0;
                v += __ldg(m + start + i);
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(~0u, v, s);
            const float quantum = __uint_as_float(((qmax >> 23) - 3u) << 23);
            v = rintf(v * (1.0f / 128.0f) / quantum) * quantum;
            if (fabsf(v) >= 2.0f * quantum) shift = (unsigned short)(__float_as_uint(v) >> 16);  // (five digits: exact)
        }
        if (lane == 0 && q - q_lo < nq_cap) {
            sC[q - q_lo] = shift;
            if (shift & 0x7fffu) s_shift = 1;
        }
    }
    vmax = __reduce_max_sync(~0u, vmax);
    vmin = __reduce_min_sync(~0u, vmin);
    if (lane == 0) {
        atomicMax(&s_max, vmax);
        atomicMin(&s_min, vmin);
    }
    if (warp == kRings) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         tc::saddr(&tmem_base)),
                     "r"(kTmem));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_base;
    const uint32_t emax = s_max >> 23, emin = s_min >> 23;  // biased exponents
    const bool zero = s_max == 0u;
    // scales stay normal floats: exponents of 2^(14 - e) within [-126, 127]
    const bool flag = !zero && (emax >= 255u || emax < 48u || emax > 206u || emin == 0u ||
                                emax - emin > kRangeExp);
    if (tid == 0) {
        flags[(long long)blockIdx.y * n_tiles + rb * (L / (8 * plan_cols)) + plan_tile] = flag ? 1 : 0;
        if (s_bad) atomicExch(err, KSC_ERR_DEVICE_BOUNDS);
    }
    // |m - constant| may reach twice the largest |m|
    const uint32_t ex = emax + (s_shift ? 1u : 0u);
    const float xscale = zero || flag ? 1.0f : __uint_as_float((127u + kXExp + 127u - ex) << 23);
    const float xunscale = zero || flag ? 1.0f : __uint_as_float((ex - kXExp) << 23);
    bool drained = true;  // no MMA in flight can still write tensor memory

    if (flag || s_bad) {
        // left to the FFMA kernel (or never expected)
    } else if (warp >= kRings) {
        // ---- the issuing warp
        if constexpr (N == 256) asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
        if (warp == kRings && lane == 0) {
            const uint32_t idesc = idesc_f16(128, N);
            const uint32_t pa0 = tc::saddr(sA), pb0 = tc::saddr(sB);
            const uint64_t a_hi = tc::desc(0, 128, kChunk * 16), b_hi = tc::desc(0, 16, 128);
            const uint32_t a_l = kPartBytes >> 4, b_l = (uint32_t)(seg_cap * 2) >> 4;
            uint32_t n_rings = 0, n_chunks = 0;
            bool ok = true;
            for (int qi = 0; qi < nq && ok; ++qi) {
                const int w = sQ[qi];
                if (w < 0) continue;
                const Window g = tile_window(w, L);
                const uint32_t b = n_rings & 1u;
                const uint32_t d = tmem + b * N;
                uint32_t acc = n_rings >= 2 ? 1u : 0u;
                const int c_lo = g.s0 / kSteps, c_hi = (g.s1 - 1) / kSteps;
                for (int cc = c_lo; cc <= c_hi; ++cc, ++n_chunks) {
                    const int c = chunk_of(cc, c_hi, g.mid);
                    const uint32_t st = n_chunks & 1u;
                    if (!wait_or_abort(&a_full[st], (n_chunks >> 1) & 1u, &s_abort)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    const int t0 = max(g.s0, kSteps * c), t1 = min(g.s1, kSteps * c + kSteps);
                    // descriptors of step s: the stage's A at 256 s bytes, B at 32 s bytes
                    const uint64_t da0 = a_hi + ((pa0 + st * kStageBytes) >> 4);
                    const uint64_t db0 = b_hi + ((pb0 + b * 4 * seg_cap) >> 4);
                    auto da = [&](int s) { return da0 + (uint32_t)((s - kSteps * c) * 16); };
                    auto db = [&](int s) { return db0 + (uint32_t)((s - g.s0) * 2); };
                    const int s_c = kSteps * c + kSteps / 2;  // the closest approach's step
                    if (c == g.mid && s_c >= t0 && s_c < t1) {
                        mma_f16(d, da(s_c) + a_l, db(s_c) + b_l, idesc, acc);
                        acc = 1u;
                    }
                    for (int s = t0; s < t1; ++s) {
                        mma_f16(d, da(s), db(s) + b_l, idesc, acc);
                        mma_f16(d, da(s) + a_l, db(s), idesc, 1u);
                        acc = 1u;
                    }
                    if (c == g.mid) {  // from the ends to the closest approach
                        for (int e = 0; e < kSteps; ++e) {
                            const int s = kSteps * c + ((e & 1) ? kSteps - 1 - (e >> 1) : e >> 1);
                            if (s >= t0 && s < t1) mma_f16(d, da(s), db(s), idesc, 1u);
                        }
                    } else {
                        for (int s = t0; s < t1; ++s) mma_f16(d, da(s), db(s), idesc, 1u);
                    }
                    tc::mma_commit(&a_free[st]);
                }
                if (!ok) break;
                tc::mma_commit(&d_done[b]);
                ++n_rings;
            }
            // every MMA has ended before the tensor memory goes (after an abort: bounded)
            if (n_chunks > 0 && !ok)
                drained = tc::mbar_wait(&a_free[(n_chunks - 1) & 1u], ((n_chunks - 1) >> 1) & 1u);
        }
        __syncwarp();
    } else {
        // ---- builder warps
        // 640 x 96 registers at launch = 512 x 112 + 128 x 32
        if constexpr (N == 256) asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        // this thread's accumulators: lane quarter warp & 3, columns (warp >> 2) kCols ..
        const uint32_t td =
            tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * kCols);
        uint32_t *wr = sW + warp * w_cap;
        const int my_r = r_first + warp;  // the ring this warp builds weights for
        int2 rg = make_int2(P.belt_hi + 1, P.belt_lo - 1);
        int base = 0, my_phase = 0;
        if (warp < n_rows && my_r >= ring_lo && my_r <= ring_hi) {  // (no weights for other rings)
            rg = P.d_range[my_r];
            base = P.d_pair_base[my_r] - rg.x;
            my_phase = P.d_rings[my_r].phase;
        }
        uint64_t tot[kCols / 2];
#pragma unroll
        for (int c = 0; c < kCols / 2; ++c) tot[c] = 0ull;
        float wsum = 0.0f, wcomp = 0.0f;
        uint32_t n_rings = 0, n_chunks = 0;
        bool ok = true;

        // fold the accumulator of ring n into the totals, leaving in it the sums' rounding
        // errors and the 2^-24 that the MMAs' cuts cost on average
        auto drain = [&](uint32_t n, bool multiplied = true) {
            const uint32_t b = n & 1u;
            if (multiplied) {
                if (!__all_sync(~0u, wait_or_abort(&d_done[b], (n >> 1) & 1u, &s_abort))) return false;
                tc::fence_after_sync();
            }
            const uint64_t m1 = pack2(0xbf800000u, 0xbf800000u);  // -1
            const uint64_t cut = pack2(0x33800000u, 0x33800000u);  // 2^-24
            uint32_t v[kStep];
#pragma unroll
            for (int c = 0; c < kCols; c += kStep) {
                const uint32_t t = td + b * N + c;
                __syncwarp();
                if constexpr (kStep == 16) tc::tmem_ld16(t, v); else tmem_ld8(t, v);
                tc::loaded(v);
#pragma unroll
                for (int e = 0; e < kStep; e += 2) {
                    const uint64_t y = pack2(v[e], v[e + 1]), t0 = tot[(c + e) / 2];
                    const uint64_t s = add2(t0, y);
                    const uint64_t r = fma2(y, cut, fma2(fma2(t0, m1, s), m1, y));
                    tot[(c + e) / 2] = s;
                    v[e] = (uint32_t)r;
                    v[e + 1] = (uint32_t)(r >> 32);
                }
                if constexpr (kStep == 16) tc::tmem_st16(t, v); else tmem_st8(t, v);
            }
            tc::tmem_wait_st();
            tc::fence_before_sync();
            return true;
        };

        for (int qi = 0; qi < nq; ++qi) {
            const int w = sQ[qi];
            if (w < 0) continue;
            const int q = q_lo + qi;
            const uint32_t b = n_rings & 1u;
            const Window g = tile_window(w, L);
            const int n_pos = 16 * (g.s1 - g.s0);
            const DevRing *Q = P.d_rings + q;
            PairInfo pi;
            pi.w = -1;
            if (q >= rg.x && q <= rg.y) pi = P.d_pairs[base + q];
            const int tdiff = my_phase - Q->phase;
            const float shift = __uint_as_float((uint32_t)sC[qi] << 16);
            const float moff = -shift * xscale;
            // ---- the input segment, scaled and split into two FP16 parts
            {
                int a = (k0 + g.d0 + 16 * g.s0) % L;
                a += a < 0 ? L : 0;
                const float *ring = m + Q->start;
                __half2 *bh = reinterpret_cast<__half2 *>(sB + b * 2 * seg_cap);
                __half2 *bl = bh + seg_cap / 2;
                const int n2 = (8 * N + n_pos) / 2;
                auto load = [&](int e, float *x0, float *x1) {
                    int i = a + 2 * e;
                    while (i >= L) i -= L;
                    *x0 = __ldg(ring + i);
                    *x1 = __ldg(ring + (i + 1 == L ? 0 : i + 1));
                };
                auto put = [&](int e, float x0, float x1) {
                    const float y0 = fmaf(x0, xscale, moff), y1 = fmaf(x1, xscale, moff);
                    const __half2 h = __floats2half2_rn(y0, y1);
                    const float2 f = __half22float2(h);
                    bh[e] = h;
                    bl[e] = __floats2half2_rn(y0 - f.x, y1 - f.y);
                };
                int e = tid;
                for (; e + kT < n2; e += 2 * kT) {  // two pairs of loads in flight
                    float x0, x1, y0, y1;
                    load(e, &x0, &x1);
                    load(e + kT, &y0, &y1);
                    put(e, x0, x1);
                    put(e + kT, y0, y1);
                }
                if (e < n2) {
                    float x0, x1;
                    load(e, &x0, &x1);
                    put(e, x0, x1);
                }
            }
            // ---- this warp's ring: its weights over the tile's window, Delta at element
            // x = Delta + x_of; all of 0 .. n_x - 1 are written
            {
                const int x_of = 8 - g.d0 - 16 * g.s0;
                const int n_x = n_pos + 16;
                const bool whole = 2 * pi.w + 1 >= L;
                const int lo = whole ? -(L / 2) : -pi.w, hi = whole ? lo + L - 1 : pi.w;
                // w(Delta) = w(tdiff - Delta): both from one evaluation, but for whole rings
                const int d_first = whole ? -x_of : (tdiff + 1) >> 1;
                const int n_d =
                    whole ? n_x : max(n_x - x_of - d_first, tdiff + x_of - d_first + 1);
                const DF A{pi.Ah, pi.Al}, B{pi.Bh, pi.Bl};
                // weight (scaled) and the scaled rounding error of its last addition
                auto weight = [&](int d, float *we) {
                    const float mf = (float)(tdiff - 2 * d);
                    const float xh = mf * P.belt_c1h;
                    const float xl = fmaf(mf, P.belt_c1h, -xh) + mf * P.belt_c1l;
                    int ti;
                    float f;
                    const bool in = chord_to_table_sel(A, B, sin_df(xh, xl), P.nint2, &ti, &f) &&
                                    d >= lo && d <= hi;  // (no ring in reach: hi < lo)
                    const float4 c = __ldg(&P.d_tab[min(ti, P.n_int - 1)]);
                    const float t = f * fmaf(f, fmaf(f, c.w, c.z), c.y);
                    const float v = c.x + t, bb = v - c.x;
                    *we = in ? ((c.x - (v - bb)) + (t - bb)) * wscale : 0.0f;
                    return in ? v * wscale : 0.0f;
                };
                auto put = [&](int i, float v, float ve) {
                    const int x = d_first + i + x_of, y = tdiff - d_first - i + x_of;
                    const __half h = __float2half_rn(v);
                    const __half l = __float2half_rn((v - __half2float(h)) + ve);
                    const uint32_t hl = (uint32_t)__half_as_ushort(l) << 16 | __half_as_ushort(h);
                    if (x < n_x) wr[x] = hl;
                    if (!whole && y >= 0) wr[y] = hl;
                    if (shift != 0.0f) {  // sum of weight x constant (Kahan)
                        const float z = (!whole && y != x ? 2.0f : 1.0f) * (v * shift) - wcomp, t = wsum + z;
                        wcomp = (t - wsum) - z;
                        wsum = t;
                    }
                };
                __syncwarp();
                int i = lane;
                if (pi.w < 0) {
                    for (; i < n_x; i += 32) wr[i] = 0u;
                } else {
                    for (; i + 32 < n_d; i += 64) {  // two evaluations in flight
                        float e0, e1;
                        const float v0 = weight(d_first + i, &e0), v1 = weight(d_first + i + 32, &e1);
                        put(i, v0, e0);
                        put(i + 32, v1, e1);
                    }
                    if (i < n_d) {
                        float e0;
                        const float v0 = weight(d_first + i, &e0);
                        put(i, v0, e0);
                    }
                }
                __syncwarp();
            }
            // ---- A, chunk by chunk
            const int c_lo = g.s0 / kSteps, c_hi = (g.s1 - 1) / kSteps;
            for (int cc = c_lo; cc <= c_hi; ++cc, ++n_chunks) {
                const int c = chunk_of(cc, c_hi, g.mid);
                const uint32_t st = n_chunks & 1u;
                if (n_chunks >= kStages &&
                    !__all_sync(~0u,
                                wait_or_abort(&a_free[st], ((n_chunks >> 1) - 1u) & 1u, &s_abort))) {
                    ok = false;
                    break;
                }
                const int t0 = max(g.s0, kSteps * c), t1 = min(g.s1, kSteps * c + kSteps);
                unsigned char *sa = sA + st * kStageBytes + warp * (kChunk * 16) +
                                    (t0 - kSteps * c) * 256;
                const uint32_t *src = wr + 8 + 16 * (t0 - g.s0);
                // core matrix e / 8, row e % 8: eight weights from element 8 (e / 8) - e % 8
                for (int e = lane; e < 16 * (t1 - t0); e += 32) {
                    const uint32_t *p = src + 8 * (e >> 3) - (e & 7);
                    uint32_t v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = p[j];
                    *reinterpret_cast<uint4 *>(sa + 16 * e) =
                        make_uint4(__byte_perm(v[0], v[1], 0x5410), __byte_perm(v[2], v[3], 0x5410),
                                   __byte_perm(v[4], v[5], 0x5410), __byte_perm(v[6], v[7], 0x5410));
                    *reinterpret_cast<uint4 *>(sa + kPartBytes + 16 * e) =
                        make_uint4(__byte_perm(v[0], v[1], 0x7632), __byte_perm(v[2], v[3], 0x7632),
                                   __byte_perm(v[4], v[5], 0x7632), __byte_perm(v[6], v[7], 0x7632));
                }
                tc::fence_async_smem();
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&a_full[st]);
            }
            if (!ok) break;
            ++n_rings;
            // the previous ring's accumulator while this ring's MMAs run
            if (n_rings >= 2 && !(ok = drain(n_rings - 2))) break;
        }
        // the last ring's accumulator, and the folds of the rings after (n_used accumulators are in
        // use: two, or one after a single ring)
        const uint32_t n_used = n_rings;
        for (int i = 0; i <= (kTrim ? s_tail : 0) && n_used > 0 && ok; ++i) {
            const uint32_t n = n_used - 1u + i;
            if (i == 0 || (n & 1u) < n_used) ok = drain(n, i == 0);
        }
        if (s_shift) {  // every builder warp comes here, after an abort too
            wsum -= wcomp;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) wsum += __shfl_xor_sync(~0u, wsum, s);
            if (lane == 0) s_wsum[warp] = wsum * wunscale;
            asm volatile("bar.sync 1, %0;" ::"r"(kT) : "memory");
        }
        if (ok) {
            // out = domega (unscale (total + what its folds still owe) + sum of weight x constant)
            const int row = (warp & 3) * 32 + lane, rr = r_first + (row >> 3);
            const bool live = (row >> 3) < n_rows && rr >= ring_lo && rr <= ring_hi;
            float *dst = o + start0 + (row >> 3) * L + k0 + (row & 7) + (warp >> 2) * kCols * 8;
            const float unscale = xunscale * wunscale;
            const float base_v = s_shift ? s_wsum[row >> 3] : 0.0f;
#pragma unroll
            for (int c = 0; c < kCols; c += 8) {
                uint32_t v0[8], v1[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v0[e] = v1[e] = 0u;
                if (n_used >= 1) tmem_ld8(td + c, v0);
                if (n_used >= 2) tmem_ld8(td + N + c, v1);
                tc::loaded(v0);
                tc::loaded(v1);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint64_t tt = tot[(c + e) / 2];
                    const float r = (__uint_as_float(v0[e]) + __uint_as_float(v1[e])) * unscale;
                    const float t = __uint_as_float((e & 1) ? (uint32_t)(tt >> 32) : (uint32_t)tt) * unscale;
                    const float hi = t + base_v;  // two-sum
                    const float bb = hi - t;
                    const float lo = ((t - (hi - bb)) + (base_v - bb)) + r;
                    if (live) dst[8 * (c + e)] = fmaf(hi, P.domega, fmaf(hi, domega_lo, lo * P.domega));
                }
            }
        }
    }
    tc::fence_before_sync();
    const bool all_drained = __syncthreads_and(drained);
    if (s_abort && tid == 0) atomicExch(err, all_drained ? KSC_ERR_TIMEOUT : KSC_ERR_TIMEOUT_UNDRAINED);
    // tensor memory that an MMA may still write is not freed
    if (warp == kRings && all_drained)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmem));
}

// blockmax[map][b] = the bits of the largest |m| over map pixels [64 b, 64 b + 64)
// (infinities and NaNs compare above every number), for the blocks of the reach (a band reads
// its own part of the map: nine belt rings of nside 2048, 4 pixels: 36 us for the whole map).
// One read of them.  Clears the n_zero words that the call's later kernels count and flag in.
__global__ void __launch_bounds__(256)
block_max_kernel(const MapSet maps, int b0, int n0, int b1, int n1,
                 uint32_t *__restrict__ blockmax, long long block_stride, int *__restrict__ zero, long long n_zero) {
    for (long long i = (blockIdx.y * (long long)gridDim.x + blockIdx.x) * 256 + threadIdx.x;
         i < n_zero; i += (long long)gridDim.x * gridDim.y * 256)
        zero[i] = 0;
    const float4 *m = reinterpret_cast<const float4 *>(maps.input(blockIdx.y));
    uint32_t *bm = blockmax + (long long)blockIdx.y * block_stride;
    const int half = (blockIdx.x * 256 + threadIdx.x) >> 4, l16 = threadIdx.x & 15;
    const int n_half = gridDim.x * 16;
    for (int i = half; i < n0 + n1; i += n_half) {
        const int b = i < n0 ? b0 + i : b1 + (i - n0);
        const float4 v = __ldg(m + (long long)b * 16 + l16);
        uint32_t x = max(max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu),
                         max(__float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu));
        const uint32_t mask = 0xffffu << (threadIdx.x & 16);
        x = __reduce_max_sync(mask, x);
        if (l16 == 0) bm[b] = x;
    }
}

template <int N>
size_t tc_smem(int wpos, int nq) {
    return (size_t)kStages * kStageBytes + 2 * 4 * (size_t)(8 * N + wpos) +
           4 * (size_t)kRings * (wpos + 16) + 4 * (size_t)((nq + 1) & ~1);
}

template <int N>
cudaError_t launch_tc(const ConvPlan &p, const BeltTc &t, const MapSet &maps, int n_maps,
                      int r0, int r1, const uint32_t *bm,
                      long long bm_stride, unsigned char *flags, int *d_err, cudaStream_t st) {
    const int lo = std::max(r0, p.belt_lo), hi = std::min(r1, p.belt_hi);
    const int b0 = (lo - p.belt_lo) / kRings, b1 = (hi - p.belt_lo) / kRings;
    const int tk = p.nside / (2 * N);
    const size_t smem = tc_smem<N>(t.wpos, t.nq);
    cudaError_t e = cudaFuncSetAttribute(conv_belt_tc_kernel<N>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kMaxDynSmem);  // (one value: calls may race)
    if (e != cudaSuccess) return e;
    dim3 grid((b1 - b0 + 1) * tk, n_maps);
    conv_belt_tc_kernel<N><<<grid, kThreads, smem, st>>>(
        p, b0, tk, r0, r1, maps, bm, bm_stride, flags, belt_tc_tiles(p, t),
        t.n_cols, t.wpos, t.nq, t.wscale, 1.0f / t.wscale,
        (float)(4.0 * 3.14159265358979323846 / p.npix - (double)p.domega), d_err);
    return cudaGetLastError();
}

} // namespace

int belt_tc_rings() { return kRings; }

int belt_tc_tiles(const ConvPlan &p, const BeltTc &t) {
    return ((p.belt_hi - p.belt_lo) / kRings + 1) * (p.nside / (2 * t.n_cols));
}

int belt_tc_positions(int w, int L) {
    const Window g = tile_window(std::min(w, L / 2), L);
    return 16 * (g.s1 - g.s0);
}

bool belt_tc_plan(int nside, int wpos, int nq, BeltTc *t) {
    t->n_cols = 0;
    if (nside < 64 || wpos <= 0) return false;
    t->wpos = wpos;
    t->nq = nq;
    const int n_blocks = (2 * nside + kRings) / kRings;
    double best = 0.0;
    for (int n = 32; n <= 256 && 2 * n <= nside; n *= 2) {
        const size_t smem = n == 256 ? tc_smem<256>(wpos, nq) : n == 128 ? tc_smem<128>(wpos, nq)
                            : n == 64 ? tc_smem<64>(wpos, nq) : tc_smem<32>(wpos, nq);
        if (smem > (size_t)kMaxDynSmem) continue;
        // waves of one CTA per SM x the larger of the MMAs' and the builders' cycles
        const double waves = std::ceil(n_blocks * (nside / (2.0 * n)) / 152.0);
        const double mma = wpos / 16.0 * 3.0 * std::max(n / 2.0, 48.0);
        const double build = 500.0 + wpos * 12.0 + n * 6.0;
        const double cost = waves * std::max(mma, build);
        if (t->n_cols == 0 || cost < best) {
            best = cost;
            t->n_cols = n;
        }
    }
    return t->n_cols > 0;
}

TcCuts tc_cuts(const RingGeom &g, int nside, double chord_cut, const float4 *tab, int n_int) {
    // For uncorrelated input a partial sum's variance V_j is that of its weights.  A cut takes 0.75
    // of 2^-24 of the sum on average (measured), the fold gives one 2^-24 of the final sum
    // back: what is left has the mean square sum min(V_i, V_j) - 2 (4/3) sum V_j + (4/3)^2 V.
    // The rings past 24 by one in `step`, the eight offsets of a core matrix by their middle.
    struct Walk {
        double v = 0.0, sum = 0.0, square = 0.0;
        void cut(double n = 1.0) {
            square += n * (2.0 * sum + n * v);
            sum += n * v;
        }
        double left() const { return square - 8.0 / 3.0 * sum + 16.0 / 9.0 * v; }
    };
    const int L = 4 * nside, r = 2 * nside - 1;
    const double pi = 3.14159265358979323846;
    const int reach = std::min((int)std::ceil(asin(std::min(1.0, chord_cut / 2.0)) * 3.0 * nside) + 1, nside);
    const int step = std::max(1, reach / 96);
    double total = 0.0;
    TcCuts out;
    for (int dq = 0; dq <= reach; dq += dq < 24 ? 1 : step) {
        const int q = r + dq;
        const double dz = g.z[q] - g.z[r], ds = g.s[q] - g.s[r], a = dz * dz + ds * ds, b = 4.0 * g.s[q] * g.s[r];
        const double left = chord_cut * chord_cut - a;
        if (left <= 0.0) break;
        const double half = left >= b ? 0.5 * pi : asin(sqrt(left / b));
        const int w = std::min((int)std::ceil(half * L / pi) + 1, L / 2);
        auto energy = [&](const Window &win, int s) {
            const double shift = 0.5 * (g.phase[q] - g.phase[r]) - 3.5 + win.d0 + 16 * s;
            double e = 0.0;
            for (int j = 0; j < 16; ++j) {
                const double h = sin(pi * (shift + j) / L), d2 = a + b * h * h;
                if (d2 > chord_cut * chord_cut) continue;
                const double u = sqrt(d2) * (n_int / chord_cut);
                const int i = std::min((int)u, n_int - 1);
                const double f = u - i, v = tab[i].x + f * (tab[i].y + f * (tab[i].z + f * (double)tab[i].w));
                e += v * v;
            }
            return e;
        };
        // the order of the issuing warps: the belt's, small products of a chunk first ...
        Walk belt, cap;
        const Window wb = tile_window(w, L);
        const int b_hi = (wb.s1 - 1) / kSteps;
        for (int cc = wb.s0 / kSteps; cc <= b_hi; ++cc) {
            const int c = chunk_of(cc, b_hi, wb.mid);
            const int t0 = std::max(wb.s0, kSteps * c), t1 = std::min(wb.s1, kSteps * c + kSteps);
            belt.cut(2 * (t1 - t0) + (c == wb.mid ? 1 : 0));
            for (int e = 0; e < kSteps; ++e) {
                const int s = kSteps * c + (c == wb.mid ? ((e & 1) ? kSteps - 1 - (e >> 1) : e >> 1) : e);
                if (s < t0 || s >= t1) continue;
                belt.v += energy(wb, s);
                belt.cut();
            }
        }
        // ... and the caps', whose small products have an accumulator of their own
        const Window wc = tc::tile_window<32>(w, L);
        const int c_hi = (wc.s1 - 1) / 2;
        for (int cc = wc.s0 / 2; cc <= c_hi; ++cc) {
            const int c = chunk_of(cc, c_hi, wc.mid);
            for (int s = std::max(wc.s0, 2 * c); s < std::min(wc.s1, 2 * c + 2); ++s) {
                cap.v += energy(wc, s);
                cap.cut();
            }
        }
        const double weight = (dq == 0 ? 1.0 : 2.0) * (dq > 24 ? step : 1);
        total += weight * belt.v;
        out.belt += weight * belt.left();
        out.cap += weight * cap.left();
    }
    if (total > 0.0) {
        out.belt /= total;
        out.cap /= total;
    }
    return out;
}

long long map_blocks(const ConvPlan &p) { return p.npix / 64; }

cudaError_t launch_block_max(const ConvPlan &p, const MapSet &maps, int n_maps,
                             const InputReach &in, uint32_t *bm, int *zero, long long n_zero,
                             cudaStream_t st) {
    const int n = in.n0 + in.n1;
    dim3 grid(std::max(1, std::min((n + 15) / 16, 152 * 8)), n_maps);
    block_max_kernel<<<grid, 256, 0, st>>>(maps, in.b0, in.n0, in.b1, in.n1, bm, map_blocks(p), zero,
                                           n_zero);
    return cudaGetLastError();
}

cudaError_t launch_conv_belt_tc(const ConvPlan &p, const BeltTc &t, const MapSet &maps,
                                int n_maps, int r0, int r1, const uint32_t *bm, unsigned char *flags,
                                int *d_err, cudaStream_t st) {
    if (r0 > p.belt_hi || r1 < p.belt_lo) return cudaSuccess;
    const long long bs = map_blocks(p);
    // Narrower tiles while twice as many are still one wave (one CTA per SM): nine rings of
    // nside 2048, 64 pixels: 0.92 -> 0.54 ms (FFMA 0.50), 16 pixels: 0.31 -> 0.17 (0.09).
    const int nb = (std::min(r1, p.belt_hi) - p.belt_lo) / kRings - (std::max(r0, p.belt_lo) - p.belt_lo) / kRings + 1;
    int n = t.n_cols;
    while (n > 32 && 2ll * nb * (p.nside / (2 * n)) * n_maps <= 152) n /= 2;
    switch (n) {
    case 256: return launch_tc<256>(p, t, maps, n_maps, r0, r1, bm, bs, flags, d_err, st);
    case 128: return launch_tc<128>(p, t, maps, n_maps, r0, r1, bm, bs, flags, d_err, st);
    case 64: return launch_tc<64>(p, t, maps, n_maps, r0, r1, bm, bs, flags, d_err, st);
    default: return launch_tc<32>(p, t, maps, n_maps, r0, r1, bm, bs, flags, d_err, st);
    }
}

} // namespace ksc
