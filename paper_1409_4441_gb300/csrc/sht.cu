// The harmonic half of the split convolution on the GPU (Fig. 1's CPU half; an
// option of this library): spherical-harmonic synthesis and analysis of HEALPix
// RING maps up to l_max, m <= l_max, real fields, declared in include/ksconv.h.
//
//   synthesis  m_p = sum_l a_l0 lambda_l0(z) + 2 Re sum_{m>0} G_m(z) e^{i m phi},
//              G_m(z) = sum_l a_lm lambda_lm(z);
//   analysis   a_lm = (4 pi / Npix) sum_rings lambda_lm(z) F_m(ring),
//              F_m = sum_k m_k e^{-i m phi_k}.
//
// lambda_lm are the normalised associated Legendre functions without the
// Condon-Shortley phase, from their three-term recurrence in l at fixed m
// (lambda_mm = sqrt((2m+1)/4pi prod_{k<=m} (2k-1)/2k) sin^m theta; lambda_{m+1,m}
// = sqrt(2m+3) z lambda_mm; lambda_lm = A_l (z lambda_{l-1,m} - lambda_{l-2,m} /
// A_{l-1}), A_l = sqrt((4l^2-1)/(l^2-m^2))).  The recurrence and the sums over l and over
// rings run on FP32 pairs (hi + lo, 48 bits): the FP64 units of a GB300 do 1/64 of its FP32
// operations, and FP64 recurrences took 100 of the 154 ms of both transforms at nside 2048,
// l_cut 1024.  After a few thousand steps a pair is still within 1e-10, far inside the FP32
// that the ring sums keep.  Near the poles sin^m theta underflows any floating format, so
// values are carried as v 2^(120 e) and summed only once e reaches 0 (while e < 0 the
// true value is below 2^-60).  North and south rings share |z| (lambda_lm(-z) = (-1)^(l+m)
// lambda_lm(z)), so each recurrence serves a ring pair through its even and odd partial
// sums.  Orders beyond l sin theta + 16 + 9 l^(1/3) stay below 2^-60 for every l <= l_max (the
// functions decay exponentially past their turning point): a ring leaves them out.
//
// Ring sums: pixel k of a ring of L pixels with phase flag t sits at phi_k = pi (2k + t) / L.
// Belt rings (L = 4 nside, a power of two) of larger transforms go through an FP32 FFT in shared
// memory, a ring and its mirror a block.  Other rings (L = 4i) are summed directly over a
// quarter: the quarter turns of pixel k1 enter order m through m mod 4 alone.  m phi_k =
// pi J / L with the exact integer J = m (2k + t) mod 2L; the twiddles advance by one complex
// product per step and are re-anchored from the exact J every 8 steps (the products'
// rounding drifts by about one FP32 ulp per step in between).
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "ksc_internal.h"

namespace ksc {
namespace {

constexpr double kPi = 3.14159265358979323846;
constexpr int kAnchor = 8;        // twiddle steps between exact re-anchors

__host__ __device__ inline long long n_alm(int lmax) {
    return (long long)(lmax + 1) * (lmax + 2) / 2;
}
__host__ __device__ inline long long alm_base(int lmax, int m) {  // index(0, m)
    return (long long)m * (2 * lmax + 1 - m) / 2;
}

// Ring r (0-based) of nside n: pixel count, first pixel, phase flag.
struct ShtRing {
    int len, start, t;
};
__device__ __forceinline__ ShtRing sht_ring(int n, int r) {
    const int i = r + 1;
    if (i < n) return {4 * i, 2 * i * (i - 1), 1};
    if (i <= 3 * n) return {4 * n, 2 * n * (n - 1) + 4 * n * (i - n), (i - n) % 2 == 0 ? 1 : 0};
    const int ip = 4 * n - i;
    return {4 * ip, 12 * n * n - 2 * ip * (ip + 1), 1};
}

// ---- FP32 pairs (hi + lo) -----------------------------------------------------
struct F2 {
    float h, l;
};
__device__ __forceinline__ F2 f2_of(double v) {
    F2 r;
    r.h = (float)v;
    r.l = (float)(v - (double)r.h);
    return r;
}
__device__ __forceinline__ F2 f2_norm(float h, float l) {
    F2 r;
    r.h = h + l;
    r.l = l - (r.h - h);
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {  // not normalised: |l| a few ulps of h
    F2 r;
    r.h = a.h * b.h;
    r.l = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -r.h)));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    const float s = a.h + b.h, t = s - a.h;
    return f2_norm(s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l));
}

__device__ __forceinline__ F2 f2_of(int v) {  // |v| below 2^30, exact
    F2 r;
    r.h = __int2float_rn(v);
    r.l = (float)(v - __float2int_rn(r.h));
    return r;
}
__device__ __forceinline__ F2 f2_div(F2 a, F2 b) {
    const float q = a.h / b.h;
    return f2_norm(q, (fmaf(-q, b.h, a.h) + fmaf(-q, b.l, a.l)) / b.h);
}
__device__ __forceinline__ F2 f2_sqrt(F2 a) {
    const float q = sqrtf(a.h);
    return q > 0.0f ? f2_norm(q, (fmaf(-q, q, a.h) + a.l) * (0.5f / q)) : F2{0.0f, 0.0f};
}
__device__ __forceinline__ F2 f2_sum(float a, float b) {  // a + b exactly
    const float s = a + b, t = s - a;
    return F2{s, (a - (s - t)) + (b - t)};
}
// s + p with s.l left to collect the rounding errors (folded in at the end): three operations
// less than f2_add, and |s.l| stays far below |s.h| over the few thousand terms of a sum.
__device__ __forceinline__ F2 f2_acc(F2 s, F2 p) {
    const float t = s.h + p.h, u = t - s.h;
    return F2{t, s.l + (((s.h - (t - u)) + (p.h - u)) + p.l)};
}

// z and sin(theta) of northern ring r (0-based) or the equator as pairs, from whole numbers
// below 2^30: in the cap 1 - z = i^2 / 3n^2, in the belt z = (4n - 2i) / 3n = a / 3n and
// sin^2 = (3n - a)(3n + a) / 9n^2.  (In FP64 the rings, powers and
// coefficients of a block cost as much as its recurrences: 36 and 26 us for the two Legendre
// kernels at nside 128, l_max 64, against 26 and 16 us.)
__device__ __forceinline__ void ring_zs(int n, int r, F2 *z, F2 *s) {
    const int i = r + 1;
    if (i < n) {
        const F2 w = f2_div(f2_of(i * i), f2_of(3 * n * n));
        *z = f2_add(F2{1.0f, 0.0f}, F2{-w.h, -w.l});
        *s = f2_sqrt(f2_mul(w, f2_add(F2{2.0f, 0.0f}, F2{-w.h, -w.l})));
    } else {
        const int a = 4 * n - 2 * i, d = 3 * n;
        *z = f2_div(f2_of(a), f2_of(d));
        *s = f2_sqrt(f2_div(f2_of((d - a) * (d + a)), f2_of(d * d)));
    }
}

// Orders above this do not reach 2^-60 on northern ring r (see the top of the file).  Some kernels
// write G or F up to it and others read up to it, so it has to come out the same in all of
// them: every step is rounded on its own, whatever the compiler does around it.
__device__ __forceinline__ int ring_limit(int nside, int r, int lmax, float extra) {
    const int i = r + 1, n = nside, a = 4 * n - 2 * i, d = 3 * n;
    float s;
    if (i < n) {
        const float w = __fdiv_rn(__int2float_rn(i * i), __int2float_rn(3 * n * n));
        s = __fsqrt_rn(__fmul_rn(w, __fsub_rn(2.0f, w)));
    } else {
        s = __fsqrt_rn(__fdiv_rn(__int2float_rn((d - a) * (d + a)), __int2float_rn(d * d)));
    }
    return min(lmax, (int)__fmaf_rn(__int2float_rn(lmax), s, extra));
}
float order_extra(int lmax) { return 16.0f + 9.0f * std::cbrt((float)lmax); }

// lambda_mm / sin^m theta = sqrt((2m + 1) / 4pi C), C = prod_{k<=m} (2k - 1) / 2k: the product
// (a factor a lane, by all lanes of a warp), or the series of Gamma(m + 1/2) / Gamma(m + 1)
// for large m (the next term is below 1e-11).
__device__ inline F2 norm_mm(int m) {
    double c;
    if (m <= 32) {
        const int k = (threadIdx.x & 31) + 1;
        c = k <= m ? (2.0 * k - 1.0) / (2.0 * k) : 1.0;
        for (int o = 16; o > 0; o >>= 1) c *= __shfl_xor_sync(~0u, c, o);
        c *= c;
    } else {
        const double x = 1.0 / m;
        const double p = 1.0 + x * (-1.0 / 8 + x * (1.0 / 128 + x * (5.0 / 1024 + x * (-21.0 / 32768 +
                                                                  x * (-399.0 / 262144)))));
        c = x / kPi * p * p;
    }
    return f2_of(sqrt(sqrt(c) * ((2.0 * m + 1.0) / (4.0 * kPi))));
}

// x = mantissa 2^ex with the mantissa's high part in [1, 2)
__device__ __forceinline__ F2 f2_mant(F2 x, int *ex) {
    const int e = ((__float_as_int(x.h) >> 23) & 255) - 127;
    const float q = __int_as_float((127 - e) << 23);  // |e| stays below 100 here
    *ex += e;
    return F2{x.h * q, x.l * q};
}

// The recurrence of one (ring, order): v1 = lambda_{l}, v2 = lambda_{l-1}, both 2^(-120 e)
// times the true values.
struct Rec {
    F2 z, v1, v2;
    int e;
    // v1 = norm s^m by binary powers (relative error below m 2^-46)
    __device__ __forceinline__ void start(int m, F2 norm, F2 zz, F2 s) {
        z = zz;
        int ex = 0, eb = 0;
        F2 b = f2_mant(s, &eb), v = f2_mant(norm, &ex);
        for (int k = m; k; k >>= 1) {
            if (k & 1) {
                v = f2_mul(v, b);
                ex += eb;
                v = f2_mant(f2_norm(v.h, v.l), &ex);
            }
            b = f2_mul(b, b);
            eb *= 2;
            b = f2_mant(f2_norm(b.h, b.l), &eb);
        }
        // e = min(0, floor((ex + 60) / 120)): below 2^60 in v1, above 2^-60 once e = 0
        e = min(0, (ex + 60 - (ex + 60 < 0 ? 119 : 0)) / 120);
        const float q = __int_as_float((127 + ex - 120 * e) << 23);
        v1 = F2{v.h * q, v.l * q};
        v2 = F2{0.0f, 0.0f};
    }
    // lambda_{l+1} = A (z lambda_l - B lambda_{l-1}), c = A as a pair, B as a pair
    __device__ __forceinline__ void step(float4 c) {
        const F2 x = f2_mul(z, v1), y = f2_mul(F2{c.z, c.w}, v2);
        const float d = x.h - y.h, t = d - x.h;
        const F2 w{d, ((x.h - (d - t)) - (y.h + t)) + (x.l - y.l)};
        const F2 r = f2_mul(F2{c.x, c.y}, w);
        v2 = v1;
        v1 = f2_norm(r.h, r.l);
        if (e < 0 && fabsf(v1.h) >= 0x1p60f) {
            const float q = 0x1p-120f;
            v1.h *= q; v1.l *= q; v2.h *= q; v2.l *= q;
            ++e;
        }
    }
};

// Powers of two that take values of largest magnitude `top` (the high word of a double, the bits of
// a float) to [2^30, 2^31), where sums over degrees or rings and the low parts of the pairs stay in
// FP32's range, and back; 1 for zeros, infinities and NaN.
constexpr int kTopExp = 30;
__device__ __forceinline__ double pow2(int e) {  // |e| <= 1022
    return __hiloint2double((1023 + e) << 20, 0);
}
__device__ __forceinline__ int scale_exp_f64(int top_hi) {
    const int e = (top_hi >> 20) - 1023;
    return top_hi == 0 || e == 1024 ? 0 : max(min(kTopExp - e, 1022), -1022);
}
__device__ __forceinline__ int scale_exp_f32(unsigned top) {
    const int e = (int)(top >> 23) - 127;
    return top == 0u || e == 128 ? 0 : min(kTopExp - e, 126);
}

constexpr int kTile = 128;  // degrees whose coefficients a block stages at a time

// Coefficients of the step to degree l (l > m): A_l and B_l = 1 / A_{l-1} (0 at l = m + 1),
// A_l^2 = (4 l^2 - 1) / (l^2 - m^2), whole numbers below 2^28.
__device__ __forceinline__ float4 step_coeffs(int l, int m) {
    const F2 a = f2_sqrt(f2_div(f2_of(4 * l * l - 1), f2_of((l - m) * (l + m))));
    const int k = l - 1;
    const F2 b = f2_sqrt(f2_div(f2_of((k - m) * (k + m)), f2_of(4 * k * k - 1)));
    return make_float4(a.h, a.l, b.h, b.l);
}

// Synthesis, Legendre part: G[ring][m] = sum_l a_lm lambda_lm(z_ring) for the northern rings
// (and their southern mirrors) of the block's range and order m = blockIdx.y, a ring a
// thread.  Orders past a ring's limit are not written (nor read).  Bound by issue: 47 FP32
// operations per ring pair, degree and order.  nside 2048, l_max 1024: 30.1 ms in FP64,
// 3.77 ms (two rings a thread for the same staged coefficients: 3.77; nside 512: 1.01
// against 1.04).
__global__ void __launch_bounds__(256)
sht_leg_synth(int nside, int lmax, float extra, const double2 *__restrict__ alm, float2 *__restrict__ G) {
    __shared__ float4 co[kTile], al[kTile];
    __shared__ F2 s_norm;
    __shared__ int s_top[8];
    const int m = blockIdx.y, nnorth = 2 * nside, nr = 4 * nside - 1;
    const int r = blockIdx.x * 256 + threadIdx.x, rs = nr - 1 - r;
    const double2 *a = alm + alm_base(lmax, m);
    int top = 0;  // largest |re|, |im| of the order's coefficients
    for (int l = m + threadIdx.x; l <= lmax; l += 256) {
        const double2 c = __ldg(a + l);
        top = max(top, max(__double2hiint(fabs(c.x)), __double2hiint(fabs(c.y))));
    }
    top = __reduce_max_sync(~0u, top);
    if ((threadIdx.x & 31) == 0) s_top[threadIdx.x >> 5] = top;
    if (threadIdx.x < 32) {
        const F2 v = norm_mm(m);
        if (threadIdx.x == 0) s_norm = v;
    }
    __syncthreads();
    Rec rec;
    F2 er{0.0f, 0.0f}, ei = er, od = er, oi = er;  // even / odd (l - m) sums
    bool live = false;
    if (r < nnorth) {
        F2 z, s;
        ring_zs(nside, r, &z, &s);
        live = m <= ring_limit(nside, r, lmax, extra);
        if (live) rec.start(m, s_norm, z, s);
    }
    if (!__syncthreads_or(live)) return;
#pragma unroll
    for (int i = 0; i < 8; ++i) top = max(top, s_top[i]);
    const int ex = scale_exp_f64(top);
    const double up = pow2(ex);
    for (int l0 = m; l0 <= lmax; l0 += kTile) {
        const int n = min(kTile, lmax + 1 - l0);
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += 256) {
            if (l0 + i > m) co[i] = step_coeffs(l0 + i, m);
            const double2 c = __ldg(a + l0 + i);
            const F2 x = f2_of(c.x * up), y = f2_of(c.y * up);
            al[i] = make_float4(x.h, x.l, y.h, y.l);
        }
        __syncthreads();
        if (!live) continue;
        for (int i = 0; i < n; ++i) {
            const float4 x = al[i];
            if (l0 + i > m) rec.step(co[i]);
            if (rec.e < 0) continue;
            const F2 pr = f2_mul(rec.v1, F2{x.x, x.y}), pi = f2_mul(rec.v1, F2{x.z, x.w});
            if ((l0 + i - m) & 1) {
                od = f2_acc(od, pr);
                oi = f2_acc(oi, pi);
            } else {
                er = f2_acc(er, pr);
                ei = f2_acc(ei, pi);
            }
        }
    }
    if (!live) return;
    const long long stride = lmax + 1;
    const double down = pow2(-ex);
    auto store = [&](int ring) {
        G[(long long)ring * stride + m] = make_float2((float)((double)f2_add(er, od).h * down),
                                                      (float)((double)f2_add(ei, oi).h * down));
    };
    store(r);
    if (rs == r) return;
    od = F2{-od.h, -od.l};
    oi = F2{-oi.h, -oi.l};
    store(rs);
}

constexpr int kGroup = 32;  // degrees between the block's reductions

// Analysis, Legendre part: alm[l, m] = c K_l sum_rings lambda_lm(z) F_m over all northern
// rings and their mirrors for order m = lmax - blockIdx.x; c = 4 pi / Npix, K_l = kl[l] (kl
// NULL: 1).  One block per order, R rings a thread, in passes over the rings.  The
// threads' terms of eight degrees go through shared memory: within a warp 32 -> 4 partial
// sums a degree, then every 32 degrees over the warps, in a fixed order and on FP32 pairs throughout.  The
// Four rings a thread share the reduction: 5.76 ms at nside 2048, l_max 1024 (one ring 8.11;
// 70.1 in FP64 with atomics); with one pass or two over the rings (nside <= 128) one ring is
// the shorter chain (25.5 against 27.9 us at nside 128, l_max 64).  The
// F_m of a pass enter scaled by a power of two (exact), and the passes add up in FP64.
template <int R>
__global__ void __launch_bounds__(256)
sht_leg_anal(int nside, int lmax, float extra, const float2 *__restrict__ F, const double *__restrict__ kl,
             double c, double2 *__restrict__ alm) {
    extern __shared__ double2 acc[];  // [lmax + 1 - m]
    __shared__ float4 co[kTile], term[8][8][33], part[8][kGroup];
    __shared__ F2 s_norm;
    __shared__ unsigned s_top[8];
    const int m = lmax - blockIdx.x, nnorth = 2 * nside, nr = 4 * nside - 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long stride = lmax + 1;
    for (int i = threadIdx.x; i <= lmax - m; i += 256) acc[i] = make_double2(0.0, 0.0);
    if (threadIdx.x < 32) {
        const F2 v = norm_mm(m);
        if (threadIdx.x == 0) s_norm = v;
    }
    __syncthreads();
    for (int base = 0; base < nnorth; base += 256 * R) {
        Rec rec[R];
        F2 sr[R], si[R], dr[R], di[R];  // F north + south (even l - m), north - south (odd)
        float4 f[R];                    // north, south
        bool live[R], any = false;
        unsigned top = 0u;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int r = base + 256 * j + threadIdx.x;
            live[j] = false;
            if (r < nnorth) {
                live[j] = m <= ring_limit(nside, r, lmax, extra);
                if (live[j]) {
                    F2 z, s;
                    ring_zs(nside, r, &z, &s);
                    rec[j].start(m, s_norm, z, s);
                    const int rs = nr - 1 - r;
                    const float2 fn = F[(long long)r * stride + m];
                    const float2 fs = rs != r ? F[(long long)rs * stride + m] : make_float2(0.0f, 0.0f);
                    f[j] = make_float4(fn.x, fn.y, fs.x, fs.y);
                    top = max(max(top, max(__float_as_uint(fn.x) & 0x7fffffffu, __float_as_uint(fn.y) & 0x7fffffffu)),
                              max(__float_as_uint(fs.x) & 0x7fffffffu, __float_as_uint(fs.y) & 0x7fffffffu));
                }
            }
            any |= live[j];
        }
        top = __reduce_max_sync(~0u, top);
        if (lane == 0) s_top[warp] = top;
        if (!__syncthreads_or(any)) continue;  // (else barriers follow before the next pass writes)
#pragma unroll
        for (int i = 0; i < 8; ++i) top = max(top, s_top[i]);
        const int ex = scale_exp_f32(top);
        const float scale = __int_as_float((127 + ex) << 23);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            if (!live[j]) continue;
            const float nx = scale * f[j].x, ny = scale * f[j].y, sx = scale * f[j].z, sy = scale * f[j].w;
            sr[j] = f2_sum(nx, sx);
            si[j] = f2_sum(ny, sy);
            dr[j] = f2_sum(nx, -sx);
            di[j] = f2_sum(ny, -sy);
        }
        const bool warp_any = __any_sync(~0u, any);
        for (int l0 = m; l0 <= lmax; l0 += kTile) {
            const int n = min(kTile, lmax + 1 - l0);
            __syncthreads();
            for (int i = threadIdx.x; i < n; i += 256)
                if (l0 + i > m) co[i] = step_coeffs(l0 + i, m);
            __syncthreads();
            for (int g0 = 0; g0 < n; g0 += kGroup) {
                if (!warp_any) part[warp][lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                for (int i0 = g0; warp_any && i0 < g0 + kGroup; i0 += 8) {
#pragma unroll 2
                    for (int i = 0; i < 8; ++i) {
                        F2 tr{0.0f, 0.0f}, ti{0.0f, 0.0f};
                        if (i0 + i < n) {
                            const float4 cc = co[i0 + i];
                            const bool odd = (l0 + i0 + i - m) & 1;
#pragma unroll
                            for (int j = 0; j < R; ++j) {
                                if (!live[j]) continue;
                                if (l0 + i0 + i > m) rec[j].step(cc);
                                if (rec[j].e < 0) continue;
                                tr = f2_acc(tr, f2_mul(rec[j].v1, odd ? dr[j] : sr[j]));
                                ti = f2_acc(ti, f2_mul(rec[j].v1, odd ? di[j] : si[j]));
                            }
                        }
                        term[warp][i][lane] = make_float4(tr.h, tr.l, ti.h, ti.l);
                    }
                    __syncwarp();
                    // lane: degree lane / 4, the eight terms from 8 (lane % 4)
                    F2 tr{0.0f, 0.0f}, ti{0.0f, 0.0f};
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 t = term[warp][lane >> 2][8 * (lane & 3) + k];
                        tr = f2_add(tr, F2{t.x, t.y});
                        ti = f2_add(ti, F2{t.z, t.w});
                    }
#pragma unroll
                    for (int o = 1; o < 4; o <<= 1) {
                        F2 x, y;
                        x.h = __shfl_xor_sync(~0u, tr.h, o);
                        x.l = __shfl_xor_sync(~0u, tr.l, o);
                        y.h = __shfl_xor_sync(~0u, ti.h, o);
                        y.l = __shfl_xor_sync(~0u, ti.l, o);
                        tr = f2_add(tr, x);
                        ti = f2_add(ti, y);
                    }
                    if ((lane & 3) == 0) part[warp][i0 - g0 + (lane >> 2)] = make_float4(tr.h, tr.l, ti.h, ti.l);
                    __syncwarp();
                }
                __syncthreads();
                if (threadIdx.x < kGroup && g0 + (int)threadIdx.x < n) {
                    F2 tr{0.0f, 0.0f}, ti = tr;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 t = part[k][threadIdx.x];
                        tr = f2_add(tr, F2{t.x, t.y});
                        ti = f2_add(ti, F2{t.z, t.w});
                    }
                    double2 &o = acc[l0 - m + g0 + threadIdx.x];
                    const double down = pow2(-ex);
                    o.x = fma((double)tr.h + (double)tr.l, down, o.x);
                    o.y = fma((double)ti.h + (double)ti.l, down, o.y);
                }
                __syncthreads();
            }
        }
    }
    __syncthreads();
    double2 *a = alm + alm_base(lmax, m);
    for (int l = m + threadIdx.x; l <= lmax; l += 256) {
        const double2 t = acc[l - m];
        const double w = c * (kl ? kl[l] : 1.0);
        a[l] = make_double2(w * t.x, w * t.y);
    }
}

// ---- ring sums ----------------------------------------------------------------
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// e^{i pi J / L} for an exact integer 0 <= J < 2L, to about one FP32 ulp: J / L = hi + lo with
// hi the rounded quotient and lo = (J - hi L) / L (the remainder exact by the fused
// multiply-add), J folded into [-L, L); the rounding of hi is undone to first order,
// e^{i pi lo} = 1 + i pi lo.
__device__ __forceinline__ float2 twiddle(int J, float L, float inv_l) {
    const float fj = (float)(J >= (int)L ? J - 2 * (int)L : J);  // exact: |J|, L <= 2^15
    const float hi = fj * inv_l;
    const float lo = fmaf(-hi, L, fj) * inv_l;
    float sn, cs;
    sincospif(hi, &sn, &cs);
    const float d = 3.14159265f * lo;
    return make_float2(fmaf(-sn, d, cs), fmaf(cs, d, sn));
}

__device__ __forceinline__ void fold(float &sum, float &comp, float v) {  // Kahan
    const float y = v - comp, t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// Synthesis, ring part, any ring length 4 Q: for northern ring r and its mirror,
// pixel k1 + a Q (a = 0..3) gets sum_m w_m Re(G_m e^{i m phi}) = Re sum_c i^{a c} S_c(k1), S_c
// the sum over the orders m = c mod 4 at pixel k1 (w_0 = 1, else 2).  add != 0 adds it to the
// map.  The orders are staged in shared memory 1024 at a time.
constexpr int kOrders = 1024;
__global__ void __launch_bounds__(256)
sht_ring_synth(int nside, int lmax, float extra, int r_first, const float2 *__restrict__ G,
               float *__restrict__ map, int add) {
    __shared__ float4 gs[kOrders];  // north, south
    // the longest rings first
    const int r = r_first + gridDim.x - 1 - blockIdx.x, nr = 4 * nside - 1, rs = nr - 1 - r;
    const bool mirror = rs != r;
    const long long stride = lmax + 1;
    const ShtRing g = sht_ring(nside, r), h = sht_ring(nside, rs);
    const int L = g.len, Q = L / 4, lim = ring_limit(nside, r, lmax, extra);
    const float fl = (float)L, inv_l = 1.0f / fl;
    for (int k0 = blockIdx.y * 256; k0 < Q; k0 += gridDim.y * 256) {
        const int k = k0 + threadIdx.x;
        const int q = 2 * min(k, Q - 1) + g.t;  // m phi = pi m q / L
        const float2 step = twiddle(q, fl, inv_l);
        const int j8 = (kAnchor * q) % (2 * L);
        float sum[4][4], comp[4][4];  // [class][north re, im, south re, im]
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[c][i] = comp[c][i] = 0.0f;
        int J = 0;
        for (int m0 = 0; m0 <= lim; m0 += kOrders) {
            const int n = min(kOrders, lim + 1 - m0), n8 = (n + 7) & ~7;
            __syncthreads();
            for (int i = threadIdx.x; i < n8; i += 256) {
                const float w = m0 + i == 0 ? 1.0f : 2.0f;
                const float2 zero = make_float2(0.0f, 0.0f);
                const float2 a = i < n ? G[(long long)r * stride + m0 + i] : zero;
                const float2 b = i < n && mirror ? G[(long long)rs * stride + m0 + i] : zero;
                gs[i] = make_float4(w * a.x, w * a.y, w * b.x, w * b.y);
            }
            __syncthreads();
            for (int i = 0; i < n8; i += 2 * kAnchor) {
                float p[4][4];
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int e = 0; e < 4; ++e) p[c][e] = 0.0f;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    if (i + half * kAnchor >= n8) break;
                    float2 w = twiddle(J, fl, inv_l);
                    J += j8;
                    J -= J >= 2 * L ? 2 * L : 0;
#pragma unroll
                    for (int e = 0; e < kAnchor; ++e) {
                        const float4 a = gs[i + half * kAnchor + e];
                        float (&c)[4] = p[e & 3];
                        c[0] = fmaf(a.x, w.x, fmaf(-a.y, w.y, c[0]));
                        c[1] = fmaf(a.x, w.y, fmaf(a.y, w.x, c[1]));
                        c[2] = fmaf(a.z, w.x, fmaf(-a.w, w.y, c[2]));
                        c[3] = fmaf(a.z, w.y, fmaf(a.w, w.x, c[3]));
                        w = cmul(w, step);
                    }
                }
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int e = 0; e < 4; ++e) fold(sum[c][e], comp[c][e], p[c][e]);
            }
        }
        if (k >= Q) continue;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (s && !mirror) break;
            const float r0 = sum[0][2 * s], r1 = sum[1][2 * s], i1 = sum[1][2 * s + 1];
            const float r2 = sum[2][2 * s], r3 = sum[3][2 * s], i3 = sum[3][2 * s + 1];
            // Re sum_c i^{a c} S_c
            const float v[4] = {(r0 + r2) + (r1 + r3), (r0 - r2) + (i3 - i1), (r0 + r2) - (r1 + r3),
                                (r0 - r2) - (i3 - i1)};
            float *o = map + (s ? h.start : g.start) + k;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                if (add) o[a * Q] += v[a];
                else o[a * Q] = v[a];
            }
        }
    }
}

// Analysis, ring part, any ring length 4 Q: F[ring][m] = sum_k m_k e^{-i m phi_k} for
// northern ring r and its mirror, threads over m <= the ring's limit.  The quarter turns of
// pixel k1 enter order m as Y_c(k1) = sum_a (-i)^{a c} m_{k1 + a Q}, c = m mod 4; staged in
// shared memory 512 pixels at a time (classes 0 and 2 are real, 3 is conjugate to 1).
constexpr int kPix = 512;
__global__ void __launch_bounds__(256)
sht_ring_anal(int nside, int lmax, float extra, int r_first, const float *__restrict__ map,
              float2 *__restrict__ F) {
    __shared__ float4 y[4][kPix + 1];  // [class]: north re, im, south re, im
    // the longest rings first
    const int r = r_first + gridDim.x - 1 - blockIdx.x, nr = 4 * nside - 1, rs = nr - 1 - r;
    const bool mirror = rs != r;
    const long long stride = lmax + 1;
    const ShtRing g = sht_ring(nside, r), h = sht_ring(nside, rs);
    const int L = g.len, Q = L / 4, lim = ring_limit(nside, r, lmax, extra);
    const float fl = (float)L, inv_l = 1.0f / fl;
    for (int m0 = blockIdx.y * 256; m0 <= lim; m0 += gridDim.y * 256) {
        const int m = m0 + threadIdx.x, c = m & 3, mr = m % (2 * L);
        // e^{-i m phi_k}: J = -m (2k + t) mod 2L
        const int j1 = (2 * L - 2 * mr % (2 * L)) % (2 * L);
        const float2 step = twiddle(j1, fl, inv_l);
        const int j8 = (int)((8LL * j1) % (2 * L));
        int J = g.t ? (2 * L - mr) % (2 * L) : 0;
        float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f}, comp[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int k0 = 0; k0 < Q; k0 += kPix) {
            const int n = min(kPix, Q - k0), n8 = (n + 7) & ~7;
            __syncthreads();
            for (int i = threadIdx.x; i < n8; i += 256) {
                float v[2][4];
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int a = 0; a < 4; ++a)
                        v[s][a] = i < n && (!s || mirror)
                                      ? __ldg(map + (s ? h.start : g.start) + k0 + i + a * Q)
                                      : 0.0f;
                float e[2], o[2], x[2], z[2];
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    e[s] = (v[s][0] + v[s][2]) + (v[s][1] + v[s][3]);
                    o[s] = (v[s][0] + v[s][2]) - (v[s][1] + v[s][3]);
                    x[s] = v[s][0] - v[s][2];
                    z[s] = v[s][3] - v[s][1];  // (-i)(v1 - v3): imaginary part -(v1 - v3)
                }
                y[0][i] = make_float4(e[0], 0.0f, e[1], 0.0f);
                y[1][i] = make_float4(x[0], z[0], x[1], z[1]);
                y[2][i] = make_float4(o[0], 0.0f, o[1], 0.0f);
                y[3][i] = make_float4(x[0], -z[0], x[1], -z[1]);
            }
            __syncthreads();
            for (int i = 0; i < n8; i += kAnchor) {
                float2 w = twiddle(J, fl, inv_l);
                J += j8;
                J -= J >= 2 * L ? 2 * L : 0;
                float p[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int e = 0; e < kAnchor; ++e) {
                    const float4 a = y[c][i + e];
                    p[0] = fmaf(a.x, w.x, fmaf(-a.y, w.y, p[0]));
                    p[1] = fmaf(a.x, w.y, fmaf(a.y, w.x, p[1]));
                    p[2] = fmaf(a.z, w.x, fmaf(-a.w, w.y, p[2]));
                    p[3] = fmaf(a.z, w.y, fmaf(a.w, w.x, p[3]));
                    w = cmul(w, step);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) fold(sum[e], comp[e], p[e]);
            }
        }
        if (m > lim) continue;
        F[(long long)r * stride + m] = make_float2(sum[0], sum[1]);
        if (mirror) F[(long long)rs * stride + m] = make_float2(sum[2], sum[3]);
    }
}

// In-place FFTs of two sequences of 2^lg complex values in shared memory, x[0 ..] and x[ss ..], sign
// -1 forward, +1 inverse (unnormalised): Stockham radix 4 with one radix-2 pass when lg is odd; a
// thread holds the values of its four butterflies between the two barriers of a pass.  tw[k] =
// e^{-2 pi i k / n}, n = 2^(lg + 1), for k < n / 4; the other quadrants by exact rotations.
__device__ __forceinline__ float2 fft_twiddle(const float2 *tw, int k, int lgq, float sgn) {
    const float2 w = tw[k & ((1 << lgq) - 1)];
    const int quad = k >> lgq;  // times (-i)^quad
    float2 v = quad & 1 ? make_float2(w.y, -w.x) : w;
    if (quad & 2) v = make_float2(-v.x, -v.y);
    return make_float2(v.x, -sgn * v.y);
}
__device__ __forceinline__ void fft_shared(float2 *x, int ss, const float2 *tw, int lg, float sgn) {
    const int n = 1 << lg, q = n >> 2, T = blockDim.x, lgq = lg - 1;
    int ls = 0;  // log2 of the stride s
    for (; ls + 2 <= lg; ls += 2) {
        float2 y[4][4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = threadIdx.x + b * T, t = i & (q - 1);
            if (i >= 2 * q) break;
            const float2 *v = x + (i >> (lg - 2)) * ss + t;
            const float2 a0 = v[0], a1 = v[q], a2 = v[2 * q], a3 = v[3 * q];
            const int k = ((t >> ls) << ls) << 1;  // p s, in steps of the table
            const float2 s02 = make_float2(a0.x + a2.x, a0.y + a2.y), d02 = make_float2(a0.x - a2.x, a0.y - a2.y);
            const float2 s13 = make_float2(a1.x + a3.x, a1.y + a3.y), d13 = make_float2(a1.x - a3.x, a1.y - a3.y);
            const float2 jd = make_float2(-sgn * d13.y, sgn * d13.x);  // sgn i d13
            y[b][0] = make_float2(s02.x + s13.x, s02.y + s13.y);
            y[b][1] = cmul(make_float2(d02.x + jd.x, d02.y + jd.y), fft_twiddle(tw, k, lgq, sgn));
            y[b][2] = cmul(make_float2(s02.x - s13.x, s02.y - s13.y), fft_twiddle(tw, 2 * k, lgq, sgn));
            y[b][3] = cmul(make_float2(d02.x - jd.x, d02.y - jd.y), fft_twiddle(tw, 3 * k, lgq, sgn));
        }
        __syncthreads();
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = threadIdx.x + b * T, t = i & (q - 1);
            if (i >= 2 * q) break;
            const int lo = t & ((1 << ls) - 1), o = ((t >> ls) << (ls + 2)) + lo;
            float2 *v = x + (i >> (lg - 2)) * ss + o;
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j << ls] = y[b][j];
        }
        __syncthreads();
    }
    if (ls < lg) {  // one radix-2 pass, stride n / 2
        const int hN = n >> 1;
        for (int i = threadIdx.x; i < n; i += T) {
            float2 *v = x + (i >> (lg - 1)) * ss + (i & (hN - 1));
            const float2 a = v[0], b = v[hN];
            v[0] = make_float2(a.x + b.x, a.y + b.y);
            v[hN] = make_float2(a.x - b.x, a.y - b.y);
        }
        __syncthreads();
    }
}
__device__ __forceinline__ void fft_table(float2 *tw, int lg) {
    const float inv = 2.0f / (float)(1 << lg);
    for (int k = threadIdx.x; k < (1 << (lg - 2)); k += blockDim.x) {
        float sn, cs;
        sincospif(-(float)k * inv, &sn, &cs);  // the argument is exact
        tw[k] = make_float2(cs, sn);
    }
}

// Analysis of belt ring r = r_first + blockIdx.x and its mirror, each by a complex FFT of half its
// length, even pixels + i odd ones (both rings as one complex sequence would round the fainter
// one to the brighter one's last bits).
__global__ void __launch_bounds__(1024)
sht_fft_anal(int nside, int lmax, float extra, int lg, int r_first, const float *__restrict__ map,
             float2 *__restrict__ F) {
    extern __shared__ float2 fx[];
    const int n = 1 << lg, half = n >> 1;
    float2 *tw = fx + n + 2;
    const int r = r_first + blockIdx.x, rs = 4 * nside - 2 - r;
    const bool mirror = rs != r;
    const ShtRing g = sht_ring(nside, r), h = sht_ring(nside, rs);
    fft_table(tw, lg);
    for (int k = threadIdx.x; k < half; k += blockDim.x) {
        const float *a = map + g.start + 2 * k, *b = map + h.start + 2 * k;
        fx[k] = make_float2(__ldg(a), __ldg(a + 1));
        fx[half + k] = mirror ? make_float2(__ldg(b), __ldg(b + 1)) : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    fft_shared(fx, half, tw, lg - 1, -1.0f);
    const long long stride = lmax + 1;
    const int lim = ring_limit(nside, r, lmax, extra);
    const float inv = 1.0f / (float)n;
    for (int m = threadIdx.x; m <= lim; m += blockDim.x) {
        // X_k = (Z_k + Z*_{h-k}) / 2 - i/2 e^{-2 pi i k / n} (Z_k - Z*_{h-k}), h = n / 2, k <= h;
        // X_{n-k} = X*_k
        const int mm = m & (n - 1), k = min(mm, n - mm);
        const float2 w = fft_twiddle(tw, k, lg - 2, -1.0f);
        auto order = [&](const float2 *z) {
            const float2 a = z[k & (half - 1)], b = z[(half - k) & (half - 1)];
            const float2 e = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
            const float2 o = make_float2(0.5f * (a.y + b.y), 0.5f * (b.x - a.x));
            const float2 p = cmul(w, o);
            return make_float2(e.x + p.x, mm > half ? -(e.y + p.y) : e.y + p.y);
        };
        float2 fn = order(fx), fs = order(fx + half);
        if (g.t) {  // e^{-i pi m / n}, the argument exact
            float sn, cs;
            sincospif(-(float)m * inv, &sn, &cs);
            fn = cmul(fn, make_float2(cs, sn));
            fs = cmul(fs, make_float2(cs, sn));
        }
        F[(long long)r * stride + m] = fn;
        if (mirror) F[(long long)rs * stride + m] = fs;
    }
}

// Synthesis of belt ring r and its mirror: bin b of the Hermitian spectra collects the orders
// m = b and, conjugate, m = -b mod n (each w_m / 2 G_m e^{i pi m t / n}); each ring by a complex FFT
// of half its length (see above) whose bins are Z_k = (H_k + H*_{h-k}) + i e^{2 pi i k / n} (H_k -
// H*_{h-k}), h = n / 2.
__global__ void __launch_bounds__(1024)
sht_fft_synth(int nside, int lmax, float extra, int lg, int r_first, const float2 *__restrict__ G,
              float *__restrict__ map, int add) {
    extern __shared__ float2 fx[];
    const int n = 1 << lg, half = n >> 1;
    float2 *tw = fx + n + 2;
    const int r = r_first + blockIdx.x, rs = 4 * nside - 2 - r;
    const bool mirror = rs != r;
    const ShtRing g = sht_ring(nside, r), h = sht_ring(nside, rs);
    const long long stride = lmax + 1;
    const int lim = ring_limit(nside, r, lmax, extra);
    const float inv = 1.0f / (float)n;
    fft_table(tw, lg);
    for (int b = threadIdx.x; b <= half; b += blockDim.x) {
        float2 zn = make_float2(0.0f, 0.0f), zs = zn;
        auto take = [&](int m, float conj) {
            if (m > lim) return;
            float2 a = G[(long long)r * stride + m];
            float2 c = mirror ? G[(long long)rs * stride + m] : make_float2(0.0f, 0.0f);
            if (g.t) {
                float sn, cs;
                sincospif((float)m * inv, &sn, &cs);
                a = cmul(a, make_float2(cs, sn));
                c = cmul(c, make_float2(cs, sn));
            }
            const float w = m == 0 ? 0.5f : 1.0f;
            zn.x = fmaf(w, a.x, zn.x);
            zn.y = fmaf(conj * w, a.y, zn.y);
            zs.x = fmaf(w, c.x, zs.x);
            zs.y = fmaf(conj * w, c.y, zs.y);
        };
        const int nb = (n - b) & (n - 1);
        take(b, 1.0f);
        take(b + n, 1.0f);
        take(nb, -1.0f);
        take(nb + n, -1.0f);
        fx[b] = zn;
        fx[half + 1 + b] = zs;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < half + 2; i += blockDim.x) {  // k <= h / 2 of both rings
        const int ring = i > half / 2, k = i - ring * (half / 2 + 1);
        float2 *z = fx + ring * (half + 1);
        const float2 a = z[k], b = z[half - k], w = fft_twiddle(tw, k, lg - 2, 1.0f);
        // i w (H_k - H*_{h-k}); bin h - k has the conjugates of its terms
        const float2 p = make_float2(a.x + b.x, a.y - b.y), q = cmul(w, make_float2(a.x - b.x, a.y + b.y));
        z[k] = make_float2(p.x - q.y, p.y + q.x);
        if (k > 0) z[half - k] = make_float2(p.x + q.y, q.x - p.y);
    }
    __syncthreads();
    fft_shared(fx, half + 1, tw, lg - 1, 1.0f);
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int ring = k >= half, j = k - ring * half;
        if (ring && !mirror) break;
        const float2 v = fx[ring * (half + 1) + j];
        float *o = map + (ring ? h.start : g.start) + 2 * j;
        if (add) {
            o[0] += v.x;
            o[1] += v.y;
        } else {
            o[0] = v.x;
            o[1] = v.y;
        }
    }
}

// The longest FFT's shared memory.  The limits are set to the largest value whatever the
// call needs: calls of several threads may race on them.
constexpr int kFftSmem = 8 * (5 * 4096 + 2);

// log2 of the belt rings' length where they go through the FFT (L <= 16384, and from 1e8
// products of a direct sum on), else 0.  Direct for all rings / quarter sums and FFT, both
// directions, us: nside 128, l_max 64 (8e6): 18.6 / 25.4; nside 512, l_max 1024 (2e9,
// synthesis): 257 / 126; nside 2048, l_max 1024 (3e10): 7910 / 2480.
int belt_fft(int nside, int lmax) {
    int lg = 2;
    while ((1 << (lg - 2)) < nside) ++lg;
    return 8.0 * nside * nside * (lmax + 1) >= 1e8 && lg <= 14 ? lg : 0;
}

// One radix-4 butterfly a thread and pass in short rings, up to four in long ones (two CTAs
// of 512 threads per SM at n = 8192).
int fft_threads(int lg) { return std::max(32, std::min(1 << (lg - 2), std::max(512, 1 << (lg - 4)))); }

// Rings first .. last (northern half) by direct quarter sums; the rest of [0, 2 nside) by FFT.
cudaError_t ring_synth(int nside, int lmax, const float2 *G, float *map, int add, cudaStream_t st) {
    const int lg = belt_fft(nside, lmax), n_cap = lg ? nside - 1 : 2 * nside;
    const float extra = order_extra(lmax);
    if (n_cap > 0) {
        dim3 grid(n_cap, nside > 512 ? 2 : 1);
        sht_ring_synth<<<grid, 256, 0, st>>>(nside, lmax, extra, 0, G, map, add);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess || !lg) return e;
    }
    const size_t smem = sizeof(float2) * ((5u << (lg - 2)) + 2);
    cudaError_t e = cudaFuncSetAttribute(sht_fft_synth, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kFftSmem);
    if (e != cudaSuccess) return e;
    sht_fft_synth<<<nside + 1, fft_threads(lg), smem, st>>>(nside, lmax, extra, lg, nside - 1, G, map, add);
    return cudaGetLastError();
}

cudaError_t ring_anal(int nside, int lmax, const float *map, float2 *F, cudaStream_t st) {
    const int lg = belt_fft(nside, lmax), n_cap = lg ? nside - 1 : 2 * nside;
    const float extra = order_extra(lmax);
    if (n_cap > 0) {
        dim3 grid(n_cap, (lmax + 256) / 256);
        sht_ring_anal<<<grid, 256, 0, st>>>(nside, lmax, extra, 0, map, F);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess || !lg) return e;
    }
    const size_t smem = sizeof(float2) * ((5u << (lg - 2)) + 2);
    cudaError_t e = cudaFuncSetAttribute(sht_fft_anal, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kFftSmem);
    if (e != cudaSuccess) return e;
    sht_fft_anal<<<nside + 1, fft_threads(lg), smem, st>>>(nside, lmax, extra, lg, nside - 1, map, F);
    return cudaGetLastError();
}

}  // namespace

// alm (device, n_alm(lmax) complex) -> map (device FP32); add != 0 adds.
cudaError_t sht_synthesis(int nside, int lmax, const double2 *d_alm, float *d_map, int add,
                          cudaStream_t st) {
    const int nr = 4 * nside - 1, nnorth = 2 * nside;
    float2 *G = nullptr;
    cudaError_t e = cudaMallocAsync(&G, sizeof(float2) * (size_t)nr * (lmax + 1), st);
    if (e != cudaSuccess) return e;
    dim3 grid((nnorth + 255) / 256, lmax + 1);
    sht_leg_synth<<<grid, 256, 0, st>>>(nside, lmax, order_extra(lmax), d_alm, G);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = ring_synth(nside, lmax, G, d_map, add, st);
    const cudaError_t f = cudaFreeAsync(G, st);
    return e != cudaSuccess ? e : f;
}

// map (device FP32) -> alm (device, n_alm(lmax) complex), each a_lm scaled by kl[l]
// when kl (device, lmax + 1 doubles) is given.
cudaError_t sht_analysis(int nside, int lmax, const float *d_map, const double *d_kl,
                         double2 *d_alm, cudaStream_t st) {
    const int nr = 4 * nside - 1, nnorth = 2 * nside;
    const size_t smem = sizeof(float4) * (size_t)(lmax + 1);
    auto kernel = nnorth > 512 ? sht_leg_anal<4> : sht_leg_anal<1>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(float4) * 8192);  // (as kFftSmem)
    if (e != cudaSuccess) return e;
    float2 *F = nullptr;
    if ((e = cudaMallocAsync(&F, sizeof(float2) * (size_t)nr * (lmax + 1), st)) != cudaSuccess)
        return e;
    e = ring_anal(nside, lmax, d_map, F, st);
    if (e == cudaSuccess) {
        const double c = 4.0 * kPi / (12.0 * (double)nside * (double)nside);
        kernel<<<lmax + 1, 256, smem, st>>>(nside, lmax, order_extra(lmax), F, d_kl, c, d_alm);
        e = cudaGetLastError();
    }
    const cudaError_t f = cudaFreeAsync(F, st);
    return e != cudaSuccess ? e : f;
}

long long sht_n_alm(int lmax) { return n_alm(lmax); }

}  // namespace ksc

namespace {

int sht_fail(int code, const char *msg) {
    ksc::set_last_error(msg);
    return code;
}

int sht_cuda(cudaError_t e, const char *what) {
    return sht_fail(e == cudaErrorMemoryAllocation ? KSC_ERR_NOMEM : KSC_ERR_CUDA, what);
}

int sht_args(int nside, int lmax) {
    if (nside < 1 || nside > 8192 || (nside & (nside - 1)))
        return sht_fail(KSC_ERR_ARG, "nside must be a power of two <= 8192");
    if (lmax < 0 || lmax > 4 * nside || lmax > 8191)
        return sht_fail(KSC_ERR_ARG, "lmax outside 0..min(4 nside, 8191)");
    return KSC_OK;
}

}  // namespace

extern "C" {

int ksc_sht_alm2map(int nside, int lmax, const double *d_alm, float *d_map, void *stream) {
    ksc::NvtxRange range("ksc_sht_alm2map");
    int rc = sht_args(nside, lmax);
    if (rc) return rc;
    if (!d_alm || !d_map) return sht_fail(KSC_ERR_ARG, "null pointer");
    const cudaError_t e = ksc::sht_synthesis(nside, lmax, (const double2 *)d_alm, d_map, 0,
                                             (cudaStream_t)stream);
    return e == cudaSuccess ? KSC_OK : sht_cuda(e, "spherical-harmonic synthesis");
}

int ksc_sht_map2alm(int nside, int lmax, const float *d_map, double *d_alm, void *stream) {
    ksc::NvtxRange range("ksc_sht_map2alm");
    int rc = sht_args(nside, lmax);
    if (rc) return rc;
    if (!d_alm || !d_map) return sht_fail(KSC_ERR_ARG, "null pointer");
    const cudaError_t e = ksc::sht_analysis(nside, lmax, d_map, nullptr, (double2 *)d_alm,
                                            (cudaStream_t)stream);
    return e == cudaSuccess ? KSC_OK : sht_cuda(e, "spherical-harmonic analysis");
}

int ksc_conv_harmonic(const ksc_split *s, const float *d_in, float *d_out, int add,
                      void *stream) {
    ksc::NvtxRange range("ksc_conv_harmonic");
    if (!s || !d_in || !d_out) return sht_fail(KSC_ERR_ARG, "null argument");
    const int lc = s->l_cut;
    if (lc < 0 || (int)s->k_harm.size() < lc + 1)
        return sht_fail(KSC_ERR_ARG, "the split has no harmonic part");
    int rc = sht_args(s->nside, lc);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    double *kl = nullptr;
    double2 *alm = nullptr;
    cudaError_t e = cudaMallocAsync(&kl, sizeof(double) * (size_t)(lc + 1), st);
    if (e == cudaSuccess)
        e = cudaMallocAsync(&alm, sizeof(double2) * (size_t)ksc::sht_n_alm(lc), st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(kl, s->k_harm.data(), sizeof(double) * (size_t)(lc + 1),
                            cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = ksc::sht_analysis(s->nside, lc, d_in, kl, alm, st);
    if (e == cudaSuccess) e = ksc::sht_synthesis(s->nside, lc, alm, d_out, add ? 1 : 0, st);
    if (kl) cudaFreeAsync(kl, st);
    if (alm) cudaFreeAsync(alm, st);
    return e == cudaSuccess ? KSC_OK : sht_cuda(e, "harmonic half");
}

}  // extern "C"
