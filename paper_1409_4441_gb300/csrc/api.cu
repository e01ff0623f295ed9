// C ABI of libksconv (declared in include/ksconv.h).
#include <algorithm>
#include <cstdint>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <new>
#include <queue>
#include <string>
#include <vector>

#include "ksc_device.cuh"
#include "ksc_internal.h"
#include "ksc_tc.cuh"

namespace {

// One CTA waits on an mbarrier nothing arrives on (phase 0 never completes); the
// bounded wait runs out and the CTA raises the error flag like a kernel would.
__global__ void wait_probe_kernel(int *err, int max_polls) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        ksc::tc::mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bool done = ksc::tc::mbar_wait(&bar, 0u, max_polls);
    if (!done && threadIdx.x == 0) atomicExch(err, KSC_ERR_TIMEOUT);
}

thread_local std::string g_last_error;

int fail(int code, const std::string &msg) {
    g_last_error = msg;
    return code;
}

int cuda_fail(cudaError_t e, const char *what) {
    return fail(e == cudaErrorMemoryAllocation ? KSC_ERR_NOMEM : KSC_ERR_CUDA,
                std::string(what) + ": " + cudaGetErrorString(e));
}

constexpr double kPi = 3.14159265358979323846;

bool valid_nside(int nside) {
    return nside >= 1 && nside <= 8192 && (nside & (nside - 1)) == 0;
}

// Device allocations of one split construction, counted for fault injection.
thread_local int g_alloc_count = 0;

cudaError_t dev_malloc(void **dst, size_t bytes) {
    if (ksc::inject_alloc_fault(++g_alloc_count)) return cudaErrorMemoryAllocation;
    return cudaMalloc(dst, bytes);
}

template <class T>
cudaError_t dev_upload(T **dst, const T *src, size_t n) {
    cudaError_t e = dev_malloc((void **)dst, sizeof(T) * (n ? n : 1));
    if (e != cudaSuccess) return e;
    if (n) e = cudaMemcpy(*dst, src, sizeof(T) * n, cudaMemcpyHostToDevice);
    return e;
}

void release(ksc_split *s) {
    if (!s) return;
    cudaFree(s->d_tab);
    cudaFree(s->d_rings);
    cudaFree(s->d_range);
    cudaFree(s->d_pairs);
    cudaFree(s->d_xinfo);
    cudaFree(s->d_xodd);
    cudaFree(s->d_pair_base);
    cudaFree(s->d_items);
    cudaFree(s->d_items_sym);
    cudaFree(s->d_items_sym_lpt);
    cudaFree(s->d_items_smma);
    cudaFree(s->d_items_smma_lpt);
    cudaFree(s->d_items_mma);
    cudaFree(s->d_ws);
    cudaFree(s->d_items_belt);
    for (ksc_split::ScratchSlot &c : s->slots) {
        cudaFree(c.mem);
        if (c.done) cudaEventDestroy(c.done);
    }
    cudaFree(s->d_cap_tiles);
    cudaFree(s->d_cap_tiles_lpt);
    cudaFree(s->d_ncut);
    cudaFree(s->d_coef_off);
    cudaFree(s->d_coef);
    cudaFree(s->d_irr_items);
    cudaFree(s->d_irr_first);
    cudaFree(s->d_irr);
    cudaFree(s->d_err);
    cudaFree(s->d_io);
    if (s->own_stream) cudaStreamDestroy(s->own_stream);
    delete s;
}

constexpr int kSms = 152;

// Without the tensor-core cap stage: the gather sums the caps.
void drop_cap_tc(ksc_split *s) {
    for (void **p : {(void **)&s->d_cap_tiles, (void **)&s->d_cap_tiles_lpt, (void **)&s->d_ncut,
                     (void **)&s->d_coef_off, (void **)&s->d_coef, (void **)&s->d_irr_items,
                     (void **)&s->d_irr_first, (void **)&s->d_irr}) {
        cudaFree(*p);
        *p = nullptr;
    }
    s->n_cap_tiles = 0;
    s->ctc = ksc::CapTc();
}

// Whether the cell polynomials carry the kernel to the gather's accuracy; top = the largest |K_r|
// within the cut, to which outputs compare (not the sum of the Legendre terms, which lies far
// above it where K_r peaks past the cut or its terms cancel), cuts = ksc::TcCuts::cap.
bool cap_polynomials_ok(const ksc_split *s, double top, double cuts) {
    // Chebyshev interpolation of degree n leaves, of a term l of the kernel, at most about
    // 4 J_{n+1}(l h / 2) ~ 4 (l h / 4)^{n+1} / (n+1)!, h the largest pixel step (1.2826 / nside
    // at the poles).  The coefficients that are multiplied in one part, c_p f^p for p >= n1,
    // |f| <= 1/2, amount to about (l h / 4)^p / (p/2)!^2 of a term (the p-th derivative of
    // J_0); one FP16 part keeps them to 2^-12 of themselves.  Error rms of cap pixels, 1e-7 of the
    // output's, stage / gather, nside 512, 640': l_max 2 nside, 3 pixels (2^-12.9 of the peak): 0.71 /
    // 1.01; 3 nside, 3 pixels (2^-11.8): 0.71 / 1.02; 3 nside, 2.5 pixels (2^-10.5, interpolation bound
    // 1.2e-7): 0.86 / 1.01; 3 nside, 3 pixels, l_cut 500 (2^-10.7): 0.88 / 1.02; 2 nside, 2.5 pixels,
    // l_cut 511 (2^-11.3): 1.09 / 0.99.
    const int n = ksc::cap_tc_degree(), n1 = ksc::cap_tc_split_powers();
    double err = 0.0, single = 0.0, fact = 1.0, half = 1.0;
    for (int i = 2; i <= n + 1; ++i) fact *= i;
    for (int i = 2; i <= n1 / 2; ++i) half *= i;
    for (int l = 0; l <= s->lmax; ++l) {
        const double a = (2.0 * l + 1.0) * std::fabs(s->c_real[l]), x = l * 1.2826 / s->nside / 4.0;
        err += a * 4.0 * std::pow(x, n + 1) / fact;
        single += a * std::pow(x, n1) / (half * half);
    }
    // And where the MMAs' cuts add up (a wide kernel, or one that rings to its cut) the gather is
    // the more accurate one.  Over 55 splits (stage / gather error)^2 is about 0.85 + 0.16 cuts +
    // 0.135 rel^2, rel the single part's share of its bound.  Cuts + 0.8 rel^2, stage / gather: nside 2048,
    // 120' 0.5: 0.77 / 0.84; 2048, 240' 1.06: 0.82 / 0.83; 512, 480' 0.76: 0.81 / 0.86; 1024, 5.8 pixels, 240'
    // 1.15: 0.88 / 0.91; 512, 3.6 pixels, l_cut 460 of 1535: 1.17, 0.90 / 0.84; 512, 3 pixels, l_cut 460 of
    // 1535: 1.3, 0.91 / 0.88; 512, 5.1 pixels, 764': 1.8, 0.95 / 0.87; 512, 6.3 pixels, 1200': 8, 1.76 / 0.99.
    const double peak = 4.0 * kPi * top, rel = single / (std::exp2(-10.5) * peak);
    return err <= 1.25e-7 * peak && rel <= 1.0 && cuts + 0.8 * rel * rel <= 1.16;
}

// Plan of the tensor-core belt stage: the widest window and the most input rings of a
// 16-ring tile, and the power of two that scales the kernel's largest value (for the cap
// stage too).
int plan_belt_tc(ksc_split *s, const ksc::RingGeom &g, const std::vector<int2> &range,
                 const std::vector<ksc::PairInfo> &pairs, const std::vector<int> &pair_base) {
    if (s->path != 0 || s->n_items_belt == 0) return KSC_OK;
    std::vector<float4> tab(s->n_int);
    const cudaError_t e = cudaMemcpy(tab.data(), s->d_tab, sizeof(float4) * tab.size(),
                                     cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "table download");
    double top = 0.0;
    for (const float4 &c : tab)
        top = std::max({top, (double)std::fabs(c.x), std::fabs((double)c.x + c.y + c.z + c.w)});
    // scaled weights and sums stay normal FP32 numbers; otherwise the FFMA kernels
    const int ex = std::isfinite(top) && top > 0.0 ? 13 - std::ilogb(top) : 1000;
    if (ex < -20 || ex > 40) {
        drop_cap_tc(s);
        return KSC_OK;
    }
    const ksc::TcCuts cuts = ksc::tc_cuts(g, s->nside, s->chord_cut, tab.data(), s->n_int);
    if (s->n_cap_tiles && !cap_polynomials_ok(s, top, cuts.cap)) drop_cap_tc(s);
    s->btc.wscale = s->ctc.wscale = (float)std::ldexp(1.0, ex);
    s->ctc.wunscale = 1.0f / s->ctc.wscale;
    s->ctc.domega_lo = (float)(4.0 * kPi / s->plan.npix - (double)s->plan.domega);
    // Below about 8e8 belt pairs the FFMA kernel is the faster one: small maps have few tiles,
    // and the block maxima (5 us) and their scratch come on top (FFMA / tensor stage, us: nside
    // 64, 360': 58 / 72; 256, 160' (2.2e8 pairs): 91 / 99; 512, 60' (5e8): 123 / 122, the call's
    // first pass 483 / 580).  From there on by the estimate at the end.
    if (2.0 / 3.0 * ksc_cost_pairs(s->nside, s->theta_cut) < 8e8) return KSC_OK;
    // The MMAs' cuts add to the error where a ring's sum keeps its size over many of them.  Cuts, stage /
    // FFMA, error rms in 1e-7 of the output's: to 1.3, 0.74 to 1.02 / 0.91 to 1.16; 1.47, 1.20 / 1.14 (the
    // table and the split of the weights err the same way at distance zero); 1.7, 1.08 / 1.09; 2.2, 1.17 / 1.09;
    // 3.7, 1.09 / 1.06; 4.8 (nside 1024, 4.4 pixels, 480'), 1.16 / 1.05; 46 (1024, 7 pixels, l_cut 1100 of 3016,
    // 860'), 2.56 / 1.16.
    if (cuts.belt > 1.4) return KSC_OK;
    const int lo = s->plan.belt_lo, hi = s->plan.belt_hi, nb = ksc::belt_tc_rings();
    int wpos = 0, nq = 0;
    for (int r0 = lo; r0 <= hi; r0 += nb) {
        int q0 = hi, q1 = lo;
        for (int r = r0; r < std::min(r0 + nb, hi + 1); ++r) {
            q0 = std::min(q0, std::max(range[r].x, lo));
            q1 = std::max(q1, std::min(range[r].y, hi));
            for (int q = std::max(range[r].x, lo); q <= std::min(range[r].y, hi); ++q) {
                const int w = pairs[(size_t)pair_base[r] + (q - range[r].x)].w;
                if (w >= 0) wpos = std::max(wpos, ksc::belt_tc_positions(w, g.len[r]));
            }
        }
        nq = std::max(nq, q1 - q0 + 1);
    }
    if (!ksc::belt_tc_plan(s->nside, wpos, nq, &s->btc)) {
        s->btc.n_cols = 0;
        return KSC_OK;
    }
    // A tile spends 2.2 (32 columns) to 3.5 us (256) on an input ring whose window has up to 150
    // positions, and a band of a few rings, which takes the same kernel for the same bits, pays
    // that for sixteen rings.  So only where the whole map's stage takes at most 0.7 of the FFMA
    // kernel's time; estimate and measured ratio: nside 128, 96 pixels 0.71 / 0.65; 256, 32 and 48
    // pixels 0.79 / 0.77 and 0.66 / 0.66; 512, 16 and 24: 0.78 / 0.77 and 0.60 / 0.62; 1024, 8 and 16: 0.79 /
    // 0.71 and 0.55 / 0.55; 2048, 8 and 16: 0.72 / 0.66 and 0.49 / 0.51.
    double ffma = 0.0;
    for (int r = lo; r <= hi; ++r) {
        int rings = 0;
        for (int q = std::max(range[r].x, lo); q <= std::min(range[r].y, hi); ++q)
            rings += pairs[(size_t)pair_base[r] + (q - range[r].x)].hw >= 0.0f;
        const int items = (g.len[r] + ksc::belt_chunk() - 1) / ksc::belt_chunk();
        ffma += items * (0.47 * rings + 0.0108 * s->cost_belt[r]);
    }
    const int waves = (s->n_items_belt + kSms - 1) / kSms;  // fewer items leave SMs short of CTAs
    ffma *= (waves <= 1 ? 3.0 : waves <= 2 ? 1.8 : waves <= 4 ? 1.25 : waves <= 8 ? 1.1 : 0.93) / kSms;
    const int n = s->btc.n_cols;
    const double step = (n >= 256 ? 3.5 : n >= 128 ? 2.9 : n >= 64 ? 2.5 : 2.2) + 0.013 * std::max(wpos - 150, 0);
    const double tensor = std::ceil(ksc::belt_tc_tiles(s->plan, s->btc) / (double)kSms) * nq * step;
    if (tensor > 0.7 * ffma) s->btc.n_cols = 0;
    return KSC_OK;
}

// Time of independent pieces of work on so many slots, the longest first.
double makespan(std::vector<double> t, int slots) {
    std::sort(t.begin(), t.end(), std::greater<double>());
    std::priority_queue<double, std::vector<double>, std::greater<double>> end;
    double last = 0.0;
    for (double x : t) {
        if ((int)end.size() == slots) {
            x += end.top();
            end.pop();
        }
        end.push(x);
        last = std::max(last, x);
    }
    return last;
}

// Plan of the tensor-core cap stage (host): the tiles of the northern rings that have a cap
// input, the sizes of the kernel's buffers, and the ring pairs that go the direct way:
// windows that are whole rings or wider than any farther from the poles, input rings of
// fewer than 32 pixels.
struct CapPlan {
    std::vector<int2> tiles;         // {rings - 1 << 16 | first ring, sectors << 16 | sector}
    std::vector<int2> tiles_lpt;     // the same, longest first
    std::vector<double> cost;        // of each tile
    std::vector<int> ncut;           // per ring pair: the largest |N| within the cut, -1: none
    std::vector<unsigned> coef_off;  // per ring pair, in units of four words; then their end
    std::vector<int> irr, irr_first; // input rings that go the direct way, per output ring
    std::vector<int2> irr_items;
    int n_ext = 0;                   // intervals of the K_r table run past the cut
};
void plan_cap_tc(ksc_split *s, const ksc_split_opts &o, const ksc::RingGeom &g,
                 const std::vector<int2> &range, const std::vector<ksc::PairInfo> &pairs,
                 const std::vector<int> &pair_base, double gather_us, CapPlan *plan) {
    const int nside = s->nside, nr = 4 * nside - 1, eq = (nr - 1) / 2;
    const int belt_lo = nside - 1, belt_hi = 3 * nside - 1;
    if (s->path != 0 || o.exact_weights || o.cap_kernel != 0 || nside < 64 || nside > 4096 ||
        s->theta_cut >= kPi || s->n_items_belt == 0)
        return;
    // Not below 8e9 pairs with a cap ring, and below 5e10 where the gather's small-table tile
    // serves (nside 256, 640' (1.8e9 pairs): gather 0.85, stage 1.09 ms); from there on by the
    // estimates at the end.
    if (ksc_cost_pairs(nside, s->theta_cut) / 3.0 < (s->sym_variant == 1 ? 5e10 : 8e9)) return;
    const double dc = s->chord_cut, n_int = s->n_int;
    const double scale2 = (n_int / dc) * (n_int / dc), nint2 = n_int * n_int;
    // room for the table past the cut (chords up to 2)
    const double h = dc / n_int;
    const int n_ext = s->n_int + (int)std::ceil(1.7 * 1.2826 / nside / h) + 4;
    if (n_ext * h >= 2.0) return;
    int last = -1;  // the last northern ring with a cap input
    for (int r = 0; r <= eq; ++r)
        if (r < belt_lo || range[r].x < belt_lo || range[r].y > belt_hi) last = r;
    auto considered = [&](int r, int q) {
        return !(r >= belt_lo && q >= belt_lo && q <= belt_hi);
    };
    // edge cell of a regular pair from its cut
    auto cell = [&](int nc, int L) { return nc >= L ? (nc - L) / (2 * L) + 1 : 0; };
    constexpr int kDirect = -2;
    plan->ncut.assign(pairs.size(), -1);
    std::vector<int> widest(last + 1, 0);  // widest regular window of a ring; -1: it has others
#pragma omp parallel for schedule(dynamic, 16)
    for (int r = 0; r <= last; ++r) {
        for (int q = range[r].x; q <= range[r].y; ++q) {
            const size_t ip = (size_t)pair_base[r] + (q - range[r].x);
            if (!considered(r, q) || pairs[ip].hw < 0.0f) continue;
            const double dz = g.z[r] - g.z[q];
            const double ds = (g.z[q] - g.z[r]) * (g.z[q] + g.z[r]) / (g.s[r] + g.s[q]);
            const double A2 = (dz * dz + ds * ds) * scale2, B2 = 4.0 * g.s[r] * g.s[q] * scale2;
            if (A2 >= nint2) continue;
            const double sx2 = (nint2 - A2) / B2, c = kPi / (2.0 * (double)g.len[r] * (double)g.len[q]);
            int nc = kDirect;
            if (sx2 < 1.0 && g.len[q] >= 32) {
                nc = (int)std::floor(std::asin(std::sqrt(sx2)) / c);
                if (2 * cell(nc, g.len[r]) + 1 > g.len[q]) nc = kDirect;
            }
            plan->ncut[ip] = nc;
            if (nc == kDirect && g.len[q] >= 32) widest[r] = -1;
            else if (widest[r] >= 0 && nc >= 0) widest[r] = std::max(widest[r], cell(nc, g.len[r]));
        }
    }
    // near the poles windows widen to whole rings: past the widest of the other rings, direct
    const int j_max = *std::max_element(widest.begin(), widest.end());
    plan->irr_first.assign(nr + 1, 0);
    long long widest_n = 0;
    for (int r = 0; r <= last; ++r) {
        plan->irr_first[r] = (int)plan->irr.size();
        for (int q = range[r].x; q <= range[r].y; ++q) {
            int &nc = plan->ncut[(size_t)pair_base[r] + (q - range[r].x)];
            if (nc >= 0 && cell(nc, g.len[r]) > j_max) nc = kDirect;
            if (nc != kDirect) continue;
            nc = -1;
            plan->irr.push_back(q);
            widest_n = std::max(widest_n, 2LL * g.len[r] * g.len[q]);
        }
        if ((int)plan->irr.size() > plan->irr_first[r])
            for (int k0 = 0; k0 < g.len[r] / 4; k0 += 32) plan->irr_items.push_back(make_int2(r, k0));
    }
    for (int r = last + 1; r <= nr; ++r) plan->irr_first[r] = (int)plan->irr.size();
    if (widest_n >= 1LL << 24) {  // (their integers are exact in FP32)
        plan->tiles.clear();
        return;
    }
    // blocks of two rings: input rings, windows, sectors
    // (cap rings or belt rings, not both; an odd ring out alone)
    struct Block {
        int r0, r1;
        int lq_max = 0, jm = 0, wpos = 0, span = 0;  // over the input rings; span: the whole ring's
        double work = 0.0;
    };
    std::vector<Block> blocks;
    for (int r0 = 0, r1; r0 <= last; r0 = r1 + 1) {
        r1 = r0 < belt_lo && ((belt_lo - r0) & 1) ? r0 : std::min(r0 + 1, r0 < belt_lo ? belt_lo - 1 : last);
        blocks.push_back({r0, r1});
    }
#pragma omp parallel for schedule(dynamic, 8)
    for (size_t i = 0; i < blocks.size(); ++i) {
        Block &b = blocks[i];
        const int L0 = g.len[b.r0], L1 = g.len[b.r1];
        const int q1 = std::max(range[b.r0].y, range[b.r1].y);
        for (int q = std::min(range[b.r0].x, range[b.r1].x); q <= q1; ++q) {
            int w = -1;
            for (int r = b.r0; r <= b.r1; ++r) {
                if (q < range[r].x || q > range[r].y) continue;
                const int nc = plan->ncut[(size_t)pair_base[r] + (q - range[r].x)];
                if (nc >= 0) w = std::max(w, cell(nc, g.len[r]));
            }
            if (w < 0) continue;
            const int Lq = g.len[q], tq = g.phase[q];
            auto pos = [&](int k, int t, int L) {
                return (int)(((long long)(2 * k + t) * Lq + (long long)(1 - tq) * L) / (2 * L));
            };
            const int lo = std::min(pos(0, g.phase[b.r0], L0), pos(0, g.phase[b.r1], L1));
            const int hi = std::max(pos(L0 - 1, g.phase[b.r0], L0), pos(L1 - 1, g.phase[b.r1], L1));
            b.span = std::max(b.span, hi - lo + 1);
            b.lq_max = std::max(b.lq_max, Lq);
            b.jm = std::max(b.jm, w);
            const int np = ksc::cap_tc_positions(w, Lq);
            b.wpos = std::max(b.wpos, np);
            // us on an SM: 5.7 for windows up to about 80 positions, then the products
            b.work += 5.7 + 0.024 * std::max(np - 80, 0);
        }
    }
    ksc::CapTc c;
    for (const Block &b : blocks) {
        // (cap rings without a regular pair have a tile too: it writes what the direct ones add to)
        if (b.lq_max == 0 && b.r0 >= belt_lo) continue;
        // a sector's positions: L' / n, the rings' different first outputs, rounding
        const int L0 = g.len[b.r0], L1 = g.len[b.r1], span = ksc::cap_tc_span();
        const int slack = (b.lq_max + L0 - 1) / L0 + 4;
        const bool one = b.span <= span;
        const int n_sec = one ? 1 : slack < span ? std::max((b.lq_max + span - slack - 1) / (span - slack), 2) : L0 + 1;
        if (n_sec > L0) {  // (the shortest rings, cuts of most of the sphere)
            plan->tiles.clear();
            return;
        }
        c.wpos = std::max(c.wpos, b.wpos);
        c.nq = std::max(c.nq, std::max(range[b.r0].y, range[b.r1].y) - std::min(range[b.r0].x, range[b.r1].x) + 1);
        c.jcap = std::max(c.jcap, b.jm + 1);
        c.tcap = std::max(c.tcap, (std::max(L0, L1) + n_sec - 1) / n_sec + 1);
        c.span = std::max(c.span, one ? b.span : (b.lq_max + n_sec - 1) / n_sec + slack);
        for (int t = 0; t < n_sec; ++t) {
            plan->tiles.push_back(make_int2((b.r1 - b.r0) << 16 | b.r0, n_sec << 16 | t));
            plan->cost.push_back(b.work);
        }
    }
    c.span = std::min((c.span + 15) & ~15, ksc::cap_tc_span());
    // the coefficients: up to 8 GB (2.4 GB at nside 2048 with a 240' cut); beyond it the
    // gather, which keeps none
    const auto words4 = [&](int r, size_t ip) {
        return plan->ncut[ip] >= 0 ? ksc::cap_tc_words(cell(plan->ncut[ip], g.len[r])) / 4 : 0;
    };
    std::vector<unsigned long long> first(last + 2, 0ull);
#pragma omp parallel for schedule(dynamic, 16)
    for (int r = 0; r <= last; ++r)
        for (size_t ip = pair_base[r]; ip < (size_t)pair_base[r + 1]; ++ip) first[r + 1] += words4(r, ip);
    for (int r = 0; r <= last; ++r) first[r + 1] += first[r];
    const unsigned long long n4 = first[last + 1];
    plan->coef_off.assign(pairs.size() + 1, 0u);
#pragma omp parallel for schedule(dynamic, 16)
    for (int r = 0; r <= last; ++r) {
        unsigned long long at = first[r];
        for (size_t ip = pair_base[r]; ip < (size_t)pair_base[r + 1]; ++ip) {
            plan->coef_off[ip] = (unsigned)at;
            at += words4(r, ip);
        }
    }
    if (!ksc::cap_tc_fits(c) || n4 * 16 > 8ull << 30) plan->tiles.clear();
    if (plan->tiles.empty()) return;
    // The stage has to be the faster one: its tiles, and the direct pairs (sixteen warps share
    // a ring's list: 20 ns a pixel), against the gather.  Measured / estimated ratio to the
    // gather, three-pixel beams: nside 256, 128 pixels 0.74 / 0.81; 512, 96 pixels 0.79 / 0.69; 1024,
    // 64 pixels 0.98 / 0.98; 2048, 16, 32 and 64 pixels 1.33 / 1.33, 1.07 / 1.06 and 0.83 / 0.85;
    // 4096, 16 pixels 1.45 / 1.49 (a tile spends 5 us on an input ring however short the window);
    // 256, 512 pixels 1.40 / 1.77 (all direct).
    std::vector<double> direct;
    for (const int2 &it : plan->irr_items) {
        double us = 0.0;
        for (int e = plan->irr_first[it.x]; e < plan->irr_first[it.x + 1]; ++e)
            us += 0.66 + 0.020 * g.len[plan->irr[e]];
        direct.push_back(us);
    }
    if (makespan(plan->cost, kSms) + makespan(direct, kSms) > gather_us) {
        plan->tiles.clear();
        return;
    }
    plan->coef_off.back() = (unsigned)n4;
    c.ring_first = 0;
    c.ring_end = last;
    plan->n_ext = n_ext;
    s->ctc = c;
}

// Uploads the cap stage's tiles and lays out its coefficients.  The stage is left out (the
// gather sums the caps) where there is no ample room for them, and where a coefficient does not fit
// an FP16 number: the scale comes from the kernel inside the cut, the polynomials of the cells
// that the cut divides from the kernel past it too, which may be larger.
int build_cap_tc(ksc_split *s, const CapPlan &cap, ksc::CapCoef cc) {
    if (s->n_cap_tiles == 0) return KSC_OK;
    // (no more than an eighth of what is free: a program that keeps many splits, or maps of its
    // own, can fill the device with them as it could before the stage)
    const size_t bytes = 16ull * cap.coef_off.back();
    size_t free_bytes = 0, total = 0;
    cudaError_t e = cudaMemGetInfo(&free_bytes, &total);
    if (e == cudaSuccess) e = bytes <= free_bytes / 8 ? dev_malloc((void **)&s->d_coef, bytes) : cudaErrorMemoryAllocation;
    if (e != cudaSuccess) {
        if (e != cudaErrorMemoryAllocation) return cuda_fail(e, "cap coefficients");
        cudaGetLastError();
        s->d_coef = nullptr;
        drop_cap_tc(s);
        return KSC_OK;
    }
    if ((e = dev_upload(&s->d_cap_tiles, cap.tiles.data(), cap.tiles.size())) != cudaSuccess ||
        (e = dev_upload(&s->d_cap_tiles_lpt, cap.tiles_lpt.data(), cap.tiles_lpt.size())) !=
            cudaSuccess ||
        (e = dev_upload(&s->d_ncut, cap.ncut.data(), cap.ncut.size())) != cudaSuccess ||
        (e = dev_upload(&s->d_coef_off, cap.coef_off.data(), cap.coef_off.size())) != cudaSuccess ||
        (e = dev_upload(&s->d_irr_items, cap.irr_items.data(), cap.irr_items.size())) != cudaSuccess ||
        (e = dev_upload(&s->d_irr_first, cap.irr_first.data(), cap.irr_first.size())) != cudaSuccess ||
        (e = dev_upload(&s->d_irr, cap.irr.data(), cap.irr.size())) != cudaSuccess)
        return cuda_fail(e, "cap tiles");
    s->ctc.d_ncut = s->d_ncut;
    s->ctc.d_coef_off = s->d_coef_off;
    s->ctc.d_coef = cc.d_coef = s->d_coef;
    int too_large = 0;
    e = cudaMemsetAsync(cc.d_too_large, 0, sizeof(int), 0);
    if (e == cudaSuccess) e = ksc::launch_cap_coef(s->plan, s->ctc, cc, 0);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&too_large, cc.d_too_large, sizeof(int), cudaMemcpyDeviceToHost, 0);
    if (e == cudaSuccess) e = cudaStreamSynchronize(0);
    if (e != cudaSuccess) return cuda_fail(e, "cap coefficients");
    if (too_large) drop_cap_tc(s);
    return KSC_OK;
}

void make_slots(ksc_split *s);

// Geometry, work list and device table for the real-space part s->c_real.
int finish_split(ksc_split *s, const ksc_split_opts &o) {
    const int nside = s->nside;
    g_alloc_count = 0;
    s->chord_cut = 2.0 * std::sin(0.5 * s->theta_cut);
    int n_int = o.n_intervals;
    // ~96 intervals per shortest l_max wavelength; the chord compresses
    // theta by cos(theta/2), so wide cuts need proportionally more
    const double squeeze = std::max(std::cos(0.5 * s->theta_cut), 1e-3);
    const double n_auto = 96.0 * s->chord_cut * std::max(s->lmax, 1) / (2.0 * kPi * squeeze);
    if (n_int <= 0) {
        n_int = (int)std::ceil(n_auto);
        n_int = std::max(256, std::min(n_int, ksc::kMaxIntervals));
    }
    if (n_int > ksc::kMaxIntervals) return fail(KSC_ERR_ARG, "n_intervals above 8192");
    s->n_int = n_int;

    ksc::RingGeom g;
    ksc::ring_geometry(nside, &g);
    const int nr = 4 * nside - 1;
    std::vector<ksc::DevRing> rings(nr);
    std::vector<double> th(nr);
    for (int r = 0; r < nr; ++r) {
        rings[r] = {g.z[r], g.s[r], g.len[r], g.start[r], g.phase[r], 0};
        th[r] = std::atan2(g.s[r], g.z[r]);
    }
    // Input-ring range of each output ring: |theta_r - theta_r'| <= theta_cut.
    std::vector<int2> range(nr);
    const double tc = s->theta_cut + 1e-9;
    for (int r = 0; r < nr; ++r) {
        if (s->theta_cut >= kPi) {
            range[r] = make_int2(0, nr - 1);
            continue;
        }
        int lo = (int)(std::lower_bound(th.begin(), th.end(), th[r] - tc) - th.begin());
        int hi = (int)(std::upper_bound(th.begin(), th.end(), th[r] + tc) - th.begin()) - 1;
        range[r] = make_int2(std::max(lo, 0), std::min(hi, nr - 1));
    }
    s->range = range;
    // Work lists (ring by ring, with per-ring prefixes for latitude bands):
    //  - all:  256-pixel chunks of every ring (pair counting, fallback);
    //  - belt: belt_chunk()-pixel chunks of belt rings (circulant kernel);
    //  - sym:  first-quarter chunks of northern rings (and the equator) for the
    //          symmetric gather: cap rings, plus belt rings that reach a cap
    //          (every northern ring when the belt kernel is not used).
    const int belt_lo = nside - 1, belt_hi = 3 * nside - 1, eq = 2 * nside - 1;
    std::vector<ksc::WorkItem> items, items_sym;
    std::vector<int2> items_belt;
    s->ring_first_item.assign(nr + 1, 0);
    s->ring_first_sym.assign(nr + 1, 0);
    s->ring_first_belt.assign(nr + 1, 0);
    const int bc = ksc::belt_chunk();
    int max_nd = 0, w_ext = 0;
    for (int r = 0; r < nr; ++r) {
        s->ring_first_item[r] = (int)items.size();
        s->ring_first_sym[r] = (int)items_sym.size();
        s->ring_first_belt[r] = (int)items_belt.size();
        for (int k0 = 0; k0 < g.len[r]; k0 += 256) items.push_back({r, k0});
        const bool belt = r >= belt_lo && r <= belt_hi;
        const bool reaches_cap = range[r].x < belt_lo || range[r].y > belt_hi;
        if (r <= eq && (!belt || reaches_cap || o.path == 1))
            for (int k0 = 0; k0 < ksc::sym_classes(g.len[r], g.phase[r]);
                 k0 += ksc::sym_chunk(nside))
                items_sym.push_back({r, k0});
        if (belt) {
            for (int k0 = 0; k0 < g.len[r]; k0 += bc) items_belt.push_back(make_int2(r, k0));
            // widest circulant window of this ring (same arithmetic as the kernel)
            const int L = g.len[r];
            for (int q = std::max(range[r].x, belt_lo); q <= std::min(range[r].y, belt_hi); ++q) {
                double ss = g.s[r] * g.s[q];
                double cdp = (1.0 - 0.5 * s->chord_cut * s->chord_cut - g.z[r] * g.z[q]) / ss;
                double dphi = cdp <= -1.0 ? 4.0 * kPi : (cdp >= 1.0 ? 0.0 : std::acos(cdp));
                int w = (int)std::ceil(dphi * L / (2.0 * kPi)) + 1;  // same as PairInfo::w
                int n = std::min(2 * w + 1, L);
                max_nd = std::max(max_nd, n);
                w_ext = std::max(w_ext, 2 * w + 1 >= L ? L / 2 : w);
            }
        }
    }
    std::vector<int2> items_mma;
    for (int r = belt_lo; r <= belt_hi; ++r)
        for (int k0 = 0; k0 < g.len[r]; k0 += ksc::belt_mma_block())
            items_mma.push_back(make_int2(r, k0));
    s->n_items_mma = (int)items_mma.size();
    s->w_cap = (max_nd + 2 * 13 + 3) & ~3;
    s->tensor = o.tensor;
    s->mma_ext0 = ((w_ext + 32) + 31) & ~31;
    s->mma_ntiles = (s->mma_ext0 + 4 * nside + (((w_ext + 160) + 31) & ~31)) / 32;
    // the belt tensor kernel needs its weight window in shared memory
    if (s->tensor == 2 && ksc::belt_mma_smem(s->w_cap) > 220u * 1024) s->tensor = 1;
    s->ring_first_item[nr] = (int)items.size();
    s->ring_first_sym[nr] = (int)items_sym.size();
    s->ring_first_belt[nr] = (int)items_belt.size();
    s->n_items = (int)items.size();
    s->n_items_sym = (int)items_sym.size();
    s->n_items_belt = (int)items_belt.size();
    // shared-memory segment: chunk + padded window + alignment, with slack for
    // rounding differences between host and device acos
    const int seg = bc + max_nd + 6 * 13 + 16;
    s->seg_cap = (seg + 3) & ~3;
    s->max_nd = max_nd;
    const bool belt_ok = s->n_items_belt > 0 && 12ull * s->seg_cap <= 200ull * 1024;
    s->path = o.path;
    if (!belt_ok && o.path == 0) {
        // belt windows too wide for shared memory: the general gather does it all
        s->path = 1;
    }
    if (s->path == 1) {
        s->n_items_belt = 0;
        s->seg_cap = 0;
    }

    // Ring-pair geometry (FP64 on the host, once per split).
    std::vector<int> pair_base(nr + 1, 0);
    for (int r = 0; r < nr; ++r) pair_base[r + 1] = pair_base[r] + (range[r].y - range[r].x + 1);
    std::vector<ksc::PairInfo> pairs((size_t)pair_base[nr]);
    std::vector<ksc::XInfo> xinfo((size_t)pair_base[nr]);
    std::vector<ksc::XOdd> xodd((size_t)pair_base[nr]);
    {
        const double dc = s->chord_cut;
        const double cos_cut = 1.0 - 0.5 * dc * dc;
        const double scale2 = ((double)n_int / dc) * ((double)n_int / dc);
        const double dc2 = s->theta_cut >= kPi ? 5.0 : dc * dc;
        // x cells are sized in intervals of the automatic table size, so a coarser
        // user table gets proportionally narrower cells (in its own intervals)
        const double xscale = std::min(1.0, (double)n_int / std::max(n_auto, 1.0));
#pragma omp parallel for schedule(dynamic, 16)
        for (int r = 0; r < nr; ++r) {
            for (int q = range[r].x; q <= range[r].y; ++q) {
                const double dz = g.z[r] - g.z[q];
                const double ds = (g.z[q] - g.z[r]) * (g.z[q] + g.z[r]) / (g.s[r] + g.s[q]);
                const double A = dz * dz + ds * ds;
                const double ss = g.s[r] * g.s[q];
                const int Lq = g.len[q];
                ksc::PairInfo pi;
                const ksc::DF a = ksc::df_from_double(A * scale2);
                const ksc::DF b = ksc::df_from_double(4.0 * ss * scale2);
                const ksc::DF c = ksc::df_from_double(kPi / (2.0 * (double)g.len[r] * (double)Lq));
                pi.Ah = a.h; pi.Al = a.l; pi.Bh = b.h; pi.Bl = b.l; pi.ch = c.h; pi.cl = c.l;
                if (A > dc2 * (1.0 + 1e-6)) {
                    pi.hw = -1.0f;
                    pi.w = -1;
                } else {
                    const double cdp = (cos_cut - g.z[r] * g.z[q]) / ss;
                    const double dphi = cdp <= -1.0 ? 4.0 * kPi : (cdp >= 1.0 ? 0.0 : std::acos(cdp));
                    pi.hw = (float)(dphi * Lq / (2.0 * kPi)) + 1.0f;
                    pi.w = (int)std::ceil(dphi * Lq / (2.0 * kPi)) + 1;
                }
                pairs[(size_t)pair_base[r] + (q - range[r].x)] = pi;
                xinfo[(size_t)pair_base[r] + (q - range[r].x)] =
                    (s->theta_cut >= kPi || o.exact_weights)
                        ? ksc::XInfo{}
                        : ksc::make_xinfo(A * scale2, 4.0 * ss * scale2,
                                          kPi / (2.0 * (double)g.len[r] * (double)Lq),
                                          (double)n_int * (double)n_int, pi.hw, g.len[r], Lq,
                                          xscale);
                xodd[(size_t)pair_base[r] + (q - range[r].x)] =
                    (s->theta_cut >= kPi || o.exact_weights)
                        ? ksc::XOdd{}
                        : ksc::make_xodd(A * scale2, 4.0 * ss * scale2,
                                         kPi / (2.0 * (double)g.len[r] * (double)Lq),
                                         (double)n_int * (double)n_int, pi.hw, g.len[r], Lq,
                                         xscale, ksc::kXCap);
            }
        }
    }

    // Work per output pixel of each ring (window positions over its input
    // rings), for ordering batched work longest first.
    s->cost_belt.assign(nr, 0.0);
    s->cost_sym.assign(nr, 0.0);
    for (int r = 0; r < nr; ++r) {
        const bool belt_r = r >= belt_lo && r <= belt_hi;
        for (int q = range[r].x; q <= range[r].y; ++q) {
            const ksc::PairInfo &pi = pairs[(size_t)pair_base[r] + (q - range[r].x)];
            if (pi.hw < 0.0f) continue;
            const double span = std::min(2.0 * pi.hw + 3.0, (double)g.len[q]);
            const bool belt_q = q >= belt_lo && q <= belt_hi;
            if (s->path == 0 && belt_r && belt_q) s->cost_belt[r] += span;
            else s->cost_sym[r] += span;
        }
    }

    std::vector<double> gather_rings, gather_pos;  // of a northern ring's items
    // Share of the symmetric gather's weight evaluations that the dphi tables serve
    // (per northern output ring: reflection classes x window positions per input ring).
    {
        const int eqr = (nr - 1) / 2;
        double all = 0.0, tab = 0.0, small = 0.0;
        gather_rings.assign(nr, 0.0);
        gather_pos.assign(nr, 0.0);
        for (int r = 0; r <= eqr; ++r) {
            const bool belt_r = r >= belt_lo && r <= belt_hi;
            const double cls = (double)ksc::sym_classes(g.len[r], g.phase[r]);
            for (int q = range[r].x; q <= range[r].y; ++q) {
                const size_t ip = (size_t)pair_base[r] + (q - range[r].x);
                if (pairs[ip].hw < 0.0f) continue;
                const bool belt_q = q >= belt_lo && q <= belt_hi;
                if (s->path == 0 && belt_r && belt_q && !items_belt.empty()) continue;
                const double pos = std::min(2.0 * pairs[ip].hw + 3.0, (double)g.len[q]), n = cls * pos;
                gather_rings[r] += 1.0;
                gather_pos[r] += pos;
                all += n;
                if (xodd[ip].nct > 0) tab += n;
                if (xodd[ip].nct > 0 && xodd[ip].nct + 1 <= ksc::kXCapSmall) small += n;
            }
        }
        s->frac_tabulated = all > 0.0 ? tab / all : 0.0;
        // 128-class items with small tables (three CTAs per SM) where nearly all pairs that
        // have a table fit one (pairs that do not take their weights one by one) and a map has
        // items for two waves of two CTAs per SM.  Full / small tables, us: nside 512, 60'
        // (about 800 items): 240 / 202; nside 256, 640' (about 300): 850 / 1070.  A batch fills
        // its waves with several maps (32 of nside 256: 23.9 / 19.0 ms; 16 of 512: 35.1 / 28.7).
        s->sym_small_ok = tab - small <= 0.01 * all;
        s->sym_variant = ksc::sym_chunk(nside) == ksc::sym_variant_chunk(0) ? 0
                         : s->sym_small_ok && s->n_items_sym >= 4 * 152    ? 1
                                                                           : 2;
    }

    // The gather's time, about: us per item, input ring and window position, by tile (measured
    // over nside 512 to 4096, 4 to 64 pixels: within 10%; with the full tables of nside 64 to
    // 256 about 30%, of which the two factors for maps of few items take half).
    double gather_us;
    {
        const double us_ring[3] = {7.06, 3.41, 1.88}, us_pos[3] = {0.140, 0.091, 0.105};
        const int v = s->sym_variant;
        std::vector<double> t;
        for (const ksc::WorkItem &it : items_sym)
            t.push_back(us_ring[v] * gather_rings[it.ring] + us_pos[v] * gather_pos[it.ring]);
        gather_us = makespan(t, (v == 1 ? 3 : 2) * kSms);
        if (v == 2 && (int)t.size() <= 6 * kSms) gather_us *= (int)t.size() <= kSms ? 0.8 : 1.25;
    }
    CapPlan cap;
    plan_cap_tc(s, o, g, range, pairs, pair_base, gather_us, &cap);
    const int n_ext = cap.n_ext;

    // The symmetric items longest first, for whole-map launches: CTAs claim items
    // in list order, so the long items start first and the short ones fill the tail.
    // The tensor cap kernel has items of its own size.
    auto lpt = [&](std::vector<ksc::WorkItem> v, int chunk) {
        auto cost = [&](const ksc::WorkItem &w) {
            const int n_cls = ksc::sym_classes(g.len[w.ring], g.phase[w.ring]);
            const int cnt = std::min(chunk, n_cls - w.k0);
            return cnt * s->cost_sym[w.ring] * (w.ring == eq ? 1.0 : 2.0);
        };
        std::stable_sort(v.begin(), v.end(), [&](const ksc::WorkItem &x, const ksc::WorkItem &y) {
            return cost(x) > cost(y);
        });
        return v;
    };
    std::vector<ksc::WorkItem> items_lpt = lpt(items_sym, ksc::sym_chunk(nside));
    // 128-class items of the tensor kernels, ring by ring (with per-ring prefixes
    // for latitude bands) and longest first
    std::vector<ksc::WorkItem> items_smma;
    s->ring_first_smma.assign(nr + 1, 0);
    {
        size_t i = 0;
        for (int r = 0; r < nr; ++r) {
            s->ring_first_smma[r] = (int)items_smma.size();
            if (i < items_sym.size() && items_sym[i].ring == r) {
                const int n_cls = ksc::sym_classes(g.len[r], g.phase[r]);
                for (int k0 = 0; k0 < n_cls; k0 += ksc::sym_mma_chunk())
                    items_smma.push_back({r, k0});
                while (i < items_sym.size() && items_sym[i].ring == r) ++i;
            }
        }
        s->ring_first_smma[nr] = (int)items_smma.size();
    }
    std::vector<ksc::WorkItem> items_smma_lpt = lpt(items_smma, ksc::sym_mma_chunk());
    {
        std::vector<int> order(cap.tiles.size());
        for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
        std::stable_sort(order.begin(), order.end(),
                         [&](int a, int b) { return cap.cost[a] > cap.cost[b]; });
        for (int i : order) cap.tiles_lpt.push_back(cap.tiles[i]);
        s->n_cap_tiles = (int)cap.tiles.size();
        s->cap_tile_us = cap.cost;
        s->cap_tile_first.assign(nr + 1, 0);
        size_t i = 0;
        for (int r = 0; r <= nr; ++r) {
            while (i < cap.tiles.size() && (cap.tiles[i].x & 0xffff) < r) ++i;
            s->cap_tile_first[r] = (int)i;
        }
        s->irr_item_first.assign(nr + 1, 0);
        i = 0;
        for (int r = 0; r <= nr; ++r) {
            while (i < cap.irr_items.size() && cap.irr_items[i].x < r) ++i;
            s->irr_item_first[r] = (int)i;
        }
    }
    const bool plan_cap = s->n_cap_tiles > 0;
    std::vector<float2> ringc(plan_cap ? nr : 0);
    for (size_t r = 0; r < ringc.size(); ++r) {
        const ksc::DF c = ksc::df_from_double(kPi / (double)g.len[r]);
        ringc[r] = make_float2(c.h, c.l);
    }
    s->n_items_smma = (int)items_smma.size();
    s->cap_kernel = o.cap_kernel;

    cudaError_t e;
    cudaGetDevice(&s->device);
    if ((e = dev_upload(&s->d_pairs, pairs.data(), pairs.size())) != cudaSuccess)
        return cuda_fail(e, "upload ring-pair table");
    if ((e = dev_upload(&s->d_xinfo, xinfo.data(), xinfo.size())) != cudaSuccess)
        return cuda_fail(e, "upload ring-pair x tables");
    if ((e = dev_upload(&s->d_xodd, xodd.data(), xodd.size())) != cudaSuccess)
        return cuda_fail(e, "upload ring-pair odd-step tables");
    if ((e = dev_upload(&s->d_pair_base, pair_base.data(), pair_base.size())) != cudaSuccess)
        return cuda_fail(e, "upload ring-pair offsets");
    if ((e = dev_upload(&s->d_rings, rings.data(), rings.size())) != cudaSuccess)
        return cuda_fail(e, "upload ring table");
    if ((e = dev_upload(&s->d_range, range.data(), range.size())) != cudaSuccess)
        return cuda_fail(e, "upload ring ranges");
    if ((e = dev_upload(&s->d_items, items.data(), items.size())) != cudaSuccess)
        return cuda_fail(e, "upload work list");
    if ((e = dev_upload(&s->d_items_sym, items_sym.data(), items_sym.size())) != cudaSuccess)
        return cuda_fail(e, "upload work list");
    if ((e = dev_upload(&s->d_items_sym_lpt, items_lpt.data(), items_lpt.size())) != cudaSuccess)
        return cuda_fail(e, "upload work list");
    if ((e = dev_upload(&s->d_items_smma, items_smma.data(), items_smma.size())) != cudaSuccess)
        return cuda_fail(e, "upload work list");
    if ((e = dev_upload(&s->d_items_smma_lpt, items_smma_lpt.data(), items_smma_lpt.size())) !=
        cudaSuccess)
        return cuda_fail(e, "upload work list");
    if ((e = dev_upload(&s->d_items_belt, items_belt.data(), items_belt.size())) != cudaSuccess)
        return cuda_fail(e, "upload work list");
    if ((e = dev_upload(&s->d_items_mma, items_mma.data(), items_mma.size())) != cudaSuccess)
        return cuda_fail(e, "upload work list");
    if ((e = dev_malloc((void **)&s->d_err, sizeof(int))) != cudaSuccess)
        return cuda_fail(e, "error flag");
    if ((e = cudaMemset(s->d_err, 0, sizeof(int))) != cudaSuccess)
        return cuda_fail(e, "error flag");

    // Table build on the GPU: FP64 Legendre recurrence per node (csrc/table.cu).
    double *d_c = nullptr;
    if ((e = dev_upload(&d_c, s->c_real.data(), s->c_real.size())) != cudaSuccess)
        return cuda_fail(e, "upload coefficients");
    // With a tensor-core cap stage the table runs past the cut; its intervals up to the
    // cut, and the entry at the cut with its higher terms dropped, are the table proper.
    const int n_build = plan_cap ? n_ext : n_int;
    // nodes | the table run past the cut, its rounding errors, pi / L per ring, a flag
    const size_t b_nodes = sizeof(double) * 2 * (size_t)(n_build + 1);
    const size_t b_ext = plan_cap ? sizeof(float4) * (size_t)(n_build + 1) : 0;
    const size_t b_lo = plan_cap ? (sizeof(float) * (size_t)n_build + 15) / 16 * 16 : 0;
    unsigned char *d_scratch = nullptr;
    if ((e = dev_malloc((void **)&d_scratch,
                        (b_nodes + 15) / 16 * 16 + b_ext + b_lo + sizeof(float2) * ringc.size() + sizeof(int))) !=
        cudaSuccess) {
        cudaFree(d_c);
        return cuda_fail(e, "allocate table nodes");
    }
    if ((e = dev_malloc((void **)&s->d_tab, sizeof(float4) * (n_int + 1))) != cudaSuccess) {
        cudaFree(d_c); cudaFree(d_scratch);
        return cuda_fail(e, "allocate table");
    }
    double *d_nodes = reinterpret_cast<double *>(d_scratch);
    float4 *d_ext = reinterpret_cast<float4 *>(d_scratch + (b_nodes + 15) / 16 * 16);
    float *d_lo = reinterpret_cast<float *>(d_ext + b_ext / sizeof(float4));
    float2 *d_ringc = reinterpret_cast<float2 *>(reinterpret_cast<unsigned char *>(d_lo) + b_lo);
    float4 *built = plan_cap ? d_ext : s->d_tab;
    ksc::TableBuild tb{d_c, s->lmax, n_build, s->chord_cut / n_int, built, d_nodes, 1};
    if (plan_cap) tb.d_lo = d_lo;
    e = ksc::launch_table_build(tb, 0);
    if (e == cudaSuccess && plan_cap) {
        e = cudaMemcpyAsync(s->d_tab, built, sizeof(float4) * (n_int + 1),
                            cudaMemcpyDeviceToDevice, 0);
        if (e == cudaSuccess) e = cudaMemsetAsync(&s->d_tab[n_int].z, 0, 2 * sizeof(float), 0);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(d_ringc, ringc.data(), sizeof(float2) * ringc.size(),
                                cudaMemcpyHostToDevice, 0);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(0);
    cudaFree(d_c);
    struct Scratch {  // freed when the construction ends, whichever way
        void *p;
        ~Scratch() { cudaFree(p); }
    } scratch_owner{d_scratch};
    if (e != cudaSuccess) return cuda_fail(e, "table build");

    ksc::ConvPlan &p = s->plan;
    p.nside = nside;
    p.npix = 12 * nside * nside;
    p.nrings = nr;
    p.d_rings = s->d_rings;
    p.d_range = s->d_range;
    p.d_pairs = s->d_pairs;
    p.d_xinfo = s->d_xinfo;
    p.d_xodd = s->d_xodd;
    p.d_pair_base = s->d_pair_base;
    p.d_tab = s->d_tab;
    p.n_int = n_int;
    p.inv_h = (float)(n_int / s->chord_cut);
    p.dc2 = (float)(s->chord_cut * s->chord_cut);
    p.scale2 = ((double)n_int / s->chord_cut) * ((double)n_int / s->chord_cut);
    p.nint2 = (float)((double)n_int * (double)n_int);
    // theta_cut = pi: every pair, whatever the rounding of antipodal chords
    if (s->theta_cut >= kPi) {
        p.dc2 = 5.0f;
        p.nint2 = (float)(1.25 * (double)n_int * (double)n_int);
    }
    p.cos_cut = 1.0 - 0.5 * s->chord_cut * s->chord_cut;
    p.domega = (float)(4.0 * kPi / (double)p.npix);
    p.belt_lo = belt_lo;
    p.belt_hi = belt_hi;
    {
        const ksc::DF c1 = ksc::df_from_double(kPi / (2.0 * 4.0 * nside));
        p.belt_c1h = c1.h;
        p.belt_c1l = c1.l;
    }
    int rc = plan_belt_tc(s, g, range, pairs, pair_base);
    ksc::CapCoef cc{d_ext, d_lo, d_ringc, nullptr, reinterpret_cast<int *>(d_ringc + ringc.size()),
                    n_ext, (float)((double)n_ext * n_ext), {}, {}};
    if (!rc && plan_cap) rc = build_cap_tc(s, cap, cc);
    if (!rc) make_slots(s);
    return rc;
}

int check_common(int lmax, int nside, double theta_cut) {
    if (lmax < 1 || lmax > 16384) return fail(KSC_ERR_ARG, "lmax outside 1..16384");
    if (!valid_nside(nside)) return fail(KSC_ERR_ARG, "nside must be a power of two in 1..8192");
    if (!(theta_cut > 0.0) || theta_cut > kPi) return fail(KSC_ERR_ARG, "theta_cut outside (0, pi]");
    return KSC_OK;
}

ksc_split_opts resolve_opts(const ksc_split_opts *opts) {
    ksc_split_opts o;
    ksc_default_opts(&o);
    if (opts) {
        o = *opts;
        if (o.oversample <= 0) o.oversample = 2;
        if (!(o.svd_rcond > 0.0)) o.svd_rcond = 1e-6;
        if (!(o.alpha > 0.0)) o.alpha = 5.0;
        if (o.path != 1) o.path = 0;
        if (o.tensor != 1 && o.tensor != 2) o.tensor = 0;
        if (o.cut_continuity < KSC_CUT_C1 || o.cut_continuity > KSC_CUT_FREE)
            o.cut_continuity = KSC_CUT_C1;
        if (o.exact_weights != 1) o.exact_weights = 0;
        if (o.cap_kernel != 1) o.cap_kernel = 0;
    }
    return o;
}

int check_maps(const ksc_split *s, const void *a, const void *b) {
    if (!s) return fail(KSC_ERR_ARG, "null split");
    if (!a || !b) return fail(KSC_ERR_ARG, "null map pointer");
    if (a == b) return fail(KSC_ERR_ARG, "in and out must be different buffers");
    if (((uintptr_t)a | (uintptr_t)b) & 15u)
        return fail(KSC_ERR_ARG, "maps must be 16-byte aligned");
    return KSC_OK;
}

// One convolution call's scratch: a slot of the split whose last call has ended (the
// stream-ordered pool gives its memory back at every synchronisation, and a call that follows
// one pays 0.1 ms for it: a band of nine belt rings runs 0.03 to 0.5 ms), else from the
// stream-ordered allocator; a captured call's is the graph's own.
struct CallScratch : ksc::ConvScratch {
    void *mem = nullptr;
    cudaStream_t st = nullptr;
    const ksc_split *split = nullptr;
    ksc_split::ScratchSlot *slot = nullptr;
    CallScratch() = default;
    CallScratch(const CallScratch &) = delete;
    CallScratch &operator=(const CallScratch &) = delete;
    ~CallScratch() {
        if (slot) {
            const cudaError_t e = cudaEventRecord(slot->done, st);
            std::lock_guard<std::mutex> lk(split->slot_mu);
            slot->taken = e != cudaSuccess;  // (without its event the slot is not used again)
        } else if (mem) {
            cudaFreeAsync(mem, st);
        }
    }
    bool take_slot(const ksc_split *s) {
        // (another thread's capture in global mode forbids event queries to this one)
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        cudaThreadExchangeStreamCaptureMode(&mode);
        std::lock_guard<std::mutex> lk(s->slot_mu);
        for (ksc_split::ScratchSlot &c : s->slots) {
            if (!c.mem || c.taken) continue;
            if (cudaEventQuery(c.done) == cudaSuccess) {
                c.taken = true;
                split = s;
                slot = &c;
                mem = c.mem;
                break;
            }
            cudaGetLastError();  // not ready
        }
        cudaThreadExchangeStreamCaptureMode(&mode);
        return slot != nullptr;
    }
};

// Takes the scratch and starts the launches that fill it.  Without room for it (npix / 16
// bytes a map) the FFMA kernels do it all.
cudaError_t start_scratch(const ksc_split *s, const ksc::MapSet &maps, int n_maps,
                          const ksc::ConvUse &use, cudaStream_t st, CallScratch *w) {
    const size_t bytes = ksc::conv_scratch_bytes(s, n_maps, use);
    if (bytes == 0) return cudaSuccess;
    w->st = st;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &capture);
    if (e != cudaSuccess) return e;
    if (bytes > s->slot_bytes || capture != cudaStreamCaptureStatusNone || !w->take_slot(s)) {
        e = cudaMallocAsync(&w->mem, bytes, st);
        if (e != cudaSuccess) {
            w->mem = nullptr;
            if (e != cudaErrorMemoryAllocation) return e;
            cudaGetLastError();
            return cudaSuccess;
        }
    }
    return ksc::start_conv_scratch(s, maps, n_maps, use, w->mem, w, st);
}

// The slots of a split with tensor-core stages (without room for them its calls allocate).
void make_slots(ksc_split *s) {
    s->slot_bytes = ksc::conv_scratch_bytes(s, 1, ksc::conv_use(s, 0, s->plan.nrings - 1, true, true));
    if (s->slot_bytes == 0) return;
    for (ksc_split::ScratchSlot &c : s->slots) {
        if (cudaEventCreateWithFlags(&c.done, cudaEventDisableTiming) != cudaSuccess ||
            dev_malloc(&c.mem, s->slot_bytes) != cudaSuccess) {
            cudaGetLastError();
            c.mem = nullptr;
        }
    }
}

// Tensor-core belt stage for a stack of maps; grows the split's pre-tiled map
// workspace on first use (calls on one split must not overlap on the GPU).
int launch_belt_tensor(const ksc_split *cs, const float *d_in, float *d_out, int n_maps,
                       long long stride, cudaStream_t st) {
    ksc_split *s = const_cast<ksc_split *>(cs);
    const int n_belt = s->plan.belt_hi - s->plan.belt_lo + 1;
    const size_t need = ksc::belt_mma_workspace_floats(n_belt, s->mma_ntiles, n_maps);
    if (s->ws_floats < need) {
        cudaFree(s->d_ws);
        s->d_ws = nullptr;
        s->ws_floats = 0;
        if (cudaMalloc(&s->d_ws, need * sizeof(float)) != cudaSuccess)
            return fail(KSC_ERR_NOMEM, "tensor-path workspace");
        s->ws_floats = need;
    }
    cudaError_t e = ksc::launch_conv_belt_mma(s->plan, s->d_items_mma, s->n_items_mma, s->w_cap,
                                              s->mma_ntiles, s->mma_ext0, s->d_ws, d_in, d_out,
                                              n_maps, stride, s->d_err, st);
    if (e != cudaSuccess) return cuda_fail(e, "tensor belt kernel launch");
    return KSC_OK;
}

// The real-space convolution of output rings [r0, r1] (0-based, inclusive).
// Default path: circulant belt kernel first (writes belt outputs), then the
// symmetric gather (writes cap outputs, adds cap inputs to belt outputs).
// path 1: the general gather alone.
int launch_conv(const ksc_split *s, const float *d_in, float *d_out, int n_maps,
                long long stride, int r0, int r1, cudaStream_t st) {
    ksc::NvtxRange range(n_maps > 1 ? "ksc_conv_real_multimap" : "ksc_conv_real");
    cudaError_t e;
    if (s->path == 1) {
        const int c = s->ring_first_item[r0], d = s->ring_first_item[r1 + 1];
        e = ksc::launch_conv_general(s->plan, s->d_items + c, d - c, d_in, d_out, n_maps,
                                     stride, 0, nullptr, st);
        if (e != cudaSuccess) return cuda_fail(e, "gather kernel launch");
        return KSC_OK;
    }
    const ksc::MapSet maps{d_in, d_out, stride};
    const bool whole = r0 == 0 && r1 == s->plan.nrings - 1;
    const bool stack = whole && n_maps >= 16;
    const bool belt_mma = stack && s->tensor == 2 && s->n_items_mma > 0;
    CallScratch w;
    e = start_scratch(s, maps, n_maps,
                      ksc::conv_use(s, r0, r1, !belt_mma, !(stack && s->tensor >= 1)), st, &w);
    if (e != cudaSuccess) return cuda_fail(e, "call scratch");
    if (belt_mma) {
        int rc = launch_belt_tensor(s, d_in, d_out, n_maps, stride, st);
        if (rc) return rc;
    } else {
        e = ksc::launch_belt(s, maps, n_maps, r0, r1, w, s->d_err, st);
        if (e != cudaSuccess) return cuda_fail(e, "belt kernel launch");
    }
    // northern rings r whose own or mirror ring (nr - 1 - r) lies in the band
    const int nr = s->plan.nrings, eq = (nr - 1) / 2;
    int lo = nr, hi = -1;
    if (r0 <= eq) { lo = r0; hi = std::min(r1, eq); }                // own ring in band
    const int m0 = std::max(0, nr - 1 - r1), m1 = std::min(nr - 1 - r0, eq);
    if (m0 <= m1) { lo = std::min(lo, m0); hi = std::max(hi, m1); }  // mirror in band
    if (lo <= hi) {
        e = ksc::launch_caps(s, maps, n_maps, lo, hi, r0, r1, stack, w, s->d_err, st);
        if (e != cudaSuccess) return cuda_fail(e, "symmetric kernel launch");
    }
    return KSC_OK;
}

} // namespace

namespace ksc {

bool has_cap_tc(const ksc_split *s) { return s->ctc.ring_end >= s->ctc.ring_first; }

ConvUse conv_use(const ksc_split *s, int r0, int r1, bool want_belt, bool want_cap) {
    ConvUse u;
    const int nr = s->plan.nrings, nside = s->nside, eq = (nr - 1) / 2;
    const int belt_lo = s->plan.belt_lo, belt_hi = s->plan.belt_hi;
    u.belt = want_belt && s->btc.n_cols > 0 && r0 <= belt_hi && r1 >= belt_lo;
    // northern rings of the band and its mirror, with the other ring of a cap tile
    const int lo = std::max(std::min(r0, nr - 1 - r1) - 1, 0);
    const int hi = std::min((r1 <= eq ? r1 : r0 >= eq ? nr - 1 - r0 : eq) + 1, eq);
    u.cap = want_cap && has_cap_tc(s) && lo <= s->ctc.ring_end;
    if (!u.belt && !u.cap) return u;
    InputReach &in = u.in;
    if (u.cap) {
        in.q0 = s->range[lo].x;
        in.q1 = s->range[hi].y;
        in.q2 = nr - 1 - in.q1;
        in.q3 = nr - 1 - in.q0;
    }
    if (u.belt) {  // whole blocks of rings
        const int nb = belt_tc_rings();
        const int a = belt_lo + (std::max(r0, belt_lo) - belt_lo) / nb * nb;
        const int b = std::min(belt_hi, belt_lo + (std::min(r1, belt_hi) - belt_lo) / nb * nb + nb - 1);
        const int q0 = std::max(s->range[a].x, belt_lo), q1 = std::min(s->range[b].y, belt_hi);
        if (!u.cap) {
            in.q0 = q0;
            in.q1 = q1;
        } else if (q0 + q1 <= nr - 1) {
            in.q0 = std::min(in.q0, q0);
            in.q1 = std::max(in.q1, q1);
        } else {
            in.q2 = std::min(in.q2, q0);
            in.q3 = std::max(in.q3, q1);
        }
    }
    if (in.q2 <= in.q1 + 1 && in.q3 >= in.q2) {  // one interval
        in.q0 = std::min(in.q0, in.q2);
        in.q1 = std::max(in.q1, in.q3);
        in.q2 = 0;
        in.q3 = -1;
    }
    const auto start = [&](int r) -> long long {  // first pixel of a ring
        const long long i = r + 1, n = nside, j = 4 * n - i;
        return i <= n ? 2 * i * (i - 1)
                      : i <= 3 * n ? 2 * n * (n - 1) + 4 * n * (i - n) : 12 * n * n - 2 * j * (j + 1);
    };
    const auto blocks = [&](int qa, int qb, int *b, int *n) {
        *b = (int)(start(qa) >> 6);
        *n = qb < qa ? 0 : (int)((start(qb + 1) - 1) >> 6) + 1 - *b;
    };
    blocks(in.q0, in.q1, &in.b0, &in.n0);
    blocks(in.q2, in.q3, &in.b1, &in.n1);
    return u;
}

size_t conv_scratch_bytes(const ksc_split *s, int n_maps, const ConvUse &use) {
    const size_t nr = (size_t)s->plan.nrings;
    if (!use.cap && !use.belt) return 0;
    size_t b = sizeof(int);  // the gather's claim counter
    b += sizeof(unsigned) * (size_t)map_blocks(s->plan);
    if (use.cap) b += sizeof(uint2) * nr + sizeof(int) * (nr + 1);
    if (use.belt) b += (size_t)belt_tc_tiles(s->plan, s->btc);
    return b * (size_t)n_maps;
}

cudaError_t start_conv_scratch(const ksc_split *s, const MapSet &maps, int n_maps,
                               const ConvUse &use, void *mem, ConvScratch *w, cudaStream_t st) {
    const bool cap = use.cap, belt = use.belt;
    if (!cap && !belt) return cudaSuccess;
    const size_t nr = (size_t)s->plan.nrings, n = (size_t)n_maps;
    unsigned char *at = static_cast<unsigned char *>(mem);
    const auto take = [&](size_t bytes) {
        unsigned char *p = at;
        at += bytes * n;
        return p;
    };
    if (cap) w->ranges = reinterpret_cast<uint2 *>(take(sizeof(uint2) * nr));
    w->counters = reinterpret_cast<int *>(take(sizeof(int)));
    if (cap) w->cap_flags = reinterpret_cast<int *>(take(sizeof(int) * (nr + 1)));
    unsigned char *const zero_end = at;
    w->bm = reinterpret_cast<unsigned *>(take(sizeof(unsigned) * (size_t)map_blocks(s->plan)));
    if (belt) w->belt_flags = at;
    const size_t n_zero = (size_t)(zero_end - (unsigned char *)w->counters);
    cudaError_t e = launch_block_max(s->plan, maps, n_maps, use.in, w->bm, w->counters,
                                     (long long)(n_zero / sizeof(int)), st);
    if (e == cudaSuccess && cap)
        e = launch_ring_range(s->plan, w->bm, n_maps, use.in, w->ranges, st);
    return e;
}

// The belt stage (belt-belt ring pairs) of output rings [r0, r1]: the tensor-core kernel
// where the split has a plan for it, then the FFMA kernel for the tiles it left (none of
// them in an ordinary map: that launch reads the flags and ends); else the FFMA kernel.
cudaError_t launch_belt(const ksc_split *s, const MapSet &maps, int n_maps, int r0, int r1,
                        const ConvScratch &w, int *d_err, cudaStream_t st) {
    const int a = s->ring_first_belt[r0], b = s->ring_first_belt[r1 + 1];
    if (a == b || s->n_items_belt == 0) return cudaSuccess;
    if (!w.belt_flags)
        return launch_conv_belt(s->plan, s->d_items_belt + a, b - a, s->seg_cap, maps, n_maps,
                                nullptr, nullptr, d_err, st);
    const cudaError_t e = launch_conv_belt_tc(s->plan, s->btc, maps, n_maps, r0, r1, w.bm,
                                              w.belt_flags, d_err, st);
    if (e != cudaSuccess) return e;
    return launch_conv_belt(s->plan, s->d_items_belt + a, b - a, s->seg_cap, maps, n_maps,
                            &s->btc, w.belt_flags, d_err, st);
}

// The cap stage for the items of northern rings [lo, hi], writing output rings
// [r0, r1]: the map-stack tensor kernel for whole-map stacks, else the FFMA gather
// or the single-map tensor kernel (ksc_split_opts.cap_kernel).  Whole maps take
// the items longest first, bands their rings' items in ring order.
cudaError_t launch_caps(const ksc_split *s, const MapSet &maps, int n_maps, int lo, int hi,
                        int r0, int r1, bool stack, const ConvScratch &w, int *d_err,
                        cudaStream_t st) {
    const bool whole = r0 == 0 && r1 == s->plan.nrings - 1;
    const int belt_split = s->n_items_belt > 0 ? 1 : 0;
    if (stack && s->tensor >= 1)
        return launch_conv_sym_mma(s->plan, s->d_items_smma_lpt, s->n_items_smma, maps.in,
                                        maps.out, n_maps, maps.stride, belt_split, d_err, st);
    if (s->cap_kernel == 1) {
        const int c = s->ring_first_smma[lo], d = s->ring_first_smma[hi + 1];
        const WorkItem *its = whole ? s->d_items_smma_lpt : s->d_items_smma + c;
        return launch_conv_sym_tc(s->plan, its, d - c, maps.in, maps.out, n_maps, maps.stride,
                                       belt_split, r0, r1, d_err, st);
    }
    const int c = s->ring_first_sym[lo], d = s->ring_first_sym[hi + 1];
    const WorkItem *its = whole ? s->d_items_sym_lpt : s->d_items_sym + c;
    if (!w.cap_flags)
        return launch_conv_sym(s->plan, its, d - c, s->sym_variant, maps, n_maps, belt_split, r0, r1, d - c,
                                    nullptr, w.counters, d_err, st);
    // the tensor-core stage, the irregular ring pairs, then the gather for the rings that
    // the first flagged (none in an ordinary map: that launch reads a flag and ends)
    // (a tile holds rings r and r + 1: from the one that may start just before lo)
    const int t0 = whole ? 0 : s->cap_tile_first[std::max(lo - 1, 0)];
    const int t1 = whole ? s->n_cap_tiles : s->cap_tile_first[hi + 1];
    // a band's tiles in ring order, from the end that takes longer
    const bool back = !whole && t1 > t0 && s->cap_tile_us[t1 - 1] > s->cap_tile_us[t0];
    cudaError_t e = launch_conv_cap_tc(
        s->plan, s->ctc, whole ? s->d_cap_tiles_lpt : s->d_cap_tiles + t0, t1 - t0, maps,
        n_maps, belt_split, r0, r1, w.ranges, w.cap_flags, back, d_err, st);
    if (e != cudaSuccess) return e;
    const int i0 = s->irr_item_first[lo], i1 = s->irr_item_first[hi + 1];
    e = launch_cap_direct(s->plan, s->d_irr_items + i0, i1 - i0, s->d_irr_first, s->d_irr,
                               maps, n_maps, r0, r1, w.cap_flags, st);
    if (e != cudaSuccess) return e;
    return launch_conv_sym(s->plan, its, d - c, s->sym_variant, maps, n_maps, belt_split, r0, r1, 0,
                                w.cap_flags, w.counters, d_err, st);
}

void set_last_error(const std::string &msg) { g_last_error = msg; }

bool inject_alloc_fault(int n) {
    const char *f = std::getenv("KSC_FAULT");
    if (!f || std::strncmp(f, "alloc:", 6) != 0) return false;
    return n == std::atoi(f + 6);
}

XInfo make_xinfo(double A2, double B2, double c, double nint2, float hw, int L, int lq,
                 double scale) {
    XInfo x{};
    // no pair within the cut, or a whole-ring window: no table
    if (hw < 0.0f || 2.0f * hw + 3.0f >= (float)lq || A2 >= nint2 || B2 <= 0.0) return x;
    const double sx2 = (nint2 - A2) / B2;  // sin^2 of x at the cut
    if (sx2 >= 1.0) return x;
    const double xcut = std::asin(std::sqrt(sx2));
    // largest du/dx on [0, xcut]: u^2 = A2 + B2 S, S = sin^2 x, du/dx = B2 sqrt(g(S)) with
    // g = S (1 - S) / (A2 + B2 S), unimodal in S with its peak where B2 S^2 + 2 A2 S = A2
    double dmax;
    if (A2 <= 0.0) {
        dmax = std::sqrt(B2);  // u = sqrt(B2) sin x
    } else {
        double S = (-A2 + std::sqrt(A2 * A2 + A2 * B2)) / B2;
        S = std::min(std::max(S, 0.0), sx2);
        dmax = B2 * std::sqrt(S * (1.0 - S) / (A2 + B2 * S));
    }
    if (!(dmax > 0.0)) return x;
    // the largest |N| within the cut: |N| c <= xcut
    const double nc = std::floor(xcut / c);
    if (nc >= 8388608.0) return x;  // |N| and the quads' reach stay below 2^24
    const int ncut = (int)nc;
    // widest power-of-two cell within kXRho intervals at the steepest point, and no
    // wider than the in-cut range (so that no node lies more than one cell beyond the
    // cut, where the K_r table is extrapolated) ...
    int shift = (int)std::floor(std::log2(scale * kXRho / (dmax * c)));
    shift = std::max(shift, 0);
    while (shift > 0 && std::ldexp(c, shift) * dmax > scale * kXRho) --shift;  // log2 rounding
    while (shift > 0 && (1 << std::min(shift, 30)) > ncut + 1) --shift;
    // ... doubled while the cells (and the reach of an edge quad) would not fit
    auto cells = [&](int sh) { return (ncut >> sh) + 1; };
    while (cells(shift) + kXPad(L, shift) > kXCap && shift < 22) ++shift;
    if (cells(shift) + kXPad(L, shift) > kXCap) return x;
    if (std::ldexp(c, shift) * dmax > scale * kXRhoMax * (1.0 + 1e-12) && shift > 0) return x;
    // integers of in-cut pairs and of positions up to 16 beyond them stay exact in FP32
    if ((double)ncut + 32.0 * (double)L + std::ldexp(1.0, shift) >= 16777216.0) return x;
    x.shift = shift;
    x.ncut = ncut;
    x.ncell = cells(shift);
    return x;
}

XOdd make_xodd(double A2, double B2, double c, double nint2, float hw, int L, int lq,
               double scale, int cap) {
    XOdd x{};
    if (hw < 0.0f || 2.0f * hw + 3.0f >= (float)lq || A2 >= nint2 || B2 <= 0.0) return x;
    const double sx2 = (nint2 - A2) / B2;  // sin^2 of x at the cut
    if (sx2 >= 1.0) return x;
    const double xcut = std::asin(std::sqrt(sx2));
    // largest du/dx on [0, xcut] (as for the power-of-two tables)
    double dmax;
    if (A2 <= 0.0) {
        dmax = std::sqrt(B2);
    } else {
        double S = (-A2 + std::sqrt(A2 * A2 + A2 * B2)) / B2;
        S = std::min(std::max(S, 0.0), sx2);
        dmax = B2 * std::sqrt(S * (1.0 - S) / (A2 + B2 * S));
    }
    if (!(dmax > 0.0)) return x;
    const double nc = std::floor(xcut / c);
    if (nc >= 8388608.0) return x;
    const long long ncut = (long long)nc;
    const long long D = 2LL * lq;
    // widest cell within kXOddRho intervals where the chord changes fastest and no
    // wider than the in-cut range; m the least odd integer giving a cell that narrow
    const double hmax = std::min(scale * kXOddRho / (dmax * c), (double)ncut + 1.0);
    long long m = (long long)std::ceil((double)D / hmax - 1e-9);
    if (m < 1) m = 1;
    if ((m & 1) == 0) ++m;
    auto cells = [&](long long mm) { return (ncut * mm) / D + 1; };  // the zero cell's index
    // wider cells (smaller odd m) while the table and its zero cell would not fit
    while (cells(m) + 1 > cap && m > 1) m -= 2;
    if (cells(m) + 1 > cap) return x;
    const double width = (double)D / (double)m;  // in |N|
    if (width * c * dmax > scale * kXRhoMax * (1.0 + 1e-12)) return x;
    // integers a quarter warp's walk reaches (see XOdd) stay exact
    const double reach = (double)ncut + 48.0 * (double)lq + 40.0 * (double)L;
    if (reach >= 16777216.0 || reach * (double)m + (double)D >= 2147483647.0) return x;
    x.m = (int)m;
    x.nct = (int)cells(m);
    x.off = (int)((long long)x.nct * D - ncut * m - 1);
    x.ncut = (int)ncut;
    const DF cm = df_from_double(c / (double)m);
    x.cmh = cm.h;
    x.cml = cm.l;
    x.hc = (float)(c * width);
    return x;
}
} // namespace ksc

extern "C" {

int ksc_default_opts(ksc_split_opts *opts) {
    if (!opts) return fail(KSC_ERR_ARG, "null opts");
    opts->mode = KSC_SPLIT_LSQ;
    opts->oversample = 2;
    opts->svd_rcond = 1e-6;
    opts->alpha = 5.0;
    opts->n_intervals = 0;
    opts->path = 0;
    opts->tensor = 0;
    opts->cut_continuity = KSC_CUT_C1;
    opts->exact_weights = 0;
    opts->cap_kernel = 0;
    return KSC_OK;
}

int ksc_make_split(const double *b_l, int lmax, int nside, int l_cut, double theta_cut,
                   const double *cl_in, const ksc_split_opts *opts, ksc_split **out) {
    ksc::NvtxRange range("ksc_make_split");
    if (!out) return fail(KSC_ERR_ARG, "null output pointer");
    *out = nullptr;
    if (!b_l) return fail(KSC_ERR_ARG, "null kernel");
    int rc = check_common(lmax, nside, theta_cut);
    if (rc) return rc;
    ksc_split_opts o = resolve_opts(opts);
    if (o.mode != KSC_SPLIT_NONE && (l_cut < 0 || l_cut >= lmax))
        return fail(KSC_ERR_ARG, "l_cut outside 0..lmax-1");
    if (o.mode < KSC_SPLIT_LSQ || o.mode > KSC_SPLIT_NONE) return fail(KSC_ERR_ARG, "bad mode");

    ksc_split *s = new (std::nothrow) ksc_split();
    if (!s) return fail(KSC_ERR_NOMEM, "host allocation");
    s->lmax = lmax; s->nside = nside; s->theta_cut = theta_cut; s->mode = o.mode;
    const int L = lmax + 1;
    try {
        if (o.mode == KSC_SPLIT_LSQ) {
            ksc::FitResult fr;
            std::string msg;
            const int n_con = o.cut_continuity == KSC_CUT_FREE ? 0
                              : (o.cut_continuity == KSC_CUT_C0 ? 1 : 2);
            rc = ksc::fit_split_lsq(b_l, lmax, l_cut, theta_cut, cl_in, o.oversample,
                                    o.svd_rcond, n_con, &fr, &msg);
            if (rc) { release(s); return fail(rc, msg); }
            s->l_cut = l_cut;
            s->k_harm = fr.k_harm; s->c_real = fr.c_real; s->k_tilde = fr.k_tilde;
            s->n_unknowns = fr.n_unknowns; s->n_kept = fr.n_kept;
        } else if (o.mode == KSC_SPLIT_SHARP) {
            s->l_cut = l_cut;
            s->k_harm.assign(b_l, b_l + l_cut + 1);
            s->c_real.assign(b_l, b_l + L);
            std::fill(s->c_real.begin(), s->c_real.begin() + l_cut + 1, 0.0);
            s->k_tilde.assign(b_l, b_l + L);  // exact before truncation
        } else {
            s->l_cut = -1;
            s->c_real.assign(b_l, b_l + L);
            s->k_tilde.assign(b_l, b_l + L);
        }
    } catch (const std::bad_alloc &) {
        release(s);
        return fail(KSC_ERR_NOMEM, "host allocation in split fit");
    }
    s->sigma_rms = ksc::sigma_rms_eq2(b_l, s->k_tilde.data(), cl_in, lmax);
    s->frac_error = ksc::frac_error_eq6(b_l, s->k_tilde.data(), cl_in, lmax, o.alpha);
    rc = finish_split(s, o);
    if (rc) { release(s); return rc; }
    *out = s;
    return KSC_OK;
}

int ksc_make_split_real(const double *c_l, int lmax, int nside, double theta_cut,
                        const ksc_split_opts *opts, ksc_split **out) {
    ksc::NvtxRange range("ksc_make_split_real");
    if (!out) return fail(KSC_ERR_ARG, "null output pointer");
    *out = nullptr;
    if (!c_l) return fail(KSC_ERR_ARG, "null coefficients");
    int rc = check_common(lmax, nside, theta_cut);
    if (rc) return rc;
    ksc_split_opts o = resolve_opts(opts);
    ksc_split *s = new (std::nothrow) ksc_split();
    if (!s) return fail(KSC_ERR_NOMEM, "host allocation");
    s->lmax = lmax; s->nside = nside; s->theta_cut = theta_cut; s->mode = KSC_SPLIT_NONE;
    s->l_cut = -1;
    s->c_real.assign(c_l, c_l + lmax + 1);
    s->k_tilde = s->c_real;
    rc = finish_split(s, o);
    if (rc) { release(s); return rc; }
    *out = s;
    return KSC_OK;
}

int ksc_dphi_table_params(double A2, double B2, double c, int n_int, double hw, int lq,
                          double scale, double *out) {
    if (!out || !(c > 0.0) || n_int < 1) return fail(KSC_ERR_ARG, "bad table parameters");
    // the output ring's length from c = pi / (2 L lq)
    const int L = lq > 0 ? (int)std::lround(kPi / (2.0 * c * (double)lq)) : 1;
    const ksc::XInfo x = ksc::make_xinfo(A2, B2, c, (double)n_int * (double)n_int, (float)hw,
                                         std::max(L, 1), lq, scale);
    out[0] = x.ncell > 0 ? std::ldexp(c, x.shift) : 0.0;
    out[1] = (double)x.ncell;
    out[2] = x.ncell > 0 ? (double)x.ncut : 0.0;
    return KSC_OK;
}

int ksc_dphi_odd_params(double A2, double B2, double c, int n_int, double hw, int lq,
                        double scale, int cap, double *out) {
    if (!out || !(c > 0.0) || n_int < 1 || lq < 1 || cap < 2)
        return fail(KSC_ERR_ARG, "bad table parameters");
    const int L = (int)std::lround(kPi / (2.0 * c * (double)lq));
    const ksc::XOdd x = ksc::make_xodd(A2, B2, c, (double)n_int * (double)n_int, (float)hw,
                                       std::max(L, 1), lq, scale, cap);
    out[0] = x.nct > 0 ? c * 2.0 * (double)lq / (double)x.m : 0.0;
    out[1] = (double)x.m;
    out[2] = (double)x.off;
    out[3] = (double)x.nct;
    out[4] = x.nct > 0 ? (double)x.ncut : 0.0;
    return KSC_OK;
}

int ksc_split_info(const ksc_split *s, ksc_split_desc *d) {
    if (!s || !d) return fail(KSC_ERR_ARG, "null argument");
    d->lmax = s->lmax; d->l_cut = s->l_cut; d->nside = s->nside; d->mode = s->mode;
    d->n_intervals = s->n_int; d->n_unknowns = s->n_unknowns; d->n_kept = s->n_kept;
    d->theta_cut = s->theta_cut; d->chord_cut = s->chord_cut;
    d->sigma_rms = s->sigma_rms; d->frac_error = s->frac_error; d->n_pairs = s->n_pairs;
    d->n_pairs_belt = s->n_pairs_belt; d->path = s->path;
    d->frac_tabulated = s->frac_tabulated;
    return KSC_OK;
}

int ksc_split_stages(const ksc_split *s, ksc_stage_desc *d) {
    if (!s || !d) return fail(KSC_ERR_ARG, "null argument");
    *d = ksc_stage_desc{};
    d->gather_variant = s->sym_variant;
    d->n_launches = 1;
    if (s->path == 1) return KSC_OK;
    const bool cap = ksc::has_cap_tc(s), belt = s->btc.n_cols > 0;
    d->belt_columns = s->btc.n_cols;
    d->cap_stage = cap;
    // block maxima, ring ranges; the belt kernel, the stage's too; the gather, the stage's too
    d->n_launches = (cap || belt) + cap + (s->n_items_belt > 0) + belt + 1 + cap;
    if (cap && s->irr_item_first.back() > 0) ++d->n_launches;
    return KSC_OK;
}

int ksc_split_harmonic(const ksc_split *s, double *k) {
    if (!s || !k) return fail(KSC_ERR_ARG, "null argument");
    std::copy(s->k_harm.begin(), s->k_harm.end(), k);
    return KSC_OK;
}

int ksc_split_real_coeffs(const ksc_split *s, double *c) {
    if (!s || !c) return fail(KSC_ERR_ARG, "null argument");
    std::copy(s->c_real.begin(), s->c_real.end(), c);
    return KSC_OK;
}

int ksc_split_model(const ksc_split *s, double *k) {
    if (!s || !k) return fail(KSC_ERR_ARG, "null argument");
    std::copy(s->k_tilde.begin(), s->k_tilde.end(), k);
    return KSC_OK;
}

int ksc_split_table(const ksc_split *s, float *h) {
    if (!s || !h) return fail(KSC_ERR_ARG, "null argument");
    cudaError_t e = cudaMemcpy(h, s->d_tab, sizeof(float4) * s->n_int, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "table download");
    return KSC_OK;
}

int ksc_conv_real(const ksc_split *s, const float *d_in, float *d_out, void *stream) {
    int rc = check_maps(s, d_in, d_out);
    if (rc) return rc;
    return launch_conv(s, d_in, d_out, 1, 0, 0, s->plan.nrings - 1, (cudaStream_t)stream);
}

int ksc_conv_real_rings(const ksc_split *s, const float *d_in, float *d_out, int ring_lo,
                        int ring_hi, void *stream) {
    int rc = check_maps(s, d_in, d_out);
    if (rc) return rc;
    const int nr = 4 * s->nside - 1;
    if (ring_lo < 1 || ring_hi > nr || ring_lo > ring_hi)
        return fail(KSC_ERR_ARG, "ring range outside 1..4 nside - 1");
    return launch_conv(s, d_in, d_out, 1, 0, ring_lo - 1, ring_hi - 1, (cudaStream_t)stream);
}

int ksc_conv_real_multimap(const ksc_split *s, const float *d_in, float *d_out, int n_maps,
                           void *stream) {
    int rc = check_maps(s, d_in, d_out);
    if (rc) return rc;
    if (n_maps < 1 || n_maps > 65535) return fail(KSC_ERR_ARG, "n_maps outside 1..65535");
    return launch_conv(s, d_in, d_out, n_maps, s->plan.npix, 0, s->plan.nrings - 1,
                       (cudaStream_t)stream);
}

int ksc_conv_real_batch(const ksc_split *const *splits, const float *const *d_in,
                        float *const *d_out, int n, void *stream) {
    if (n < 0 || (n > 0 && (!splits || !d_in || !d_out)))
        return fail(KSC_ERR_ARG, "bad batch arrays");
    if (n == 0) return KSC_OK;
    for (int i = 0; i < n; ++i) {
        int rc = check_maps(splits[i], d_in[i], d_out[i]);
        if (rc) return rc;
    }
    ksc_batch_opts o;
    ksc_batch_default_opts(&o);
    o.use_graph = 0;
    ksc_batch *b = nullptr;
    int rc = ksc_batch_create(splits, n, &o, &b);
    if (rc) return rc;
    rc = ksc_batch_run(b, d_in, d_out, stream);
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
    ksc_batch_free(b);
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "batch synchronize");
    return KSC_OK;
}

int ksc_conv_real_host(const ksc_split *cs, const float *h_in, float *h_out) {
    ksc::NvtxRange range("ksc_conv_real_host");
    if (!cs || !h_in || !h_out) return fail(KSC_ERR_ARG, "null argument");
    ksc_split *s = const_cast<ksc_split *>(cs);
    // the split's host-path stream and buffers serve one call at a time
    std::lock_guard<std::mutex> lk(s->host_mu);
    cudaError_t e;
    const size_t bytes = sizeof(float) * (size_t)s->plan.npix;
    if (!s->d_io) {
        g_alloc_count = 0;
        if ((e = dev_malloc((void **)&s->d_io, 2 * bytes)) != cudaSuccess) {
            s->d_io = nullptr;
            return fail(KSC_ERR_NOMEM, "device buffers for the host path");
        }
    }
    if (!s->own_stream) {
        if ((e = cudaStreamCreateWithFlags(&s->own_stream, cudaStreamNonBlocking)) != cudaSuccess)
            return cuda_fail(e, "stream create");
    }
    float *din = s->d_io, *dout = s->d_io + s->plan.npix;
    if ((e = cudaMemcpyAsync(din, h_in, bytes, cudaMemcpyHostToDevice, s->own_stream)) != cudaSuccess)
        return cuda_fail(e, "host to device copy");
    int rc = launch_conv(s, din, dout, 1, 0, 0, s->plan.nrings - 1, s->own_stream);
    if (rc) return rc;
    if ((e = cudaMemcpyAsync(h_out, dout, bytes, cudaMemcpyDeviceToHost, s->own_stream)) != cudaSuccess)
        return cuda_fail(e, "device to host copy");
    if ((e = cudaStreamSynchronize(s->own_stream)) != cudaSuccess)
        return cuda_fail(e, "host path synchronize");
    return ksc_device_status(s, s->own_stream);
}

int ksc_device_status(const ksc_split *s, void *stream) {
    if (!s) return fail(KSC_ERR_ARG, "null split");
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "stream synchronize");
    int flag = 0;
    if ((e = cudaMemcpyAsync(&flag, s->d_err, sizeof(int), cudaMemcpyDeviceToHost,
                             (cudaStream_t)stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize((cudaStream_t)stream)) != cudaSuccess)
        return cuda_fail(e, "error flag read");
    if (flag != 0) {
        // cleared in order on the caller's stream (the flag is shared by every
        // stream that uses the split: clear it where no call on this split runs)
        if ((e = cudaMemsetAsync(s->d_err, 0, sizeof(int), (cudaStream_t)stream)) != cudaSuccess ||
            (e = cudaStreamSynchronize((cudaStream_t)stream)) != cudaSuccess)
            return cuda_fail(e, "error flag clear");
        return fail(flag, "a device-side check fired during an earlier call");
    }
    return KSC_OK;
}

int ksc_probe_wait_timeout(const ksc_split *s, int max_polls, void *stream) {
    if (!s) return fail(KSC_ERR_ARG, "null split");
    if (max_polls <= 0 || max_polls > ksc::tc::kMaxWait) max_polls = ksc::tc::kMaxWait;
    wait_probe_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(s->d_err, max_polls);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "wait probe launch");
    return KSC_OK;
}

int ksc_count_pairs(ksc_split *s, long long *n_pairs) {
    if (!s || !n_pairs) return fail(KSC_ERR_ARG, "null argument");
    unsigned long long *d_cnt = nullptr;
    cudaError_t e = cudaMalloc(&d_cnt, 2 * sizeof(unsigned long long));
    if (e != cudaSuccess) return cuda_fail(e, "count buffer");
    cudaMemset(d_cnt, 0, 2 * sizeof(unsigned long long));
    e = ksc::launch_conv_general(s->plan, s->d_items, s->n_items, nullptr, nullptr, 1, 0, 0,
                                 d_cnt, 0);
    if (e == cudaSuccess)
        e = ksc::launch_conv_general(s->plan, s->d_items, s->n_items, nullptr, nullptr, 1, 0, 1,
                                     d_cnt + 1, 0);
    unsigned long long h[2] = {0, 0};
    if (e == cudaSuccess) e = cudaMemcpy(h, d_cnt, sizeof(h), cudaMemcpyDeviceToHost);
    cudaFree(d_cnt);
    if (e != cudaSuccess) return cuda_fail(e, "pair count");
    s->n_pairs = (long long)h[0];
    s->n_pairs_belt = (long long)h[1];
    *n_pairs = s->n_pairs;
    return KSC_OK;
}

int ksc_conv_real_multimap_stage(const ksc_split *s, const float *d_in, float *d_out,
                                 int n_maps, int stage, void *stream) {
    int rc = check_maps(s, d_in, d_out);
    if (rc) return rc;
    if (n_maps < 1 || n_maps > 65535) return fail(KSC_ERR_ARG, "n_maps outside 1..65535");
    cudaStream_t st = (cudaStream_t)stream;
    const long long stride = s->plan.npix;
    if (stage != 1 && stage != 2) return fail(KSC_ERR_ARG, "stage must be 1 or 2");
    const ksc::MapSet maps{d_in, d_out, stride};
    CallScratch w;
    const bool belt_mma = n_maps >= 16 && s->tensor == 2 && s->n_items_mma > 0;
    cudaError_t e = cudaSuccess;
    if (s->path != 1)
        e = start_scratch(s, maps, n_maps,
                          ksc::conv_use(s, 0, s->plan.nrings - 1, stage == 1 && !belt_mma,
                                        stage == 2 && !(n_maps >= 16 && s->tensor >= 1)), st, &w);
    if (e != cudaSuccess) return cuda_fail(e, "call scratch");
    if (stage == 1) {
        if (s->path == 1) return KSC_OK;
        if (belt_mma)
            return launch_belt_tensor(s, d_in, d_out, n_maps, stride, st);
        else
            e = ksc::launch_belt(s, maps, n_maps, 0, s->plan.nrings - 1, w, s->d_err, st);
    } else {
        if (s->path == 1)
            e = ksc::launch_conv_general(s->plan, s->d_items, s->n_items, d_in, d_out, n_maps,
                                         stride, 0, nullptr, st);
        else
            e = ksc::launch_caps(s, maps, n_maps, 0, (s->plan.nrings - 1) / 2, 0,
                                 s->plan.nrings - 1, n_maps >= 16, w, s->d_err, st);
    }
    if (e != cudaSuccess) return cuda_fail(e, "stage launch");
    return KSC_OK;
}

int ksc_conv_real_stage(const ksc_split *s, const float *d_in, float *d_out, int stage,
                        void *stream) {
    int rc = check_maps(s, d_in, d_out);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    if (stage != 1 && stage != 2) return fail(KSC_ERR_ARG, "stage must be 1 or 2");
    const ksc::MapSet maps{d_in, d_out, 0};
    CallScratch w;
    cudaError_t e = cudaSuccess;
    if (s->path != 1)
        e = start_scratch(s, maps, 1,
                          ksc::conv_use(s, 0, s->plan.nrings - 1, stage == 1, stage == 2), st, &w);
    if (e != cudaSuccess) return cuda_fail(e, "call scratch");
    if (stage == 1) {
        e = ksc::launch_belt(s, maps, 1, 0, s->plan.nrings - 1, w, s->d_err, st);
    } else {
        if (s->path == 1)
            e = ksc::launch_conv_general(s->plan, s->d_items, s->n_items, d_in, d_out, 1, 0, 0,
                                         nullptr, st);
        else
            e = ksc::launch_caps(s, maps, 1, 0, (s->plan.nrings - 1) / 2, 0, s->plan.nrings - 1,
                                 false, w, s->d_err, st);
    }
    if (e != cudaSuccess) return cuda_fail(e, "stage launch");
    return KSC_OK;
}

void ksc_free_split(ksc_split *s) { release(s); }

const char *ksc_status_string(int st) {
    switch (st) {
    case KSC_OK: return "KSC_OK";
    case KSC_ERR_ARG: return "KSC_ERR_ARG";
    case KSC_ERR_NOMEM: return "KSC_ERR_NOMEM";
    case KSC_ERR_CUDA: return "KSC_ERR_CUDA";
    case KSC_ERR_TIMEOUT: return "KSC_ERR_TIMEOUT";
    case KSC_ERR_DEVICE_BOUNDS: return "KSC_ERR_DEVICE_BOUNDS";
    case KSC_ERR_SVD: return "KSC_ERR_SVD";
    case KSC_ERR_UNSUPPORTED: return "KSC_ERR_UNSUPPORTED";
    case KSC_ERR_TIMEOUT_UNDRAINED: return "KSC_ERR_TIMEOUT_UNDRAINED";
    default: return "KSC_ERR_UNKNOWN";
    }
}

const char *ksc_last_error(void) { return g_last_error.c_str(); }

} // extern "C"
