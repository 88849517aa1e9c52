// pz_line.cu -- windowed Voigt line-opacity sum (Eqs. 4-5) and its adjoint
// (Sec. 6), FP32-mixed and plain FP64 forms, plus the per-device Voigt tables.
//
// Mixed-precision kernels.  A windowed sum is shared by three families, which own
// every (line, point, layer) exactly once between them:
//   box expansions (pz_box.cuh)  pairs of boxes of B points at least n_c boxes apart, inside
//                                the window of every line of the source box;
//   far wings (pz_far.cuh)       the nearer boxes down to the core: series in 1/v^2;
//   near cores (below)           the points of the core, the full Voigt function.
//
// The far-wing work is a queue of items (star, lambda tile, depth group, line
// range) built on the host: lines are sorted by centre within each star, and an
// item's range [lo, hi) holds the star's lines whose window |i - i_l| <= W
// touches the tile (with boxes: whose box is near the tile; the lines further
// out that the expansions leave are gathered from one bit per line).  The
// kernels are persistent: every CTA takes the next item from an atomic counter
// until the queue is empty, and the items are ordered longest first, so stars
// and tiles of very different line counts share one launch.  An item covers a
// tile of T = 32 J grid points and GW x DS layers; warp w sweeps layers
// [d0 + w DS, d0 + (w+1) DS) and lane l owns the J contiguous points
// t0 + l J + [0, J).  Each warp stages LC lines at a time in its own part of
// shared memory (the prefactors of Eqs. 4-5 and the series coefficients, formed
// by all lanes), then every thread accumulates its J x DS (lambda, depth) sums
// in registers.  How a line is summed over the tile and slab (far_form) is
// decided once per line and warp.  Per-chunk FP32 partial sums are folded into a
// compensated (hi, lo) pair (2Sum).  The frequency offset is formed in index
// space: v = expm1((x_l - i) ln r) c/dv_D with x_l - i = (i_l - i) + frac_l, the
// integer part exact, avoiding the cancellation of lambda_l/lambda_i - 1.
#include <cuda_runtime.h>

#include <atomic>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>
#include <vector>

#include "pz_internal.h"
#include "pz_far.cuh"
#include "pz_voigt.cuh"
#include "pz_box.cuh"

namespace pz {

// ---------------------------------------------------------------------------
// Host construction of the tables (FP64), once per device.
// ---------------------------------------------------------------------------

// Weideman coefficients: Fourier cosine coefficients of psi(t) = (L^2 + t^2) e^{-t^2}
// under t = L tan(theta/2), L = (N/sqrt 2)^(1/2), by the midpoint rule on 8N points.
static void weideman_coeffs(int N, std::vector<double> &a, double &L) {
    L = std::sqrt(N / std::sqrt(2.0));
    int M = 4 * N;
    a.assign(N + 1, 0.0);
    for (int k = 0; k < 2 * M; ++k) {
        double th = kPI * (k - M + 0.5) / M;
        double t = L * std::tan(0.5 * th);
        double psi = (L * L + t * t) * std::exp(-t * t);
        for (int n = 0; n <= N; ++n) a[n] += psi * std::cos(n * th);
    }
    for (int n = 0; n <= N; ++n) a[n] /= 2 * M;
}

// Dawson's integral D(x) = e^{-x^2} Int_0^x e^{t^2} dt = x Int_0^1 e^{-x^2 (1 - s^2)} ds,
// composite 8-point Gauss-Legendre on 256 panels.
static double dawson_quad(double x) {
    static const double gx[8] = {-0.9602898564975363, -0.7966664774136267, -0.5255324099163290,
                                 -0.1834346424956498, 0.1834346424956498,  0.5255324099163290,
                                 0.7966664774136267,  0.9602898564975363};
    static const double gw[8] = {0.1012285362903763, 0.2223810344533745, 0.3137066458778873,
                                 0.3626837833783620, 0.3626837833783620, 0.3137066458778873,
                                 0.2223810344533745, 0.1012285362903763};
    const int P = 256;
    double sum = 0.0, h = 1.0 / P;
    for (int p = 0; p < P; ++p)
        for (int k = 0; k < 8; ++k) {
            double s = (p + 0.5 * (gx[k] + 1.0)) * h;
            sum += 0.5 * h * gw[k] * std::exp(-x * x * (1.0 - s * s));
        }
    return x * sum;
}

// Node coefficients D^(k)(x_j)/k! from D' = 1 - 2xD, D^(k+1) = -2x D^(k) - 2k D^(k-1),
// stored coefficient-major: tab[k * kDawsonNodes + j].
static void dawson_table(std::vector<float> &tab) {
    tab.assign(kDawsonNodes * (kDawsonK + 1), 0.0f);
    for (int j = 0; j < kDawsonNodes; ++j) {
        double x = (double)j / kDawsonPerUnit;
        double D[kDawsonK + 2];
        D[0] = dawson_quad(x);
        D[1] = 1.0 - 2.0 * x * D[0];
        for (int k = 1; k < kDawsonK; ++k) D[k + 1] = -2.0 * x * D[k] - 2.0 * k * D[k - 1];
        double fact = 1.0;
        for (int k = 0; k <= kDawsonK; ++k) {
            if (k > 0) fact *= k;
            tab[k * kDawsonNodes + j] = (float)(D[k] / fact);
        }
    }
}

pz_status ensure_device_tables() {
    static std::mutex mu;
    static bool host_ready = false;
    static std::vector<float> weid, daw;
    static std::vector<double> weid64;
    static float weidL;
    static double weidL64;
    static bool done[64] = {false};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_check(e, "cudaGetDevice");
    std::lock_guard<std::mutex> lk(mu);
    if (!host_ready) {
        std::vector<double> a;
        double L;
        weideman_coeffs(kWeidN, a, L);
        weid.assign(a.begin(), a.end());
        weidL = (float)L;
        weideman_coeffs(kWeidN64, weid64, weidL64);
        dawson_table(daw);
        host_ready = true;
    }
    if (dev < 0 || dev >= 64) return fail(PZ_EINVAL, "device ordinal out of range");
    if (done[dev]) return PZ_OK;
    if ((e = cudaMemcpyToSymbol(c_weid, weid.data(), sizeof(float) * (kWeidN + 1))) != cudaSuccess ||
        (e = cudaMemcpyToSymbol(c_weidL, &weidL, sizeof(float))) != cudaSuccess ||
        (e = cudaMemcpyToSymbol(c_weid64, weid64.data(), sizeof(double) * (kWeidN64 + 1))) != cudaSuccess ||
        (e = cudaMemcpyToSymbol(c_weidL64, &weidL64, sizeof(double))) != cudaSuccess ||
        (e = cudaMemcpyToSymbol(g_dawson, daw.data(), sizeof(float) * daw.size())) != cudaSuccess)
        return cuda_check(e, "upload Voigt tables");
    done[dev] = true;
    return PZ_OK;
}

// ---------------------------------------------------------------------------
// Mixed-precision kernels (far-wing device code in pz_far.cuh)
// ---------------------------------------------------------------------------

// The line record of every (depth group, line), whose amask has bit w set when
// a^2 <= kFast2A2 at every layer of slab w (DS layers) of the group, and bit 8 + w when
// the centre test rejects every layer of slab w (its warp skips the line).
// Bit 4 + w: a^2 <= kWideA2 at every layer of slab w.  Bits 16 + 3w..: the line's box separation
// class at slab w: the smallest c whose nearest distance (n_c - 1) B has |v| >= 9 a at every layer
// (thresholds of |v| >= 20 are in n_c), or kBoxClasses.  Lines of class >= 1 that keep a layer are also marked in the words of wide.
// Depth group = blockIdx.y; warp w of each half of the block takes slab w (of at most 4) of 32
// consecutive lines, one word of wide (with one thread per line over all slabs a short list
// waited on the chain of table loads: 11 -> 6 us at 5,300 lines; 50 us at 2 10^5 either way).
constexpr int kInfoLines = 64;     // lines per block
__global__ void __launch_bounds__(256, 6) k_far_info(LineArgs gq, int DC, int DS, LineInfo *info) {
    __shared__ int s_mask[4][kInfoLines];
    const int grp = blockIdx.y, w = (threadIdx.x >> 5) & 3, col = (threadIdx.x & 31) + (threadIdx.x >> 7) * 32;
    const int64_t l = (int64_t)blockIdx.x * kInfoLines + col;
    const bool in = l < gq.nl;
    const int st = in ? gq.star[l] : 0;
    const LineArgs g = star_view(gq, st);
    int amask = 0;
    if (w < DC / DS) {
        bool ok = true, wide = true, none = true;
        float need = 0.0f;
        if (in) {
            const LineScalars L = load_line(g, l);
            const int d1 = min(grp * DC + (w + 1) * DS, g.nd);
            for (int dd = grp * DC + w * DS; dd < d1; ++dd) {
                const DepthParams q = depth_params<0>(g, L, dd);
                ok = ok && q.a2 <= kFast2A2;
                wide = wide && q.a2 <= kWideA2;
                none = none && !pair_kept(g.keep, l, dd);
                need = fmaxf(need, sqrtf(q.a2) / q.k);
            }
        }
        amask = (ok ? 1 << w : 0) | (wide ? 16 << w : 0) | (none ? 256 << w : 0);
        int cls = kBoxClasses;
        if (gq.bgeo) {
            if (in && g.boxB) {
                need *= 9.0f / (gq.lnr * gq.shrink);
                const int *n = gq.nmin + ((int64_t)st * gq.nslab + grp * (DC / DS) + w) * 4;
                for (int c = kBoxClasses - 1; c >= 0; --c)
                    if (n[c] < kBoxNever && (float)((n[c] - 1) * g.boxB) >= need) cls = c;
            }
            for (int c = 1; c <= kBoxClasses; ++c) {
                const unsigned m = __ballot_sync(0xffffffffu, in && !none && cls >= c);
                if ((threadIdx.x & 31) == 0 && (l >> 5) < gq.wwords)
                    gq.wide[((int64_t)(c - 1) * gq.nslab + grp * (DC / DS) + w) * gq.wwords + (l >> 5)] = m;
            }
        }
        amask |= cls << (16 + 3 * w);
    }
    s_mask[w][col] = amask;
    __syncthreads();
    if (w == 0 && in) {
        LineInfo r;
        r.ilf = g.ilf[l];
        r.frac = g.frac[l];
        r.sp = g.sp[l];
        r.amask = s_mask[0][col] | s_mask[1][col] | s_mask[2][col] | s_mask[3][col];
        info[(int64_t)grp * gq.nl + l] = r;
    }
}

// ---- mbarrier waits (the bounded-wait probe) ---------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for phase `parity` of the barrier to complete; false after limit_ns.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t limit_ns) {
    if (mbar_test(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    for (;;) {
        if (mbar_test(bar, parity)) return true;
        if (global_ns() - t0 > limit_ns) return false;
    }
}


// ---------------------------------------------------------------------------
// Near-core kernels: the cells that the far-wing kernels leave.  At a slab whose damping the
// series forms take those are the points with U < cut by the far kernels' own U (a^2 <= kFast2A2 at
// every layer: the core x^2 < 36 of the slab's widest layer; a^2 <= kWideA2: x^2 < 400); otherwise the mid wing and
// core, |v|^2 + a^2 < 400, classified with the same prefactors, offset and test as the masked far
// form.  Every cell is counted exactly once across the two kernels.
//
// A CTA takes a (tile, group of ND layers) and a range of lines; its warps take the lines that
// reach the tile in turn.  In a warp, lane = (layer, point): ND layers of 32 / ND neighbouring points, so a line's
// prefactors are formed once per layer in the lanes that use them, its core (25 to 60 points,
// nearly the same at neighbouring layers) is swept 32 / ND points at a step with all lanes busy,
// and every lane owns its cell: the forward adds into the warp's own [point][layer] sums in
// shared memory without atomics, the reverse pass sums in registers and reduces once per line.
// (Before, lanes swept the concatenated cells of 32 (line, layer) items: finding a cell's item,
// fetching its 48 bytes, the shared-memory float atomics and the segmented scan of the reverse pass
// cost more than the profile, about 250 instructions per core cell.)
// Measured on 2e5 lines x 37,550 points: forward 2.11 -> 1.63 ms, reverse 3.50 -> 1.89 ms (5,300
// lines x 1,500 points, forward items cut by lines: 0.090 -> 0.086, reverse 0.146 -> 0.086 ms).
// ---------------------------------------------------------------------------

constexpr int kNearWarps = 8;        // warps per near-core CTA
constexpr int kNearBatch = 512;      // lines looked at together
struct NearList {
    int cnt[kNearBatch / 32];        // lines of each 32 whose near zone reaches the tile
    int line[kNearBatch];            // their places in the 32 | slabs (of the group) with only the core left << 8
                                     // | slabs cut at x^2 = 400 << 12
};

// Sweep of the near cells of lines [nlo, nhi) in the tile at the lane's layer: cell(i, A, H, dH)
// takes each cell that the lane owns, end(l, A, damping) closes a line (all lanes together) with the
// factors A a6 (and A a_rad, A a_Stark) of the NG damping sums.
template <int T, int ND, int NG, class Cell, class End>
__device__ __forceinline__ void near_sweep(const LineArgs &g, int t0, int nlo, int nhi, int dbase, NearList &list,
                                           const float *s_daw, Cell &&cell, End &&end) {
    constexpr int NP = 32 / ND;
    constexpr bool D = NG > 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = dbase + lane % ND, po = lane / ND;
    const float t0f = (float)t0, tendf = (float)(t0 + T - 1);
    const int sl0 = dbase / g.tDS, sl1 = (min(dbase + ND, g.nd) - 1) / g.tDS;   // slabs of the group's layers
    const int dc = min(d, g.nd - 1), slab = dc / g.tDS;
    for (int b0 = nlo; b0 < nhi; b0 += kNearBatch) {
        const int nch = (min(kNearBatch, nhi - b0) + 31) / 32;
        __syncthreads();
        for (int ch = warp; ch < nch; ch += kNearWarps) {
            // lane = line: does its near zone reach the tile at any slab of the group
            const int l = min(b0 + ch * 32 + lane, nhi - 1), sp = g.sp[l];
            const float il = g.ilf[l], fr = g.frac[l];
            const float dmin = fmaxf(0.0f, fmaxf(t0f - il - fr, il - tendf + fr));
            bool need = false;
            int core = 0;
            for (int sl = sl0; sl <= sl1; ++sl) {
                const int gs = sl * g.tDS / g.tDC, ws = sl - gs * (g.tDC / g.tDS);
                const int m = g.finfo[(int64_t)gs * g.nl + l].amask;
                const bool series = (m >> ws) & 1;
                core |= series ? 256 << (sl - sl0) : (m >> (4 + ws)) & 1 ? 4096 << (sl - sl0) : 0;
                need = need || (dmin < (series ? kCoreV : 1.0f) * __ldg(g.thr + sp * g.nslab + sl) && !((m >> (8 + ws)) & 1));
            }
            need = need && b0 + ch * 32 + lane < nhi;
            const unsigned m = __ballot_sync(0xffffffffu, need);
            if (need) list.line[ch * 32 + __popc(m & ((1u << lane) - 1u))] = lane | core;
            if (lane == 0) list.cnt[ch] = __popc(m);
        }
        __syncthreads();
        // the warps take the listed lines NP at a time (fewer where the list is short) in turn: lane
        // (q, layer) forms line q's prefactors and span at its layer, then the lanes sweep the lines
        // one after the other
        int total = 0;
        for (int k = 0; k < nch; ++k) total += list.cnt[k];
        const int per = max(1, min(NP, (total + kNearWarps - 1) / kNearWarps));
        int ch = 0, r = warp * per;         // (r counts on from list ch)
        for (;;) {
            while (ch < nch && r >= list.cnt[ch]) r -= list.cnt[ch++];
            if (ch >= nch) break;
            int mch = ch, mr = r + po;      // this lane's line
            while (mch < nch && mr >= list.cnt[mch]) mr -= list.cnt[mch++];
            const bool have = mch < nch && po < per;
            const int e = have ? list.line[mch * 32 + mr] : 0;
            const int l = have ? b0 + mch * 32 + (e & 31) : nlo;
            r += kNearWarps * per;
            const LineScalars L = load_line(g, l);
            const float ilf = g.ilf[l], frac = g.frac[l];
            const bool wide = (e >> (12 + slab - sl0)) & 1, series = wide || ((e >> (8 + slab - sl0)) & 1);
            const DepthParams p = depth_params<NG>(g, L, d);
            // the points that may be near [lo, hi], and (series slabs) those that certainly are; |u| <= reach
            // there, and u = expm1(Delta ln r) differs from Delta ln r by less than 0.6 reach of it
            const float cut = (wide ? kWideCut : 1.0f) * __ldg(g.cut + L.sp * g.nslab + slab);
            const float r2 = kFar2 - p.a2;
            const float reach = series ? sqrtf(cut * g.kunscale) : sqrtf(fmaxf(r2, 0.0f)) / p.k;
            int lo = 1 << 30, hi = -(1 << 30), ilo = 0, in = -1;
            if (have && p.k > 0.0f && (series || r2 > 0.0f) && pair_kept(g.keep, l, d)) {
                const float span = reach / g.lnr, m = fmaf(fmaf(0.6f, reach, 1e-3f), span, 0.01f);
                const int ic = (int)ilf;
                lo = max(max(t0, ic + (int)ceilf(frac - span - m)), ic - g.W);
                hi = min(min(t0 + T - 1, ic + (int)floorf(frac + span + m)), ic + g.W);
                if (series) {
                    ilo = max(lo, ic + (int)ceilf(frac - span + m));
                    in = min(hi, ic + (int)floorf(frac + span - m)) - ilo;
                }
            }
            const float ma = D ? p.a : sqrtf(p.a2), mcut = series ? cut : -1.0f;
            for (int q = 0; q < per; ++q) {
                const int src = q * ND + lane % ND;
                if (!__shfl_sync(0xffffffffu, (int)have, q * ND)) break;
                const int lq = __shfl_sync(0xffffffffu, l, q * ND);
                const float qil = __shfl_sync(0xffffffffu, ilf, q * ND), qfr = __shfl_sync(0xffffffffu, frac, q * ND);
                const float k = __shfl_sync(0xffffffffu, p.k, src), a = __shfl_sync(0xffffffffu, ma, src);
                const float a2 = __shfl_sync(0xffffffffu, p.a2, src), A = __shfl_sync(0xffffffffu, p.A, src);
                float damp[NG > 0 ? NG : 1];
#pragma unroll
                for (int f = 0; f < NG; ++f) damp[f] = __shfl_sync(0xffffffffu, p.damp[f], src);
                const float qcut = __shfl_sync(0xffffffffu, mcut, src);
                const int qlo = __shfl_sync(0xffffffffu, lo, src), qhi = __shfl_sync(0xffffffffu, hi, src);
                const int qilo = __shfl_sync(0xffffffffu, ilo, src), qin = __shfl_sync(0xffffffffu, in, src);
                const int i0 = __reduce_min_sync(0xffffffffu, qlo), i1 = __reduce_max_sync(0xffffffffu, qhi);
                for (int i = i0 + po; i <= i1; i += NP) {
                    bool own = qin >= 0 && (unsigned)(i - qilo) <= (unsigned)qin;
                    const float x = fabsf(offset_u((qil - (float)i) + qfr, g.lnr) * k);
                    const float z2 = fmaf(x, x, a2);
                    if (!own && i >= qlo && i <= qhi)
                        own = qcut >= 0.0f ? point_u2(g, qil - (float)i, qfr) < qcut : z2 < kFar2;
                    if (own) {
                        float H, dH;
                        if (z2 < kMid2)
                            voigt_core<D>(x, a, H, dH, s_daw);
                        else
                            voigt_mid<D>(x, a, H, dH);
                        cell(i, A, H, dH);
                    }
                }
                end(lq, A, damp);
            }
        }
    }
}

// Forward near-core sums into knear.  Work items: (star, tile, group of ND layers).
template <int T, int ND>
__global__ void __launch_bounds__(32 * kNearWarps) k_line_near_fwd(LineArgs gq, bool split) {
    extern __shared__ float4 smem4[];
    float *s_acc = reinterpret_cast<float *>(smem4);                  // [warps][T][ND]
    float *s_daw = s_acc + kNearWarps * T * ND;                       // Dawson table
    __shared__ NearList list;
    for (int k = threadIdx.x; k < kDawsonNodes * (kDawsonK + 1); k += blockDim.x) s_daw[k] = g_dawson[k];
    for_each_item(gq, [&](const LineArgs &g, int tile, int group, int nlo, int nhi, int) {
        const int t0 = tile * T, dbase = group * ND, ndg = min(ND, g.nd - dbase);
        for (int k = threadIdx.x; k < kNearWarps * T * ND; k += blockDim.x) s_acc[k] = 0.0f;
        __syncthreads();
        float *mine = s_acc + (threadIdx.x >> 5) * T * ND + (threadIdx.x & 31) % ND;
        near_sweep<T, ND, 0>(
            g, t0, nlo, nhi, dbase, list, s_daw,
            [&](int i, float A, float H, float) { mine[(i - t0) * ND] += A * H; }, [&](int, float, const float *) {});
        __syncthreads();
        for (int k = threadIdx.x; k < ndg * T; k += blockDim.x) {
            const int dl = k / T, q = k - dl * T;
            float v = 0.0f;
#pragma unroll
            for (int w = 0; w < kNearWarps; ++w) v += s_acc[(w * T + q) * ND + dl];
            float *out = g.knear + (int64_t)(dbase + dl) * g.ld + t0 + q;
            if (split)
                atomicAdd(out, v);     // one of the pieces of this item's lines (knear starts at zero)
            else
                *out = v;
        }
        __syncthreads();
    });
}

// Backward: per-line sums over the near cells of G stim A H and G stim A a6 dH/da (NG = 3: for every
// damping family), one FP64 add per (line, tile, layer group) and sum.
template <int T, int ND, int NG>
__global__ void __launch_bounds__(32 * kNearWarps, 4) k_line_near_bwd(LineArgs gq) {
    extern __shared__ float4 smem4[];
    float *s_g = reinterpret_cast<float *>(smem4);                    // [T][ND] G * stim
    float *s_daw = s_g + T * ND;                                      // Dawson table
    __shared__ NearList list;
    for (int k = threadIdx.x; k < kDawsonNodes * (kDawsonK + 1); k += blockDim.x) s_daw[k] = g_dawson[k];
    for_each_item(gq, [&](const LineArgs &g, int tile, int group, int nlo, int nhi, int) {
        const int t0 = tile * T, dbase = group * ND;
        for (int k = threadIdx.x; k < ND * T; k += blockDim.x) {
            const int dl = k / T, q = k - dl * T;
            s_g[q * ND + dl] = (dbase + dl < g.nd && t0 + q < g.nlam) ? g.Gt[(int64_t)(dbase + dl) * g.ld + t0 + q] : 0.0f;
        }
        __syncthreads();
        const float *mine = s_g + (threadIdx.x & 31) % ND;
        float S1 = 0.0f, S2 = 0.0f;
        near_sweep<T, ND, NG>(
            g, t0, nlo, nhi, dbase, list, s_daw,
            [&](int i, float, float H, float dH) {
                const float gs = mine[(i - t0) * ND];
                S1 = fmaf(gs, H, S1);
                S2 = fmaf(gs, dH, S2);
            },
            [&](int l, float A, const float *damp) {
                float v[1 + NG];
                v[0] = S1 * A;
#pragma unroll
                for (int f = 0; f < NG; ++f) v[1 + f] = S2 * damp[f];
                S1 = S2 = 0.0f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int q = 0; q <= NG; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
                if ((threadIdx.x & 31) == 0) {
#pragma unroll
                    for (int q = 0; q <= NG; ++q)
                        if (v[q] != 0.0f) atomicAdd(g.gacc + far_row(q) * g.nl + l, (double)v[q]);
                }
            });
        __syncthreads();
    });
}

template <int T, int ND, bool BWD>
constexpr size_t near_smem() {
    return ((size_t)(BWD ? 1 : kNearWarps) * ND * T + (size_t)kDawsonNodes * (kDawsonK + 1)) * sizeof(float);
}

static LineArgs make_args(pz_ctx *c) {
    LineArgs g;
    g.nlam = c->nlam;
    g.ld = c->ld;
    g.nd = c->nd;
    g.W = c->W;
    g.lnr = (float)c->lnr;
    for (int j = 0; j < 4; ++j) {
        g.rj[j] = (float)std::exp(-j * c->lnr);
        g.rm1j[j] = std::ldexp((float)std::expm1(-j * c->lnr), c->uexp);
    }
    g.uscale = std::ldexp(1.0f, c->uexp);
    g.kunscale = std::ldexp(1.0f, -2 * c->uexp);
    g.star = c->L.star;
    g.fext = nullptr;
    g.fpart = c->d_fpart;
    g.fcnt = c->d_fcnt;
    g.finfo = reinterpret_cast<const LineInfo *>(c->d_finfo);
    g.keep = c->d_keep;
    g.lam0cm = (float)(c->lambda0_nm * 1e-7);
    g.ilf = c->L.ilf;
    g.frac = c->L.frac;
    g.E = c->L.E;
    g.lamcm = c->L.lamcm;
    g.grad = c->L.grad;
    g.g4 = c->L.g4;
    g.g6 = c->L.g6;
    g.Q = c->L.Q;
    g.sp = c->L.sp;
    g.R = c->d_R;
    g.invdv = c->d_invdv;
    g.Ksd = c->d_Ksd;
    g.thr = c->d_thr;
    g.cut = c->d_cut;
    g.nslab = c->nslab;
    g.beta_hi = c->d_beta_hi;
    g.beta_lo = c->d_beta_lo;
    g.ne = c->d_ne;
    g.npert = c->d_npert;
    g.c2T = c->d_c2T;
    g.kline = (float *)c->d_kline;
    g.knear = c->d_knear;
    g.Gt = c->d_Gt;
    g.gacc = c->d_gacc + c->gacc_off;
    g.nl = c->L.n;
    g.items = nullptr;
    g.n_items = 0;
    g.ngroups = 1;
    g.ctr = nullptr;
    g.sstride = (int64_t)c->ns * c->nd;
    g.dstride = c->nd;
    g.bstride = (int64_t)c->nd * c->ld;
    g.tstride = (int64_t)c->ns * c->nslab;
    g.tDC = c->tiling.depth_per_cta();
    g.tDS = c->tiling.DS;
    g.boxB = g.boxsh = g.s_lo = g.nbox = 0;
    g.bgeo = c->box.d_geo;
    g.brow = c->box.stride;
    g.shrink = (float)std::max(0.5, 1.0 - 0.5 * (c->W + 1024.0) * c->lnr);
    g.nmin = c->box.d_nmin;
    g.bstart = c->box.d_start;
    g.wide = c->box.d_wide;
    g.wwords = (c->L.n + 31) / 32;
    return g;
}

// NG: damping families of the reverse pass (0: forward)
template <int T, int NG>
static cudaError_t launch_near(pz_ctx *c, LineArgs g, cudaStream_t s) {
    constexpr int ND = kNearDepths;
    constexpr bool BWD = NG > 0;
    g.items = BWD ? c->d_nitems_b : c->d_nitems_f;
    g.n_items = BWD ? c->n_nitems_b : c->n_nitems_f;
    if (g.n_items == 0) return cudaSuccess;
    g.ngroups = (c->nd + ND - 1) / ND;
    g.ctr = c->d_ctr + (BWD ? 3 : 0);
    constexpr size_t smem = near_smem<T, ND, BWD>();
    static std::atomic<bool> attr_set[kMaxDevices];
    const void *fn = BWD ? (const void *)k_line_near_bwd<T, ND, BWD ? NG : 1> : (const void *)k_line_near_fwd<T, ND>;
    if (!attr_set[c->device].load(std::memory_order_acquire)) {
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        attr_set[c->device].store(true, std::memory_order_release);
    }
    const int grid = persistent_grid(c, fn, 32 * kNearWarps, smem, g.n_items);
    if (!BWD && c->near_split) {
        const cudaError_t e = cudaMemsetAsync(c->d_knear, 0, sizeof(float) * (size_t)c->S * c->nd * c->ld, s);
        if (e != cudaSuccess) return e;
    }
    cudaEvent_t ev = prof_begin(c, s);
    if (BWD)
        k_line_near_bwd<T, ND, BWD ? NG : 1><<<grid, 32 * kNearWarps, smem, s>>>(g);
    else
        k_line_near_fwd<T, ND><<<grid, 32 * kNearWarps, smem, s>>>(g, c->near_split);
    prof_end(c, s, BWD ? PZ_K_NEAR_BWD : PZ_K_NEAR_FWD, ev);
    c->launches++;
    return cudaGetLastError();
}

// Dynamic shared memory of the far-wing kernels at LC lines per chunk: the warps' stages (layer
// constants, line records, prefactors) and (forward) the compensated sums of every thread, or
// (backward) the per-line sums.
static size_t far_fwd_smem(const Tiling &t, int LC, int NQ = kNQF) {
    return (size_t)t.GW * warp_stage_quads(LC, t.DS, NQ) * sizeof(float4) +
           (size_t)t.DS * 32 * t.GW * 2 * sizeof(float4);
}
static size_t far_bwd_smem(const Tiling &t, int LC, int NQ, int NS = 1) {
    return (size_t)t.GW * warp_stage_quads(LC, t.DS, NQ) * sizeof(float4) +
           (size_t)NS * 2 * LC * t.GW * sizeof(float2) + (size_t)NS * t.GW * kBwdBatch * 32 * sizeof(float2);
}

// A tiling is taken if its chunk fits with two (three) quads per depth pair and line; the lines
// that the kernels stage at a time are cut to what fits with the series' coefficients.
bool tiling_fits(const Tiling &t) {
    return far_fwd_smem(t, t.LC, 2) <= kFarSmemMax && far_bwd_smem(t, t.LCB, 3) <= kFarSmemMax;
}
static int far_fwd_chunk(const Tiling &t) {
    int LC = t.LC;
    while (LC > 1 && far_fwd_smem(t, LC) > kFarSmemMax) --LC;
    return LC;
}
static int far_bwd_chunk(const Tiling &t, int NQ, int NS) {
    int LC = t.LCB;
    while (LC > 1 && far_bwd_smem(t, LC, NQ, NS) > kFarSmemMax) --LC;
    return LC;
}

// Line records of the far-wing kernels for the current tiling, into the context's
// buffer (sized by ensure_far_tables).  They depend on the corrections, the centre test and
// the tiling; the reverse pass after a forward finds the forward's (finfo_valid).
static cudaError_t launch_far_info(pz_ctx *c, const LineArgs &g, int ngroups, cudaStream_t s) {
    const dim3 grid((unsigned)((c->L.n + kInfoLines - 1) / kInfoLines), (unsigned)ngroups);
    k_far_info<<<grid, 256, 0, s>>>(g, c->tiling.depth_per_cta(), c->tiling.DS, reinterpret_cast<LineInfo *>(c->d_finfo));
    c->launches++;
    return cudaGetLastError();
}

size_t far_info_bytes(const pz_ctx *c) {
    const int DC = c->tiling.depth_per_cta();
    const int ng = (c->nd + DC - 1) / DC;
    return (size_t)ng * std::max<int64_t>(c->L.n, 1) * sizeof(LineInfo);
}

// ---- box expansions: host side -------------------------------------------------
// Which stars use the expansions, and their geometry.  A box of B points, a power of two near half
// the star's widest near zone (20 Doppler widths in grid points), so that the nearest pairs are 3 or 4
// boxes apart: smaller boxes raise the pairs as 1/B^2, larger ones the points left to the direct sum.
void box_choose(pz_ctx *c, const std::vector<int64_t> &evals) {
    BoxPlan &p = c->box;
    p.of.assign(c->S, -1);
    if (c->prec != PZ_MIXED) return;
    std::vector<int> size(c->S, 0);      // log2 B of each star, 0: no boxes
    const size_t row = (size_t)c->ns * c->nd;
    for (int st = 0; st < c->S; ++st) {
        // the expansions cost a fixed amount per (point, layer) and some 0.1 ms of latency per pass:
        // below about 200 lines per window, or 2e8 (line, point, layer) terms, the direct sum
        // is as fast (574 points x 1,416 lines, 3.5e7 terms: 0.63 ms direct, 0.72 ms with boxes; 4,000 x
        // 2,000, 2.5e8: 0.22 against 0.18 ms; 2,200 x 12,000, 1.7e9, with the reverse pass: 1.35 against
        // 0.92 ms; 37,550 x 200,000, 4.3e10: 23.0 against 7.0 ms, near cores aside)
        const double lines = (double)(c->h_line_off[st + 1] - c->h_line_off[st]);
        const double per_window = lines / (double)c->nlam * (2.0 * c->W + 1.0);
        if (per_window < 200.0 || (double)evals[st] < 2e8) continue;
        const auto inv = c->h_invdv.begin() + st * row;
        const double thr = 20.0 / (kC * (double)*std::min_element(inv, inv + row) * c->lnr);
        int sh = 2;
        while (sh < 5 && thr >= 2.5 * (1 << sh)) ++sh;
        // the window ends' tables need a wide offset (few moments), and at least some whole boxes
        if ((c->W + 1) / (1 << sh) - 1 >= 8) size[st] = sh;
    }
    for (int sh = 2; sh <= 5; ++sh) {
        BoxGroup b;
        b.first = (int)p.stars.size();
        for (int st = 0; st < c->S; ++st)
            if (size[st] == sh) {
                p.of[st] = (int)p.groups.size();
                p.stars.push_back(st);
            }
        b.count = (int)p.stars.size() - b.first;
        if (b.count == 0) continue;
        b.sh = sh;
        b.B = 1 << sh;
        b.omax = (c->W + 1) / b.B - 1;
        b.rem = c->W + 1 - (b.omax + 1) * b.B;
        b.s_lo = -((c->W + b.B - 1) / b.B);
        b.nbox = (int)((c->nlam - 1 + c->W) / b.B) - b.s_lo + 1;
        b.ntb = (int)((c->nlam + b.B - 1) / b.B);
        b.KE = box_order(b.omax + 1) + 1 <= 5 ? 5 : 8;
        p.stride = std::max<int64_t>(p.stride, (int64_t)kBoxSplit * b.nbox + 1);
        p.groups.push_back(b);
    }
}

// Forward launches take whole stars while they fit, then parts of one star's source boxes (the field
// of a part is added to the near-core sums as the whole's is); the reverse pass keeps the moments of
// G of whole stars, 56 bytes per layer and box.
size_t box_cut(pz_ctx *c, size_t bytes) {
    constexpr int kLeastBoxes = 16;
    size_t most = 0;
    for (BoxGroup &b : c->box.groups) {
        const size_t per_box = sizeof(float) * (kBoxClasses * kBoxK + (size_t)b.B * b.KE) * c->nd;
        const size_t bwd = sizeof(float) * (size_t)b.ntb * kBoxK * c->nd, star = std::max(per_box * b.nbox, bwd);
        b.chunk = (int)std::min<size_t>(b.count, std::max<size_t>(1, bytes / star));
        b.span = (int)std::min<size_t>(b.nbox, std::max<size_t>(1, bytes / per_box));
        const size_t need = std::max(per_box * b.span, bwd) * b.chunk;
        if (need > bytes && b.span < std::min(kLeastBoxes, b.nbox)) return 0;
        most = std::max(most, need);
    }
    return most;
}
size_t box_wide_bytes(const pz_ctx *c) {
    return (size_t)kBoxClasses * c->nslab * (size_t)((c->L.n + 31) / 32) * sizeof(uint32_t);
}

static cudaError_t launch_box_group_tables(pz_ctx *c, const BoxGroup &b) {
    k_box_tables<<<dim3(b.omax + 2, 2), 256>>>(b.B, c->lnr, b.omax, b.d_C);
    k_box_edges<<<dim3(b.B, 2, 2), 32>>>(b.B, b.omax, b.KE, b.d_C, b.d_E);
    k_box_start<<<dim3(kBoxSplit * b.nbox / 256 + 1, b.count), 256>>>(
        kBoxSplit * b.nbox, b.s_lo, b.B, c->box.d_stars + b.first, c->L.il32, c->d_line_off, c->box.stride, c->box.d_start);
    // operators of f^2, f^3, f^4 on the Chebyshev basis: column k of (1/m)(d + p eps)(d + q eps)
    const double eps = 0.5 * b.B * c->lnr;
    std::vector<double> cur((size_t)kBoxK * kBoxK, 0.0);   // [k][j]: image of T_k as coefficients of T_j
    for (int k = 0; k < kBoxK; ++k) cur[k * kBoxK + k] = 1.0;
    auto apply = [&](double *v, double add) {                // v <- (d/dx + add) v in Chebyshev coefficients
        double dv[kBoxK + 2] = {0.0};
        for (int j = kBoxK - 1; j >= 1; --j) dv[j - 1] = dv[j + 1] + 2.0 * j * v[j];
        dv[0] *= 0.5;
        for (int j = 0; j < kBoxK; ++j) v[j] = dv[j] + add * v[j];
    };
    std::vector<float> A((size_t)3 * kBoxK * kBoxK);
    const double m[3] = {6.0, 20.0, 42.0};
    for (int q = 0; q < 3; ++q)
        for (int k = 0; k < kBoxK; ++k) {
            double *v = &cur[(size_t)k * kBoxK];
            apply(v, (2 * q + 2) * eps);
            apply(v, (2 * q + 3) * eps);
            for (int j = 0; j < kBoxK; ++j) {
                v[j] /= m[q];
                A[((size_t)q * kBoxK + k) * kBoxK + j] = (float)v[j];
            }
        }
    const cudaError_t e = cudaMemcpy(b.d_A, A.data(), A.size() * sizeof(float), cudaMemcpyHostToDevice);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_box_tables(pz_ctx *c) {
    for (const BoxGroup &b : c->box.groups) {
        const cudaError_t e = launch_box_group_tables(c, b);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Arguments of the stars [first, ...) of BoxPlan::stars, all of group p, and its source boxes [box0, box0 + nbox).
static BoxArgs box_args(const pz_ctx *c, const BoxGroup &p, int first, int box0, int nbox) {
    BoxArgs b;
    b.B = p.B;
    b.omax = p.omax;
    b.rem = p.rem;
    b.s_lo = p.s_lo + box0;
    b.nbox = nbox;
    b.ntb = p.ntb;
    b.box0 = box0;
    b.tgt0 = std::max(0, b.s_lo - p.omax - 2);       // first box that the sources reach
    b.DC = c->tiling.depth_per_cta();
    b.DS = c->tiling.DS;
    b.stars = c->box.d_stars + first;
    b.invh = 2.0f / p.B;
    b.ctr = 0.5f * (p.B - 1);
    const double eps = 0.5 * p.B * c->lnr;
    b.kapscale = (float)(1.0 / (std::ldexp(eps, c->uexp) * std::ldexp(eps, c->uexp)));
    b.A = p.d_A;
    b.C = p.d_C;
    b.E = p.d_E;
    b.nmin = c->box.d_nmin;
    b.M = c->box.d_ws;
    b.PM = c->box.d_ws + (size_t)p.chunk * p.span * kBoxClasses * kBoxK * c->nd;
    b.N = c->box.d_ws;
    return b;
}

// Fewer than two boxes per SM: the boxes' blocks are cut further (by indices of the box or layers).
static bool box_few(const pz_ctx *c, const BoxGroup &p) {
    return (int64_t)p.nbox * std::min(p.chunk, p.count) < 2 * (int64_t)c->n_sm;
}

// Forward: moments of the lines, then the far field of every point into knear.
template <int KE, int NP>
static cudaError_t launch_box_fwd_parts(pz_ctx *c, const BoxGroup &p, const LineArgs &g, cudaStream_t s) {
    static std::atomic<bool> attr_set[kMaxDevices];
    if (!attr_set[c->device].load(std::memory_order_acquire)) {
        const cudaError_t e = cudaFuncSetAttribute(k_box_moments<KE, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)box_moment_smem<NP>(kMaxDepth));
        if (e != cudaSuccess) return e;
        const cudaError_t ef = cudaFuncSetAttribute(k_box_field<KE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    (int)box_field_smem(32, kMaxDepth));
        if (ef != cudaSuccess) return ef;
        attr_set[c->device].store(true, std::memory_order_release);
    }
    const int thr_m = (NP * c->nd + 31) / 32 * 32, thr_f = (kBoxSplit * c->nd + 31) / 32 * 32;
    for (int k = 0; k < p.count; k += p.chunk)
        for (int box0 = 0; box0 < p.nbox; box0 += p.span) {
            const int n = std::min(p.chunk, p.count - k);
            const BoxArgs b = box_args(c, p, p.first + k, box0, std::min(p.span, p.nbox - box0));
            const int tgt = std::min(p.ntb, b.s_lo + b.nbox + p.omax + 2) - b.tgt0;
            if (tgt <= 0) continue;
            k_box_moments<KE, NP><<<dim3(b.nbox, n), thr_m, box_moment_smem<NP>(c->nd), s>>>(g, b);
            k_box_field<KE><<<dim3(tgt, n), thr_f, box_field_smem(b.B, c->nd), s>>>(g, b);
            c->launches += 2;
        }
    return cudaGetLastError();
}
template <int KE>
static cudaError_t launch_box_fwd(pz_ctx *c, const BoxGroup &p, const LineArgs &g, cudaStream_t s) {
    return box_few(c, p) ? launch_box_fwd_parts<KE, kBoxSplit>(c, p, g, s) : launch_box_fwd_parts<KE, 1>(c, p, g, s);
}

// Backward: moments of G, then every line's sums over the points its boxes reach, into gacc.
template <int KE, bool FOUR>
static cudaError_t launch_box_bwd(pz_ctx *c, const BoxGroup &p, const LineArgs &g, cudaStream_t s) {
    const int thr = (c->nd + 31) / 32 * 32;
    // several blocks per box, each with part of the layers, where the lines fill few boxes
    const int nz = box_few(c, p) ? std::min(3, c->nd) : 1;
    const size_t smem = box_grad_smem(p.B, KE, (c->nd + nz - 1) / nz);
    static std::atomic<bool> attr_set[kMaxDevices];
    if (!attr_set[c->device].load(std::memory_order_acquire)) {
        const cudaError_t e = cudaFuncSetAttribute(k_box_grad<KE, FOUR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)box_grad_smem(32, KE, kMaxDepth));
        if (e != cudaSuccess) return e;
        attr_set[c->device].store(true, std::memory_order_release);
    }
    for (int k = 0; k < p.count; k += p.chunk) {
        const int n = std::min(p.chunk, p.count - k);
        const BoxArgs b = box_args(c, p, p.first + k, 0, p.nbox);
        k_box_gmoments<<<dim3(b.ntb, n), thr, sizeof(float) * c->nd * (b.B + 1), s>>>(g, b);
        k_box_grad<KE, FOUR><<<dim3(b.nbox, n, nz), 32 * kBoxGradWarps, smem, s>>>(g, b);
        c->launches += 2;
    }
    return cudaGetLastError();
}

template <int J, int DS, int MINB>
static cudaError_t launch_fwd_t(pz_ctx *c, cudaStream_t s) {
    if (c->n_fitems == 0) return cudaErrorInvalidConfiguration;   // the tiling's tables could not be allocated
    const Tiling &t = c->tiling;
    LineArgs g = make_args(c);
    const int LC = far_fwd_chunk(t);
    const size_t smem = far_fwd_smem(t, LC);
    // with a centre test the kernel stages only the lines each warp's slab sweeps (GATHER)
    const bool gather = c->d_keep != nullptr;
    auto kern = gather ? k_line_fwd<J, DS, MINB, true> : k_line_fwd<J, DS, MINB, false>;
    static std::atomic<bool> attr_set[kMaxDevices][2];
    if (!attr_set[c->device][gather].load(std::memory_order_acquire)) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFarSmemMax);
        attr_set[c->device][gather].store(true, std::memory_order_release);
    }
    cudaError_t e = cudaMemsetAsync(c->d_ctr, 0, 2 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    const int ngroups = (c->nd + t.depth_per_cta() - 1) / t.depth_per_cta();
    if (c->L.n > 0) {
        e = launch_far_info(c, g, ngroups, s);
        if (e != cudaSuccess) return e;
        c->finfo_valid = true;
    }
    e = launch_near<32 * J, 0>(c, g, s);
    if (e != cudaSuccess) return e;
    g.items = c->d_fitems;
    g.fext = c->d_fext;
    g.n_items = c->n_fitems;
    g.ngroups = ngroups;
    g.ctr = c->d_ctr + 1;
    for (const BoxGroup &p : c->box.groups) {
        e = p.KE == 5 ? launch_box_fwd<5>(c, p, g, s) : launch_box_fwd<8>(c, p, g, s);
        if (e != cudaSuccess) return e;
    }
    if (c->n_fsplit > 0) {
        e = cudaMemsetAsync(c->d_fcnt, 0, sizeof(int) * c->n_fsplit, s);
        if (e != cudaSuccess) return e;
    }
    int grid = persistent_grid(c, kern, 32 * t.GW, smem, g.n_items);
    kern<<<grid, 32 * t.GW, smem, s>>>(g, t.GW, LC);
    c->launches++;
    return cudaGetLastError();
}

// Reverse pass of the lines; four: with the radiative and Stark damping sums.
cudaError_t launch_line_bwd_mixed(pz_ctx *c, cudaStream_t s, bool four) {
    if (c->n_fitems == 0) return cudaErrorInvalidConfiguration;
    const Tiling &t = c->tiling;
    const LineArgs g = make_args(c);
    cudaError_t e = cudaMemsetAsync(c->d_ctr + 2, 0, 2 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    if (c->n_bitems > 0) {
        LineArgs gb = g;
        gb.items = c->d_bitems;
        gb.n_items = c->n_bitems;
        gb.ngroups = (c->nd + t.depth_per_cta() - 1) / t.depth_per_cta();
        gb.ctr = c->d_ctr + 2;
        gb.fext = c->d_bext;
        if (!c->finfo_valid) {
            e = launch_far_info(c, gb, gb.ngroups, s);
            if (e != cudaSuccess) return e;
        }
        for (const BoxGroup &p : c->box.groups) {
            e = p.KE == 5 ? (four ? launch_box_bwd<5, true>(c, p, gb, s) : launch_box_bwd<5, false>(c, p, gb, s))
                          : (four ? launch_box_bwd<8, true>(c, p, gb, s) : launch_box_bwd<8, false>(c, p, gb, s));
            if (e != cudaSuccess) return e;
        }
        const int NQ = four ? kNQB4 : kNQB, NS = four ? 2 : 1, LC = far_bwd_chunk(t, NQ, NS);
        e = (four ? launch_far_bwd4 : launch_far_bwd)(c, gb, LC, far_bwd_smem(t, LC, NQ, NS), s);
        if (e != cudaSuccess) return e;
    }
    if (t.J == 4) return four ? launch_near<128, 3>(c, g, s) : launch_near<128, 1>(c, g, s);
    return four ? launch_near<64, 3>(c, g, s) : launch_near<64, 1>(c, g, s);
}

#define PZ_TILE_FWD(A, B, M) \
    if (c->tiling.J == A && c->tiling.DS == B && c->tiling.minb == M) return launch_fwd_t<A, B, M>(c, s);
cudaError_t launch_line_fwd_mixed(pz_ctx *c, cudaStream_t s) {
    PZ_TILE_LIST(PZ_TILE_FWD)
    return cudaErrorInvalidConfiguration;
}

bool tiling_supported(int J, int DS, int minb) {
#define PZ_TILE_OK(A, B, M) \
    if (J == A && DS == B && minb == M) return true;
    PZ_TILE_LIST(PZ_TILE_OK)
#undef PZ_TILE_OK
    return false;
}

// ---------------------------------------------------------------------------
// Plain FP64 GPU form: one thread per (lambda, depth), FP64 Voigt, no expansions and no
// compensation; every line term of every window point is summed in line order.
// ---------------------------------------------------------------------------

struct Fp64Args {
    int64_t nlam, ld, nl;
    int nd, ns, W;
    double lnr, lam0cm;
    const int32_t *il;       // integer centres, sorted within each star's segment
    const int64_t *line_off; // [S+1] star segments
    const int32_t *star;
    const double *x64;       // fractional centre
    const int32_t *sp;
    const float *lg_gf, *dgf, *E, *lg_rad, *lg_4, *lg_6, *dg6, *dgrad, *dg4;
    const double *T, *rho, *ne, *npert, *pop, *mass, *xi, *dab;   // [S][nd], [S][ns][nd], [S][ns], [S]
    int dsel;                // backward: damping family of the second sum (0 vdW, 1 rad, 2 Stark)
    const int32_t *eos;
    double *kline;           // [S][nd][ld]
    const double *Gt;        // [S][nd][ld]
    double *gacc;
    const uint32_t *keep;    // centre-test mask [nl][kKeepWords] or NULL (all kept)
    const double *kc;        // [S][nd][ld] continuum opacity (centre test)
};

struct LineTerm64 {
    double A, a, a6, kv;   // strength, damping, the selected family's part of it, c/dv_D
};

__device__ __forceinline__ LineTerm64 term64(const Fp64Args &g, int64_t l, int st, int d) {
    LineTerm64 q;
    const int s = g.sp[l];
    const int64_t sd = (int64_t)st * g.nd + d;
    const double T = g.T[sd];
    const double xi = g.xi[st];
    const double dv = sqrt(2.0 * kKB * T / (g.mass[(int64_t)st * g.ns + s] * kAMU) + xi * xi);
    const double lamcm = g.lam0cm * exp(g.x64[l] * g.lnr);
    const double inv_dnu = lamcm / dv;
    const double gf = exp10((double)g.lg_gf[l] + (double)g.dgf[l]);
    const double dab = (g.eos && g.eos[s] >= 0) ? g.dab[g.eos[s]] : 0.0;
    const double pop = g.pop[((int64_t)st * g.ns + s) * g.nd + d] * exp10(dab);
    const double boltz = exp(-(double)g.E[l] * kEV / (kKB * T));
    q.A = (kPI * kE * kE / (kME * kC)) / kSQRTPI * gf * (pop / g.rho[sd]) * boltz * inv_dnu;
    const double g6n = exp10((double)g.lg_6[l] + (double)g.dg6[l]) * g.npert[sd];
    const double grad = exp10((double)g.lg_rad[l] + (double)g.dgrad[l]);
    const double g4n = exp10((double)g.lg_4[l] + (double)g.dg4[l]) * g.ne[sd];
    // (a^2 stays finite: voigt64 takes 1/(v^2 + a^2) by Newton's iteration, and H is zero there in any case)
    q.a = fmin((grad + g4n + g6n) * inv_dnu / (4.0 * kPI), 1e150);
    q.a6 = (g.dsel == 0 ? g6n : (g.dsel == 1 ? grad : g4n)) * inv_dnu / (4.0 * kPI);
    q.kv = kC / dv;
    return q;
}

__device__ __forceinline__ int64_t lower_bound_i32(const int32_t *a, int64_t lo, int64_t hi, int32_t key) {
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (a[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// One thread per (lambda, depth, star); loops over the lines whose window covers lambda.  The
// block's threads form the terms of kFp64Lines lines at a time, once per block (the exponentials and
// powers of ten of a term cost more than ten profiles: 600 lines x 1,019 points, 2.2e7 profiles, 17.3 ->
// 4.6 ms with the cheaper profile; bound by the FP64 pipe, about 110 operations a profile).
constexpr int kFp64Lines = 128;
__global__ void __launch_bounds__(kFp64Lines) k_line_fwd_fp64(Fp64Args g) {
    __shared__ LineTerm64 s_q[kFp64Lines];
    __shared__ double s_x[kFp64Lines];
    __shared__ int s_il[kFp64Lines];
    const int64_t i0 = (int64_t)blockIdx.x * kFp64Lines, i = i0 + threadIdx.x;
    const int d = blockIdx.y, st = blockIdx.z;
    const int64_t b0 = g.line_off[st], b1 = g.line_off[st + 1];
    const int64_t l0 = lower_bound_i32(g.il, b0, b1, (int32_t)(i0 - g.W));
    const int64_t l1 = lower_bound_i32(g.il, b0, b1, (int32_t)(i0 + kFp64Lines + g.W));
    double sum = 0.0;
    for (int64_t c0 = l0; c0 < l1; c0 += kFp64Lines) {
        const int n = (int)min((int64_t)kFp64Lines, l1 - c0);
        __syncthreads();
        if (threadIdx.x < n) {
            const int64_t l = c0 + threadIdx.x;
            const bool kept = pair_kept(g.keep, l, d);
            if (kept) s_q[threadIdx.x] = term64(g, l, st, d);
            s_x[threadIdx.x] = g.x64[l];
            s_il[threadIdx.x] = kept ? g.il[l] : INT32_MAX / 2;    // (rejected pairs are out of every window)
        }
        __syncthreads();
        for (int j = 0; j < n; ++j) {
            if (llabs((long long)s_il[j] - (long long)i) > g.W) continue;
            const LineTerm64 &q = s_q[j];
            const double u = expm1_small((s_x[j] - (double)i) * g.lnr);   // lambda_l/lambda_i - 1
            double H, dH;
            voigt64<false>(u * q.kv, q.a, H, dH);
            sum += q.A * H;
        }
    }
    if (i >= g.nlam) return;
    const double lam = g.lam0cm * exp((double)i * g.lnr);
    const double stim = -expm1(-kC2 / (lam * g.T[(int64_t)st * g.nd + d]));
    g.kline[((int64_t)st * g.nd + d) * g.ld + i] = stim * sum;
}

// one thread per (line, depth); loops over the line's window
__global__ void k_line_bwd_fp64(Fp64Args g) {
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int d = blockIdx.y;
    if (l >= g.nl || !pair_kept(g.keep, l, d)) return;
    const int st = g.star[l];
    LineTerm64 q = term64(g, l, st, d);
    const int64_t il = g.il[l];
    const int64_t i0 = max((int64_t)0, il - g.W), i1 = min(g.nlam - 1, il + g.W);
    const double *Grow = g.Gt + ((int64_t)st * g.nd + d) * g.ld;
    double s1 = 0.0, s2 = 0.0;
    for (int64_t i = i0; i <= i1; ++i) {
        const double u = expm1_small((g.x64[l] - (double)i) * g.lnr);
        double H, dH;
        voigt64<true>(u * q.kv, q.a, H, dH);
        double gs = Grow[i];
        s1 += gs * q.A * H;
        s2 += gs * q.A * dH * q.a6;
    }
    atomicAdd(g.gacc + l, s1);
    atomicAdd(g.gacc + g.nl + l, s2);
}

static Fp64Args make_args64(pz_ctx *c) {
    Fp64Args g;
    g.nlam = c->nlam;
    g.ld = c->ld;
    g.nl = c->L.n;
    g.nd = c->nd;
    g.ns = c->ns;
    g.W = c->W;
    g.lnr = c->lnr;
    g.lam0cm = c->lambda0_nm * 1e-7;
    g.il = c->L.il32;
    g.line_off = c->d_line_off;
    g.star = c->L.star;
    g.x64 = c->L.x64;
    g.sp = c->L.sp;
    g.lg_gf = c->L.lg_gf;
    g.dgf = c->L.dgf;
    g.E = c->L.E;
    g.lg_rad = c->L.lg_rad;
    g.lg_4 = c->L.lg_4;
    g.lg_6 = c->L.lg_6;
    g.dg6 = c->L.dg6;
    g.dgrad = c->L.dgrad;
    g.dg4 = c->L.dg4;
    g.dsel = c->bwd_dsel;
    g.T = c->d_T;
    g.rho = c->d_rho64;
    g.ne = c->d_ne64;
    g.npert = c->d_npert64;
    g.pop = c->d_pop64;
    g.mass = c->d_mass64;
    g.xi = c->d_xi64;
    g.dab = c->d_dab;
    g.eos = c->n_elem > 0 ? c->d_eos : nullptr;
    g.kline = (double *)c->d_kline;
    g.Gt = c->d_Gt64;
    g.gacc = c->d_gacc + c->gacc_off;
    g.keep = c->d_keep;
    g.kc = c->d_kc;
    return g;
}

// Centre-test mask, once per call of pz_set_centre_test, in FP64 (the decision is the
// same rule as the FP64 oracle's): the pair (l, d) is kept when the peak of its term at
// its centre grid point ic (i_l clipped to the grid), bounded with H(a, 0) <= 1,
// reaches eta times the continuum there:
//   (1 - exp(-h c / (lambda_ic k T_d))) A_ld >= eta kappa_c(ic, d).
// One thread per (line, depth); kept pairs set their bit and are counted.
__global__ void k_centre_mask(Fp64Args g, double eta, uint32_t *keep, unsigned long long *count) {
    const int64_t n = g.nl * g.nd;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = k / g.nd;
        const int d = (int)(k - l * g.nd);
        const int st = g.star[l];
        const LineTerm64 q = term64(g, l, st, d);
        const int64_t ic = min(max((int64_t)g.il[l], (int64_t)0), g.nlam - 1);
        const double lam = g.lam0cm * exp((double)ic * g.lnr);
        const double stim = -expm1(-kC2 / (lam * g.T[(int64_t)st * g.nd + d]));
        const double kc = g.kc[((int64_t)st * g.nd + d) * g.ld + ic];
        if (stim * q.A >= eta * kc) {
            atomicOr(keep + l * kKeepWords + (d >> 5), 1u << (d & 31));
            if (count) atomicAdd(count, 1ull);
        }
    }
}

cudaError_t launch_centre_mask(pz_ctx *c, double eta, unsigned long long *d_count, cudaStream_t s) {
    Fp64Args g = make_args64(c);
    const int64_t n = c->L.n * (int64_t)c->nd;
    if (n == 0) return cudaSuccess;
    const int grid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)std::max(c->n_sm, 1) * 32);
    k_centre_mask<<<grid, 256, 0, s>>>(g, eta, c->d_keep, d_count);
    return cudaGetLastError();
}

cudaError_t launch_line_fwd_fp64(pz_ctx *c, cudaStream_t s) {
    Fp64Args g = make_args64(c);
    dim3 grid((unsigned)((c->nlam + kFp64Lines - 1) / kFp64Lines), c->nd, c->S);
    k_line_fwd_fp64<<<grid, kFp64Lines, 0, s>>>(g);
    c->launches++;
    return cudaGetLastError();
}

cudaError_t launch_line_bwd_fp64(pz_ctx *c, cudaStream_t s) {
    if (c->L.n == 0) return cudaSuccess;
    Fp64Args g = make_args64(c);
    dim3 grid((unsigned)((c->L.n + 127) / 128), c->nd);
    k_line_bwd_fp64<<<grid, 128, 0, s>>>(g);
    c->launches++;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// corrections (Eq. 10): the per-line values are gathered from the caller-order (master)
// corrections, Q_l = Qbase_l 10^dgf, gamma_beta,l = gamma_beta,l(base) 10^dbeta for the
// three damping families, R_sd = Rbase_sd 10^dab
// ---------------------------------------------------------------------------
struct CorrArgs {
    int64_t n;
    const int32_t *orig;
    const double *Qbase;
    const float *g6base, *gradbase, *g4base;
    const float *mdgf, *mdg6, *mdgrad, *mdg4;   // caller order
    float *dgf, *dg6, *dgrad, *dg4;             // per line
    float *Q, *g6, *grad, *g4;
};

__global__ void k_apply_line_corr(CorrArgs a) {
    int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= a.n) return;
    const int32_t o = a.orig[l];
    const float cgf = a.mdgf[o], c6 = a.mdg6[o], cr = a.mdgrad[o], c4 = a.mdg4[o];
    a.dgf[l] = cgf;
    a.dg6[l] = c6;
    a.dgrad[l] = cr;
    a.dg4[l] = c4;
    a.Q[l] = (float)(a.Qbase[l] * exp10((double)cgf));
    a.g6[l] = (float)((double)a.g6base[l] * exp10((double)c6));
    a.grad[l] = (float)((double)a.gradbase[l] * exp10((double)cr));
    a.g4[l] = (float)((double)a.g4base[l] * exp10((double)c4));
}

// R over [S][ns][nd]
__global__ void k_apply_abund(int64_t n, int ns, int nd, const double *Rbase, const double *dab, const int32_t *eos,
                              int use, float *R) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n) return;
    int s = (int)((idx / nd) % ns);
    double f = (use && eos[s] >= 0) ? exp10(dab[eos[s]]) : 1.0;
    R[idx] = (float)(Rbase[idx] * f);
}

cudaError_t launch_apply_corrections(pz_ctx *c, cudaStream_t s) {
    c->finfo_valid = false;
    if (c->L.n > 0) {
        CorrArgs a{c->L.n,     c->L.orig,  c->L.Qbase, c->L.g6base, c->L.gradbase, c->L.g4base,
                   c->d_mdgf,  c->d_mdg6,  c->d_mdgrad, c->d_mdg4, c->L.dgf,      c->L.dg6,
                   c->L.dgrad, c->L.dg4,   c->L.Q,     c->L.g6,     c->L.grad,     c->L.g4};
        k_apply_line_corr<<<(unsigned)((c->L.n + 255) / 256), 256, 0, s>>>(a);
        c->launches++;
    }
    int64_t n = (int64_t)c->S * c->ns * c->nd;
    k_apply_abund<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, c->ns, c->nd, c->d_Rbase, c->d_dab, c->d_eos,
                                                             c->n_elem > 0, c->d_R);
    c->launches++;
    return cudaGetLastError();
}

// plain gradient step on the caller-order corrections: delta -= lr * dL/ddelta
__global__ void k_update_corr(int64_t n, const double *gline, float lr_gf, float lr_g6, float *mdgf, float *mdg6) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    mdgf[k] = (float)((double)mdgf[k] - (double)lr_gf * gline[k]);
    mdg6[k] = (float)((double)mdg6[k] - (double)lr_g6 * gline[n + k]);
}

__global__ void k_update_abund(int n, const double *gab, double lr, double *dab) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) dab[k] -= lr * gab[k];
}

cudaError_t launch_update(pz_ctx *c, float lr_gf, float lr_g6, float lr_ab, cudaStream_t s) {
    if (c->nl_caller > 0) {
        k_update_corr<<<(unsigned)((c->nl_caller + 255) / 256), 256, 0, s>>>(c->nl_caller, c->d_gline, lr_gf, lr_g6,
                                                                            c->d_mdgf, c->d_mdg6);
        c->launches++;
    }
    if (c->n_elem > 0) {
        k_update_abund<<<(c->n_elem + 255) / 256, 256, 0, s>>>(c->n_elem, c->d_gab, (double)lr_ab, c->d_dab);
        c->launches++;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// linked correction groups (Sec. 6): every member l of group q takes the group's four
// corrections, delta_{q(l)}, and the group's gradient is the sum of its members'
// ---------------------------------------------------------------------------
// x: [4][G] (gf, rad, Stark, vdW) -> caller-order masters; lines without a group take 0
__global__ void k_group_gather(int64_t n, int64_t G, const int32_t *grp, const float *x, float *mdgf, float *mdgrad,
                               float *mdg4, float *mdg6) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int32_t q = grp[k];
    const bool in = q >= 0;
    mdgf[k] = in ? x[q] : 0.0f;
    mdgrad[k] = in ? x[G + q] : 0.0f;
    mdg4[k] = in ? x[2 * G + q] : 0.0f;
    mdg6[k] = in ? x[3 * G + q] : 0.0f;
}

// one thread per group: FP64 sums over the members in CSR order (deterministic) of the
// caller-order gradients gline [4][n] = (gf, vdW, rad, Stark) -> g [4][G] (gf, rad, Stark, vdW)
__global__ void k_group_reduce(int64_t G, int64_t n, const int64_t *off, const int32_t *mem, const double *gline,
                               float *g) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= G) return;
    double sgf = 0.0, s6 = 0.0, sr = 0.0, s4 = 0.0;
    for (int64_t k = off[q]; k < off[q + 1]; ++k) {
        const int64_t l = mem[k];
        sgf += gline[l];
        s6 += gline[n + l];
        sr += gline[2 * n + l];
        s4 += gline[3 * n + l];
    }
    g[q] = (float)sgf;
    g[G + q] = (float)sr;
    g[2 * G + q] = (float)s4;
    g[3 * G + q] = (float)s6;
}

cudaError_t launch_group_gather(pz_ctx *c, const float *x, cudaStream_t s) {
    const int64_t n = c->nl_caller;
    if (n == 0) return cudaSuccess;
    k_group_gather<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, c->n_groups, c->d_grp_of, x, c->d_mdgf,
                                                              c->d_mdgrad, c->d_mdg4, c->d_mdg6);
    c->launches++;
    return cudaGetLastError();
}

cudaError_t launch_group_reduce(pz_ctx *c, float *g, cudaStream_t s) {
    const int64_t G = c->n_groups;
    if (G == 0) return cudaSuccess;
    k_group_reduce<<<(unsigned)((G + 255) / 256), 256, 0, s>>>(G, c->nl_caller, c->d_grp_off, c->d_grp_mem,
                                                              c->d_gline, g);
    c->launches++;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// probe: the FP32 Voigt exactly as the mixed kernels evaluate it
// (far region through the same pre-scaled polynomial with A = 1, a6 = 1)
// ---------------------------------------------------------------------------
__global__ void k_probe_voigt(const float *a, const float *v, int64_t n, float *H, float *dH) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    float aa = a[k], x = fabsf(v[k]);
    float a2 = aa * aa;
    float r2 = fmaf(x, x, a2);
    float h, dh;
    if (r2 >= kFar2) {
        float B1 = aa * kInvSqrtPiF;
        float t = rcp_approx(r2);
        float p = fmaf(t, 12.0f * a2 * a2 * B1, -15.0f * a2 * B1);
        p = fmaf(t, p, fmaf(-2.0f, a2, 3.75f) * B1);
        p = fmaf(t, p, 1.5f * B1);
        p = fmaf(t, p, B1);
        h = t * p;
        float C1 = kInvSqrtPiF;
        float q = fmaf(t, -120.0f * a2 * a2 * a2 * C1, 180.0f * a2 * a2 * C1);
        q = fmaf(t, q, a2 * fmaf(12.0f, a2, -67.5f) * C1);
        q = fmaf(t, q, fmaf(-12.0f, a2, 3.75f) * C1);
        q = fmaf(t, q, fmaf(-2.0f, a2, 1.5f) * C1);
        q = fmaf(t, q, C1);
        dh = t * q;
    } else {
        voigt_general<true>(x, aa, h, dh);
    }
    H[k] = h;
    if (dH) dH[k] = dh;
}

cudaError_t launch_probe_voigt(const float *a, const float *v, int64_t n, float *H, float *dH, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_probe_voigt<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, v, n, H, dH);
    return cudaGetLastError();
}

// Pipe-throughput probes (roofline denominators).  Every thread runs 8 independent
// dependency chains for `iters` rounds; the chains stay bounded (x -> 1/(x + 1), which
// no algebraic rewrite removes, for the reciprocal; a contraction toward a fixed point
// for the FMA) and one result per thread is stored so that the work is live.
//   kind 0: packed f32x2 FMA, 16 FP32 operations per thread per round;
//   kind 1: rcp.approx.ftz.f32 (plus one FP32 add), 8 MUFU operations per thread per round;
//   kind 2: FP64 FMA, 8 FP64 FMA operations per thread per round.
__global__ void k_probe_pipe(int kind, int iters, float *out) {
    const float seed = 1.0f + 1e-3f * (float)(threadIdx.x & 63);
    float r = 0.0f;
    if (kind == 0) {
        f2_t x[8];
        const f2_t m = f2_pack(0.999f, 0.998f), c = f2_pack(1e-3f, 2e-3f);
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = f2_pack(seed + k, seed - k);
        for (int it = 0; it < iters; ++it) {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = f2_fma(x[k], m, c);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float lo, hi;
            f2_unpack(x[k], lo, hi);
            r += lo + hi;
        }
    } else if (kind == 1) {
        float x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = seed + (float)k;
        for (int it = 0; it < iters; ++it) {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = rcp_approx(x[k] + 1.0f);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) r += x[k];
    } else {
        double x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = (double)seed + k;
        for (int it = 0; it < iters; ++it) {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = fma(x[k], 0.999, 1e-3);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) r += (float)x[k];
    }
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = r;
}

cudaError_t launch_probe_pipe(int kind, int iters, int blocks, float *out, cudaStream_t s) {
    k_probe_pipe<<<blocks, kProbeThreads, 0, s>>>(kind, iters, out);
    return cudaGetLastError();
}

// Bounded-wait probe: one CTA waits on an mbarrier phase that nothing completes, gives
// up after limit_ns and records the failure in the status word.
__global__ void k_probe_wait(uint64_t limit_ns, int32_t *status) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bool ok = mbar_wait(&bar, 0, limit_ns);
    if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicOr(status, kStatusWaitGaveUp);
}

cudaError_t launch_probe_wait(uint64_t limit_ns, int32_t *status, cudaStream_t s) {
    k_probe_wait<<<1, 32, 0, s>>>(limit_ns, status);
    return cudaGetLastError();
}

}  // namespace pz
