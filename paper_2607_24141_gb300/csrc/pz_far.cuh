// pz_far.cuh -- device code of the far-wing line kernels, shared by the translation units that
// instantiate them (pz_line.cu the forward, pz_line_bwd.cu and pz_line_bwd4.cu the reverse
// passes; they compile in parallel).  The mapping is described in pz_line.cu.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "pz_internal.h"

namespace pz {

// ---------------------------------------------------------------------------
// Mixed-precision kernels
// ---------------------------------------------------------------------------

struct LineInfo;
constexpr int kBoxClasses = 4;             // box separation classes (class 4: never, pz_box.cuh)

// Kernel arguments.  Line arrays are indexed by absolute line; the per-star tables
// and buffers point at star 0 and are advanced by star_view().
struct LineArgs {
    int64_t nlam, ld;
    int nd, W;
    float lnr, lam0cm;
    const float *ilf, *frac, *E, *lamcm, *grad, *g4, *g6, *Q;
    const int32_t *sp;
    const float *R, *invdv, *thr;                   // [ns][nd], [ns][nd], [ns][nslab] of the star
    const float *cut;                               // [ns][nslab] 36 K of the slab's widest layer
    const float *Ksd;                               // [ns][nd] K = 4^uexp/k^2 of the star
    int nslab;
    const float *beta_hi, *beta_lo, *ne, *npert, *c2T;   // [nd] of the star
    float *kline;                                   // forward output [nd][ld] of the star
    float *knear;                                   // near-core sums [nd][ld] of the star
    const float *Gt;                                // backward input [nd][ld] of the star
    double *gacc;                                   // backward output [2][nl]
    int64_t nl;
    // work queue: items (star, tile * ngroups + group, lo, hi), longest first
    const int4 *items;
    const int4 *fext;                               // pieces: (first slot, pieces, counter, piece)
    float4 *fpart;                                  // partial sums of split forward items [slot][DS][threads][2]
    int *fcnt;                                      // pieces finished per split forward item
    int n_items, ngroups;
    int *ctr;
    int64_t sstride, dstride, bstride, tstride;     // per-star strides of the tables above
    float uscale, kunscale;                         // 2^uexp and 4^-uexp: scaled offset u 2^uexp, 1/k^2 = K 4^-uexp
    float rj[4], rm1j[4];                           // r^-j and (r^-j - 1) 2^uexp, j = 0..3 (r = 1 + 1/R)
    const int32_t *star;                            // [nl] star of each line
    const LineInfo *finfo;                          // far-wing line records [ngroups][nl] (k_far_info)
    const uint32_t *keep;                           // centre-test mask [nl][kKeepWords] or NULL (all kept)
    // box expansions (pz_box.cuh): pairs they sum are skipped by the far-wing kernels
    int tDC, tDS;                                   // layers per depth group and slab of the line records
    int boxB, boxsh, s_lo, nbox;                    // of the star: box points (0: off) and log2, first source box, boxes
    const int4 *bgeo;                               // [S] the four above (NULL: off for every star)
    int64_t brow;                                   // row of bstart
    float shrink;                                   // |v| >= |Delta| ln r shrink k over a window
    const int *nmin;                                // [S][nslab][4] nearest offset of each class
    const int32_t *bstart;                          // [S][brow] first line of each quarter of a box
    uint32_t *wide;                                 // [4][nslab][wwords] lines of class >= 1..4
    int64_t wwords;
};

// Centre-test decision of the pair (l, d): kept unless a mask is set and its bit is clear.
__device__ __forceinline__ bool pair_kept(const uint32_t *keep, int64_t l, int d) {
    return !keep || ((keep[l * kKeepWords + (d >> 5)] >> (d & 31)) & 1u);
}

__device__ __forceinline__ LineArgs star_view(const LineArgs &g, int s) {
    LineArgs v = g;
    v.R += s * g.sstride;
    v.invdv += s * g.sstride;
    v.Ksd += s * g.sstride;
    v.thr += s * g.tstride;
    v.cut += s * g.tstride;
    v.beta_hi += s * g.dstride;
    v.beta_lo += s * g.dstride;
    v.ne += s * g.dstride;
    v.npert += s * g.dstride;
    v.c2T += s * g.dstride;
    v.kline += s * g.bstride;
    v.knear += s * g.bstride;
    v.Gt += s * g.bstride;
    if (g.bgeo) {
        const int4 q = __ldg(g.bgeo + s);
        v.boxB = q.x;
        v.boxsh = q.y;
        v.s_lo = q.z;
        v.nbox = q.w;
    }
    return v;
}

// Persistent work loop: every CTA takes the next item of the queue until it is empty.
template <class F>
__device__ __forceinline__ void for_each_item(const LineArgs &g, F &&f) {
    __shared__ int s_it;
    for (;;) {
        if (threadIdx.x == 0) s_it = atomicAdd(g.ctr, 1);
        __syncthreads();
        const int it = s_it;
        __syncthreads();
        if (it >= g.n_items) break;
        const int4 item = g.items[it];
        f(star_view(g, item.x), item.y / g.ngroups, item.y % g.ngroups, item.z, item.w, it);
    }
}

// Per-line scalars of the prefactors (one load per line, shared by its depths).
struct LineScalars {
    int sp;
    float E, Q, lamcm, g4, grad, g6;
};
__device__ __forceinline__ LineScalars load_line(const LineArgs &g, int64_t l) {
    LineScalars L;
    L.sp = g.sp[l];
    L.E = g.E[l];
    L.Q = g.Q[l];
    L.lamcm = g.lamcm[l];
    L.g4 = g.g4[l];
    L.grad = g.grad[l];
    L.g6 = g.g6[l];
    return L;
}

// Per-(line, depth) prefactors of the near-core kernels: k = c/dv_D, the damping parameter a and its square, the
// strength A, and (NG > 0) A times the parts of a that the damping families contribute: van der Waals
// gamma6 n_pert/(4 pi dnu_D) and (NG = 3) radiative gamma_rad and Stark gamma4 n_e alike (Eq. 10 scales
// one family by 10^delta, so d a / d delta = ln10 a_family).  Layers past the last one: no width, no strength.
// The damping products are rounded explicitly (no contraction), so that every kernel
// that classifies a cell by |v|^2 + a^2 -- the far-wing and near-core passes -- forms
// k and a^2 with identical roundings.
struct DepthParams {
    float k, a2, A, a, damp[3];
};
template <int NG>
__device__ __forceinline__ DepthParams depth_params(const LineArgs &g, const LineScalars &L, int d) {
    DepthParams q{0.0f, 1.0f, 0.0f, 0.0f, {0.0f, 0.0f, 0.0f}};
    if (d >= g.nd) return q;
    const int id = L.sp * g.nd + d;
    const float invdv = __ldg(g.invdv + id);
    const float bh = __ldg(g.beta_hi + d), bl = __ldg(g.beta_lo + d);
    const float p = L.E * bh;
    const float r = fmaf(L.E, bh, -p) + L.E * bl;      // E beta = p + r
    const float boltz = expf(-p) * (1.0f - r);
    const float lw = __fmul_rn(__fmul_rn(L.lamcm, invdv), (float)(1.0 / (4.0 * kPI)));
    const float g6n = __fmul_rn(L.g6, __ldg(g.npert + d));
    q.a = __fmul_rn(fmaf(L.g4, __ldg(g.ne + d), __fadd_rn(L.grad, g6n)), lw);
    q.a2 = __fmul_rn(q.a, q.a);
    q.k = __fmul_rn((float)kC, invdv);
    q.A = L.Q * __ldg(g.R + id) * boltz;
    if (NG > 0) q.damp[0] = q.A * g6n * lw;
    if (NG == 3) {
        q.damp[1] = q.A * L.grad * lw;
        q.damp[2] = q.A * __fmul_rn(L.g4, __ldg(g.ne + d)) * lw;
    }
    return q;
}

// index-space frequency offset u = lambda_l/lambda_i - 1 = expm1(Delta ln r)
__device__ __forceinline__ float offset_u(float delta, float lnr) {
    float y = delta * lnr;
    return fmaf(y * y, fmaf(y, 0.16666667f, 0.5f), y);
}

// Line record of the far-wing tables: centre, species and the per-slab reduced-form
// mask of the line's depth group.
struct alignas(16) LineInfo {
    float ilf, frac;
    int sp, amask;
};

// Box separation class of a line at slab w of its record's depth group, and the nearest box
// offset that the expansions take over for it.
__device__ __forceinline__ int box_class(int amask, int w) { return (amask >> (16 + 3 * w)) & 7; }

// The warp's view of the box expansions: nearest offsets of its slab by class, the tile's boxes
// and the lane's box.
struct BoxView {
    int n0, n1, n2, n3, ta, tb, tl;
};
__device__ __forceinline__ BoxView box_view(const LineArgs &g, int st, int slab, int t0, int T, int lam_thr) {
    BoxView v;
    const int4 n = *reinterpret_cast<const int4 *>(g.nmin + ((int64_t)st * g.nslab + slab) * 4);
    v.n0 = n.x;
    v.n1 = n.y;
    v.n2 = n.z;
    v.n3 = n.w;
    v.ta = t0 >> g.boxsh;
    v.tb = (t0 + T - 1) >> g.boxsh;
    v.tl = lam_thr >> g.boxsh;
    return v;
}
__device__ __forceinline__ int box_nmin(const BoxView &v, int cls) {
    return cls == 0 ? v.n0 : cls == 1 ? v.n1 : cls == 2 ? v.n2 : cls == 3 ? v.n3 : kBoxNever;
}
// The lane's points are summed directly for this line (not by the expansions).
__device__ __forceinline__ bool box_near(const LineArgs &g, const BoxView &v, const LineInfo &info, int w) {
    return abs(((int)info.ilf >> g.boxsh) - v.tl) < box_nmin(v, box_class(info.amask, w));
}


// ---- packed FP32 pairs ------------------------------------------------------
// The far-wing kernels evaluate two depths of one (line, lambda) cell with one
// instruction: a register pair {value at depth d, value at depth d + 1} and the
// f32x2 forms of mul and fma (each half rounded exactly as the scalar op).  This
// halves the FP32 issue slots of the inner loop; the two reciprocals stay scalar.
typedef unsigned long long f2_t;

__device__ __forceinline__ f2_t f2_pack(float lo, float hi) {
    f2_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(f2_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2_t f2_mul(f2_t a, f2_t b) {
    f2_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2_t f2_fma(f2_t a, f2_t b, f2_t c) {
    f2_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// reciprocal of both halves (rcp.approx.ftz, as rcp_approx)
__device__ __forceinline__ f2_t f2_rcp(f2_t a) {
    f2_t r;
    asm("{\n\t.reg .f32 lo, hi;\n\tmov.b64 {lo, hi}, %1;\n\trcp.approx.ftz.f32 lo, lo;\n\t"
        "rcp.approx.ftz.f32 hi, hi;\n\tmov.b64 %0, {lo, hi};\n\t}"
        : "=l"(r) : "l"(a));
    return r;
}
__device__ __forceinline__ f2_t f2_splat(float v) { return f2_pack(v, v); }
__device__ __forceinline__ float f2_lo(f2_t v) {
    float lo, hi;
    f2_unpack(v, lo, hi);
    return lo;
}
__device__ __forceinline__ float f2_hi(f2_t v) {
    float lo, hi;
    f2_unpack(v, lo, hi);
    return hi;
}

// ---- far-wing prefactors ------------------------------------------------------
// A far-wing CTA stages LC lines at a time.  For each line of the chunk and each of
// the (DC/2) depth pairs of its group it forms NQ quads, quad q holding
// {p_2q(d), p_2q(d + 1), p_2q+1(d), p_2q+1(d + 1)} (one 16-byte shared-memory load
// returns the packed depth pairs of two parameters):
//   forward  (NQ = 5): (K, a^2) (B1 K, B2' K^2) (B3' K^3, B4' K^4) .. (B7' K^7, B8' K^8)
//   backward (NQ = 9): the same, then (C1 K, C2' K^2) .. (C7' K^7, C8' K^8)
//   backward, all damping families (NQ = 11): C without its family factor gamma n, then the three
//   families' factors (van der Waals, radiative) (Stark, -)
// with k = c/dv_D, K = 4^uexp/k^2 (the power of four brings the largest K of the context to 1/4..1
// and keeps every product of the prefactors, K^8 among them, and of the offsets inside FP32), B2' = B2 - B1 a^2
// = B1 (1.5 - a^2) and C2' = C2 - C1 a^2 = C1 (1.5 - 3a^2).  The far kernels take the
// squared offsets scaled alike, U = 4^uexp u^2, so that with s = 1/U
//   reduced form:  H sqrt(pi)/A = (B1 K) s + (B2' K^2) s^2   (p = K s exactly, see below)
//   full form:     r = 1/(U + a^2 K) and t = 1/|z|^2 = K r, so B1 t (...) = (B1 K) r (...)
// and the masked lines recover B1 = (B1 K) k^2 4^-uexp (and C1 alike) per depth pair.
// Each warp stages the quads of its own slab, par[li][pair][q] in its part of shared
// memory; the polynomial in t of the large-damping lines (B3..B5, C3..C6) follows from a^2
// and B1 K (C1 K) in registers.  Lane li computes line li's quads from the line data and the
// star's per-(species, depth) tables (Eqs. 4-5, with the roundings of depth_params), so
// no per-(line, depth) array exists in device memory: the quads are recomputed for each
// tile the line's window reaches.  The only per-line device array of the far kernels is
// the 16-byte line record of each depth group (k_far_info).
constexpr int kPolyN = 8;          // terms of the series in p = K s
constexpr int kNQF = 1 + kPolyN / 2, kNQB = 1 + kPolyN, kNQB4 = kNQB + 2;
constexpr int kBwdBatch = 16;   // lines per transposed partial-sum batch of the far-wing backward (2 lanes per line)

// Reduced far-wing form.  Far from the core the polynomial in t = 1/|z|^2 is cut
// after its t^2 term: H sqrt(pi)/(A a) = t (1 + 1.5 t) and, for dH/da, C1 t (1 +
// (1.5 - 2a^2) t).  With |v| >= 100 (t <= 1e-4) and a^2 <= 1.5 (s = a^2 t <= 1.5e-4)
// the dropped terms, (3.75 t^2 + 2 s t + 15 s t^2 + 12 s^2 t^2) relative for H, stay
// below 7e-8 (about one FP32 rounding) and below 2.2e-7 for dH/da.
// In the same region t is expanded about p = 1/(u k)^2 = (1/U) K:
// t = p/(1 + a^2 p) = p - a^2 p^2 + O((a^2 p)^2 p), so that
//   H sqrt(pi)/A = B1 p + B2' p^2 = (B1 K) s + (B2' K^2) s^2,   s = 1/U,
// and dH/da sqrt(pi)/(A a6) = (C1 K) s + (C2' K^2) s^2, with B2' = B1 (1.5 - a^2),
// C2' = C1 (1.5 - 3a^2); the further dropped terms, (a^2 p)^2 and 3 a^2 p^2 relative,
// stay below 5e-8.  s and s^2 depend on the line and the point only, so one MUFU
// reciprocal serves all the depths of a warp, and the forward adds two products per
// cell.  In the backward the sums over the cells of one depth factor:
//   sum_i G_i [(B1 K) s_i + (B2' K^2) s_i^2] = (B1 K) X1 + (B2' K^2) X2,
//   X1 = sum_i G_i s_i,  X2 = sum_i G_i s_i^2,
// and X1, X2 serve both gradients (the C coefficients multiply the same sums).
constexpr float kFast2V = 5.0f;      // distance threshold factor: |v| >= 5 x 20
// The same expansion to N terms, H sqrt(pi)/A = sum_n B1 beta_n(a^2) (K s)^(n+1) and dH/da
// sqrt(pi)/(A a6) = sum_n C1 gamma_n(a^2) (K s)^(n+1), reaches the nearer cells: with a^2 <= 1.5 the
// dropped terms stay below 2.6e-8 (H) and 4.6e-8 (dH/da) relative with N = 3 at |v| >= 30, below
// 3e-9 with N = 4 at |v| >= 20 and below 6.3e-8 (dH/da: 1.2e-7 of its scale 1/v^2) with N = 8 at |v| >= 6.
// Eight multiply-adds per cell and no per-cell branch (one cut in U serves all layers of a slab, so the
// points of the core have s = 0): the mid wing 6 <= |v| < 20, which the
// near-core kernels summed cell by cell at about 140 instructions each, and the masked far cells
// beside it (two reciprocals and a polynomial in t per depth pair) are one sweep of the tile.
// Measured on 2e5 lines x 37,550 points: far + near-core forward 6.9 -> 4.3 ms, reverse 9.9 ->
// 6.8 ms.
constexpr float kCoreV = 0.3f;       // distance threshold factor: |v| >= 0.3 x 20 = 6
constexpr float kFast3V = 1.5f;      // distance threshold factor: |v| >= 1.5 x 20
constexpr float kFast2A2 = 1.5f;     // a^2 bound
// Larger damping, a^2 <= 44 (a <= 20/3): the eight terms hold where |v| >= 20, so |v| >= 3a (H below
// 3.6e-9, dH/da below 7e-8 of its scale); those lines keep the whole near zone, U < 400 K of the slab's
// widest layer, in the near-core kernels.  They are few in giants but a third of the deepest layers'
// lines in dwarfs, where the polynomial in t (two reciprocals per depth pair and cell, and a mask)
// took most of the far-wing time: two-star fit on 10^5 lines, far
// forward 2.45 -> 2.2 ms, reverse 3.8 -> 3.3 ms (the fill by all lanes included).
constexpr float kWideA2 = 44.0f;
constexpr float kWideCut = 400.0f / 36.0f;   // its cut over the core's

// c_n = x K^n beta_n(a^2) (D: gamma_n(a^2)), n = 0..7: beta_n = sum_k (-1)^k c_(n-k) binom(2n + 1,
// 2k + 1) a^2k with c_m = (2m - 1)!!/2^m, from the expansion of Re w(v + i a) about 1/v, and gamma_n =
// sum_k (2k + 1) (..) a^2k, its derivative.
template <bool D>
__device__ __forceinline__ void poly_coeffs(float x, float K, float s, float (&c)[kPolyN]) {
#define PZ_Q(k, v) ((D ? 2.0f * (k) + 1.0f : 1.0f) * (v))
    c[0] = x;
    x *= K;
    c[1] = x * fmaf(s, PZ_Q(1, -1.0f), PZ_Q(0, 1.5f));
    x *= K;
    c[2] = x * fmaf(s, fmaf(s, PZ_Q(2, 1.0f), PZ_Q(1, -5.0f)), PZ_Q(0, 3.75f));
    x *= K;
    c[3] = x * fmaf(s, fmaf(s, fmaf(s, PZ_Q(3, -1.0f), PZ_Q(2, 10.5f)), PZ_Q(1, -26.25f)), PZ_Q(0, 13.125f));
    x *= K;
    c[4] = x * fmaf(s, fmaf(s, fmaf(s, fmaf(s, PZ_Q(4, 1.0f), PZ_Q(3, -18.0f)), PZ_Q(2, 94.5f)), PZ_Q(1, -157.5f)),
                    PZ_Q(0, 59.0625f));
    x *= K;
    c[5] = x * fmaf(s, fmaf(s, fmaf(s, fmaf(s, fmaf(s, PZ_Q(5, -1.0f), PZ_Q(4, 27.5f)), PZ_Q(3, -247.5f)),
                                    PZ_Q(2, 866.25f)), PZ_Q(1, -1082.8125f)), PZ_Q(0, 324.84375f));
    x *= K;
    c[6] = x * fmaf(s, fmaf(s, fmaf(s, fmaf(s, fmaf(s, fmaf(s, PZ_Q(6, 1.0f), PZ_Q(5, -39.0f)), PZ_Q(4, 536.25f)),
                                            PZ_Q(3, -3217.5f)), PZ_Q(2, 8445.9375f)), PZ_Q(1, -8445.9375f)),
                    PZ_Q(0, 2111.484375f));
    x *= K;
    c[7] = x * fmaf(s, fmaf(s, fmaf(s, fmaf(s, fmaf(s, fmaf(s, fmaf(s, PZ_Q(7, -1.0f), PZ_Q(6, 52.5f)),
                                                            PZ_Q(5, -1023.75f)), PZ_Q(4, 9384.375f)),
                                            PZ_Q(3, -42229.6875f)), PZ_Q(2, 88682.34375f)), PZ_Q(1, -73901.953125f)),
                    PZ_Q(0, 15836.1328125f));
#undef PZ_Q
}

// Prefactors of line l at layer d (one half of a depth pair), with the roundings of
// depth_params for k and a^2 (the cells' near / far classification depends on them):
// K = 4^uexp/k^2, a^2, the series coefficients c (B1 K, B2' K^2, ..) and (NQ = kNQB) e (C1 K, C2' K^2, ..).  dc holds the layer's
// {beta_hi, beta_lo, n_e, n_pert}.  Layers past the last one get K = 0, a^2 = 1 and zero
// coefficients, pairs rejected by the centre test zero coefficients.
template <int NQ>
__device__ __forceinline__ void far_depth_prefactors(const LineArgs &g, const LineScalars &L, int64_t l, int d,
                                                     const float4 dc, float &K, float &a2, float (&c)[kPolyN],
                                                     float (&e)[kPolyN], float (&gb)[3]) {
    if (d >= g.nd) {
        K = 0.0f;
        a2 = 1.0f;
#pragma unroll
        for (int n = 0; n < kPolyN; ++n) c[n] = e[n] = 0.0f;
        gb[0] = gb[1] = gb[2] = 0.0f;
        return;
    }
    const int id = L.sp * g.nd + d;
    const float invdv = __ldg(g.invdv + id);
    const float p = L.E * dc.x;
    const float r = fmaf(L.E, dc.x, -p) + L.E * dc.y;      // E beta = p + r
    const float boltz = expf(-p) * (1.0f - r);
    const float A = L.Q * __ldg(g.R + id) * boltz;
    const float lw = __fmul_rn(__fmul_rn(L.lamcm, invdv), (float)(1.0 / (4.0 * kPI)));
    const float g6n = __fmul_rn(L.g6, dc.w);
    const float a = __fmul_rn(fmaf(L.g4, dc.z, __fadd_rn(L.grad, g6n)), lw);
    a2 = __fmul_rn(a, a);
    K = __ldg(g.Ksd + id);
    const bool kept = pair_kept(g.keep, l, d);
    poly_coeffs<false>(kept ? A * a * kInvSqrtPiF * K : 0.0f, K, a2, c);
    if (NQ == kNQB) poly_coeffs<true>(kept ? A * g6n * lw * kInvSqrtPiF * K : 0.0f, K, a2, e);
    if (NQ == kNQB4) {
        poly_coeffs<true>(kept ? A * lw * kInvSqrtPiF * K : 0.0f, K, a2, e);
        gb[0] = g6n;
        gb[1] = L.grad;
        gb[2] = __fmul_rn(L.g4, dc.z);
    }
}

// Per-warp staging of a chunk of lines.  Each warp keeps, in its own part of shared
// memory, the layer constants of its slab (dc: DS x {beta_hi, beta_lo, n_e, n_pert}),
// and for the chunk's lines their records and the prefactor quads of its DP depth pairs
// (par: [LC][DP][NQ]).  Lanes li and li + 16 fill line li (li + 16, ...); a
// warp barrier publishes the chunk, and the next fill waits on a warp barrier so that
// no lane still reads the previous chunk.  No CTA-wide barrier is involved.
struct WarpStage {
    float4 *dc;          // [DS]
    float4 *par;         // [LC][DP * NQ]
    LineInfo *info;      // [LC]
    int *idx;            // [LC] line of each staged slot (forward: gathered by warp_gather)
};

__host__ __device__ constexpr size_t warp_stage_quads(int LC, int DS, int NQ) {
    return (size_t)DS + (size_t)LC * (DS / 2) * NQ + (size_t)LC + ((size_t)LC + 3) / 4;
}
__device__ __forceinline__ WarpStage make_stage(float4 *mine, int LC, int DS, int NQ) {
    LineInfo *info = reinterpret_cast<LineInfo *>(mine + DS + (size_t)LC * (DS / 2) * NQ);
    return WarpStage{mine, mine + DS, info, reinterpret_cast<int *>(info + LC)};
}

template <int DS>
__device__ __forceinline__ void warp_stage_depths(const LineArgs &g, const WarpStage &ws, int dfirst, int lane) {
    __syncwarp();
    if (lane < DS) {
        const int d = dfirst + lane;
        ws.dc[lane] = d < g.nd ? make_float4(__ldg(g.beta_hi + d), __ldg(g.beta_lo + d), __ldg(g.ne + d),
                                              __ldg(g.npert + d))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncwarp();
}

// The forward's next chunk: up to LC lines from cur on that slab w has to sweep (all lines
// without the centre test; with it, those with a layer of the slab kept), their indices in
// ws.idx in line order.  Returns the count and leaves cur after the last line looked at.
__device__ __forceinline__ int warp_gather(const WarpStage &ws, const LineInfo *ginfo, int &cur, int hi, int LC,
                                           int w, int lane) {
    int count = 0;
    __syncwarp();
    while (count < LC && cur < hi) {
        const int l = cur + lane;
        const bool need = l < hi && !((ginfo[l].amask >> (8 + w)) & 1);
        const unsigned m = __ballot_sync(0xffffffffu, need);
        const int n = __popc(m);
        const int take = min(n, LC - count);
        const int slot = count + __popc(m & ((1u << lane) - 1u));
        if (need && slot < LC) ws.idx[slot] = l;
        cur += take < n ? __fns(m, 0, take) + 1 : 32;   // after the last line taken
        count += take;
    }
    __syncwarp();
    return count;
}

// Up to LC lines of [cur, hi) whose bit is set in words (one bit per line), in line order, into
// ws.idx; returns the count and leaves cur after the last line looked at.
__device__ __forceinline__ int warp_gather_bits(const WarpStage &ws, const uint32_t *words, int &cur, int hi, int LC,
                                                int lane) {
    int count = 0;
    __syncwarp();
    while (count < LC && cur < hi) {
        const int w0 = cur >> 5, first = (w0 + lane) << 5;
        uint32_t m = first < hi ? words[w0 + lane] : 0u;
        if (first < cur) m &= ~0u << (cur - first);            // (lane 0 alone holds lines before cur)
        if (first < hi && hi - first < 32) m &= (1u << (hi - first)) - 1u;
        const int n = __popc(m);
        int inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const int total = __shfl_sync(0xffffffffu, inc, 31);
        int slot = count + inc - n;
        for (; m && slot < LC; ++slot) {
            ws.idx[slot] = first + __ffs(m) - 1;
            m &= m - 1u;
        }
        __syncwarp();
        if (count + total <= LC) {
            count += total;
            cur = (w0 + 32) << 5;
        } else {
            count = LC;
            cur = ws.idx[LC - 1] + 1;
        }
    }
    __syncwarp();
    return count;
}

// The lines beyond the tile's near boxes that warp's slab still sums directly, ring by ring:
// between the nearest offsets of class c - 1 (n0g: that of the whole group) and of class c, the
// lines of class >= c; beyond class 3, the lines no class takes.  f(lines) runs for every gathered
// chunk.  Piece q of P takes its share of every ring.
template <class F>
__device__ __forceinline__ void box_rings(const LineArgs &g, const BoxView &v, int st, int slab, int n0g, int t0, int T,
                                          int q, int P, const WarpStage &ws, int LC, int lane, F &&f) {
    if (!g.boxB || n0g >= kBoxNever) return;
    const int32_t *bs = g.bstart + (int64_t)st * g.brow;
    int below = n0g;
    for (int c = 1; c <= kBoxClasses; ++c) {
        const int n = box_nmin(v, c);
        const int upto = max(n, below);
        const uint32_t *words = g.wide + ((int64_t)(c - 1) * g.nslab + slab) * g.wwords;
        for (int side = 0; side < 2 && upto > below; ++side) {
            // boxes of the ring, clipped to those the windows reach
            int s0 = side ? v.ta - upto + 1 : v.tb + below;
            int s1 = side ? v.ta - below : v.tb + upto - 1;
            s0 = max(max(s0, (t0 - g.W) >> g.boxsh), g.s_lo);
            s1 = min(min(s1, (t0 + T - 1 + g.W) >> g.boxsh), g.s_lo + g.nbox - 1);
            if (s0 > s1) continue;
            const int a = bs[kBoxQuarters * (s0 - g.s_lo)], b = bs[kBoxQuarters * (s1 - g.s_lo + 1)];
            int cur = a + (int)((int64_t)(b - a) * q / P);
            const int hi = a + (int)((int64_t)(b - a) * (q + 1) / P);
            while (cur < hi) {
                const int nl = warp_gather_bits(ws, words, cur, hi, LC, lane);
                if (nl > 0) f(nl);
            }
        }
        below = upto;
    }
}

// Nearest offset of class 0 over the slabs of a depth group (the group's near boxes).
__device__ __forceinline__ int box_group_n0(const LineArgs &g, int st, int group, int GW) {
    int n = 0;
    for (int w = 0; w < GW; ++w) n = max(n, g.nmin[((int64_t)st * g.nslab + group * GW + w) * 4]);
    return n;
}

template <int NQ, int DS>
__device__ __forceinline__ void warp_fill(const LineArgs &g, const WarpStage &ws, const LineInfo *ginfo,
                                          int64_t first, int nl, int dfirst, int lane, bool listed = false) {
    constexpr int DP = DS / 2;
    __syncwarp();
    // lane = (line, half of the slab's layers): a chunk of 16 lines occupies the whole warp
    const int half = lane >> 4;
    for (int li = lane & 15; li < nl; li += 16) {
        const int64_t l = listed ? (int64_t)ws.idx[li] : first + li;
        if (half == 0) ws.info[li] = ginfo[l];
        const LineScalars L = load_line(g, l);
        float *dst = reinterpret_cast<float *>(ws.par + (size_t)li * DP * NQ);
#pragma unroll
        for (int q = 0; q < DP; ++q) {
            const int dd = half * DP + q;                 // layer of the slab
            float K, a2, c[kPolyN], e[kPolyN], gb[3];
            far_depth_prefactors<NQ>(g, L, l, dfirst + dd, ws.dc[dd], K, a2, c, e, gb);
            float *o = dst + (dd >> 1) * NQ * 4 + (dd & 1);
            o[0] = K;
            o[2] = a2;
#pragma unroll
            for (int n = 0; n < kPolyN; ++n) {
                o[4 + 2 * n] = c[n];
                if (NQ >= kNQB) o[4 + 2 * (kPolyN + n)] = e[n];
            }
            if (NQ == kNQB4) {
                o[4 * kNQB] = gb[0];
                o[4 * kNQB + 2] = gb[1];
                o[4 * kNQB + 4] = gb[2];
            }
        }
    }
    __syncwarp();
}

// How a warp sums a line over its slab and tile.
enum FarForm {
    kFormSkip = 0,      // the centre test rejects every layer, or the box expansions sum every pair
    kFormTwo,           // every cell |v| >= 100: two terms
    kFormThree,         // |v| >= 30: three
    kFormFour,          // |v| >= 20: four
    kFormEight,         // eight, the points with U < cut (x^2 < 36 at the slab's widest layer) left to the
                        // near-core kernels at every layer of the slab
    kFormWide,          // kFast2A2 < a^2 <= kWideA2 somewhere in the slab: eight, the points with U < kWideCut cut
                        // left to the near-core kernels
    kFormLarge,         // a^2 > kWideA2 somewhere in the slab, |v| >= 20, the window covers the tile: polynomial in t
    kFormLargeMask,     // a^2 > kWideA2: the cells with |z| >= 20 inside the window, the others left to the
                        // near-core kernels
    kFormFull = 8       // bit: the window covers the tile
};
__device__ __forceinline__ int far_form(const LineArgs &g, const LineInfo &info, float t0f, float tendf, int slab, int w,
                                        const BoxView &bv) {
    const float dlo = info.ilf - t0f + info.frac;      // x_l - t0
    const float dhi = info.ilf - tendf + info.frac;    // x_l - (t0 + T - 1)
    const float dmin = fmaxf(0.0f, fmaxf(-dlo, dhi));
    const bool full = (info.ilf - (float)g.W <= t0f) && (info.ilf + (float)g.W >= tendf);
    if ((info.amask >> (8 + w)) & 1) return kFormSkip;
    const int sbox = (int)info.ilf >> g.boxsh, nb = box_nmin(bv, box_class(info.amask, w));
    if (sbox <= bv.ta - nb || sbox >= bv.tb + nb) return kFormSkip;
    const float thr = __ldg(g.thr + info.sp * g.nslab + slab);   // 20 Doppler widths of the slab's widest layer
    if (!((info.amask >> w) & 1)) {
        if ((info.amask >> (4 + w)) & 1) return kFormWide | (full ? kFormFull : 0);
        return full && dmin >= thr ? kFormLarge : kFormLargeMask;
    }
    const int f = dmin >= kFast2V * thr ? kFormTwo
                  : dmin >= kFast3V * thr ? kFormThree
                  : dmin >= thr ? kFormFour
                                : kFormEight;
    return f | (full ? kFormFull : 0);
}

// Points with U below it belong to the near-core kernels (series forms).
__device__ __forceinline__ float far_cut(const LineArgs &g, int form, int sp, int slab) {
    if ((form & 7) < kFormEight) return 0.0f;
    const float cut = __ldg(g.cut + sp * g.nslab + slab);
    return (form & 7) == kFormWide ? kWideCut * cut : cut;
}

// k = c/dv_D of the warp's depth pairs, rounded exactly as depth_params forms it, for the
// masked lines, whose cells are classified near / far with the near-core kernels' own
// arithmetic (x = u k, |z|^2 = x^2 + a^2).  Layers past the last one get 0.
template <int DP>
__device__ __forceinline__ void far_kpairs(const LineArgs &g, int sp, int dfirst, f2_t (&kp)[DP]) {
#pragma unroll
    for (int dp = 0; dp < DP; ++dp) {
        const int da = dfirst + 2 * dp, db = da + 1;
        const float ka = da < g.nd ? __fmul_rn((float)kC, __ldg(g.invdv + sp * g.nd + da)) : 0.0f;
        const float kb = db < g.nd ? __fmul_rn((float)kC, __ldg(g.invdv + sp * g.nd + db)) : 0.0f;
        kp[dp] = f2_pack(ka, kb);
    }
}

// Compensated-sum slots of depth dd of thread tid: the (hi, lo) quads of its J points, hi
// at quad 2 dd nthr + tid and lo at quad (2 dd + 1) nthr + tid, so that the threads of a
// warp touch consecutive quads (16-byte accesses without bank conflicts).  They live in
// shared memory and are touched once per line chunk.
__device__ __forceinline__ float4 *comp_hi(float *s_comp, int dd, int tid, int nthr) {
    return reinterpret_cast<float4 *>(s_comp) + (size_t)(2 * dd) * nthr + tid;
}
__device__ __forceinline__ float4 *comp_lo(float *s_comp, int dd, int tid, int nthr) {
    return reinterpret_cast<float4 *>(s_comp) + (size_t)(2 * dd + 1) * nthr + tid;
}

// Coefficients of the polynomial in t from a^2 and B1 (B2 = 1.5 B1):
// B3 = (3.75 - 2a^2) B1, B4 = -15 a^2 B1, B5 = 12 a^4 B1.
__device__ __forceinline__ void far_b345(f2_t a2, f2_t B1, f2_t &B3, f2_t &B4, f2_t &B5) {
    B3 = f2_mul(f2_fma(a2, f2_splat(-2.0f), f2_splat(3.75f)), B1);
    B4 = f2_mul(f2_mul(a2, f2_splat(-15.0f)), B1);
    B5 = f2_mul(f2_mul(f2_mul(a2, f2_splat(12.0f)), a2), B1);
}
// C3 = (3.75 - 12 a^2) C1, C4 = a^2 (12 a^2 - 67.5) C1, C5 = 180 a^4 C1, C6 = -120 a^6 C1.
__device__ __forceinline__ void far_c3456(f2_t a2, f2_t C1, f2_t &C3, f2_t &C4, f2_t &C5, f2_t &C6) {
    C3 = f2_mul(f2_fma(a2, f2_splat(-12.0f), f2_splat(3.75f)), C1);
    C4 = f2_mul(f2_mul(a2, f2_fma(a2, f2_splat(12.0f), f2_splat(-67.5f))), C1);
    const f2_t a4 = f2_mul(a2, a2);
    C5 = f2_mul(f2_mul(a4, f2_splat(180.0f)), C1);
    C6 = f2_mul(f2_mul(f2_mul(a4, f2_splat(-120.0f)), a2), C1);
}

// Reciprocals s_j = 1/U_j of the squared scaled offsets of one line at the thread's J
// points (and their squares), for the reduced forms: offsets from the first point's,
// u_j = u_0 r^-j + (r^-j - 1) scaled by 2^uexp; points outside the line's window get
// s = 0 unless the window covers the tile (full), points of a lane whose box is left to the
// box expansions (not near) too.
template <int J>
__device__ __forceinline__ void far_scaled_u2(const LineArgs &g, const LineInfo &info, float lamf, float (&U)[J]) {
    // scalar chain: the offsets depend on the line and the point only, not on the depth
    const float u0 = offset_u((info.ilf - lamf) + info.frac, g.lnr) * g.uscale;
    U[0] = u0 * u0;
#pragma unroll
    for (int j = 1; j < J; ++j) {
        const float u = fmaf(u0, g.rj[j], g.rm1j[j]);
        U[j] = u * u;
    }
}

template <int J>
__device__ __forceinline__ void far_reduced_s(const LineArgs &g, const LineInfo &info, bool full, bool near,
                                              float lamf, int lam_thr, f2_t (&sp)[J], f2_t (&sq)[J]) {
    float U[J];
    far_scaled_u2<J>(g, info, lamf, U);
    if (full || !near) {
#pragma unroll
        for (int j = 0; j < J; ++j) sp[j] = f2_splat(near ? rcp_approx(U[j]) : 0.0f);
    } else {
        const int il = (int)info.ilf;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int di = lam_thr + j - il;
            sp[j] = f2_splat(di >= -g.W && di <= g.W ? rcp_approx(U[j]) : 0.0f);
        }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) sq[j] = f2_mul(sp[j], sp[j]);
}

// U = 4^uexp u^2 of one point by itself (il_i = i_l - i, exact).  Within 20 Doppler widths of a line the
// chain of far_scaled_u2 would carry the rounding of the lane's first point to points nearer the line
// (on grids of R = 10^4, where a core is one point wide, F was 1.6e-8 from FP64 and is 1.1e-8).
__device__ __forceinline__ float point_u2(const LineArgs &g, float il_i, float frac) {
    const float u = offset_u(il_i + frac, g.lnr) * g.uscale;
    return u * u;
}
// The same for two neighbouring points i, i + 1 (the packed operations round each half as the scalar ones).
__device__ __forceinline__ f2_t point_u2(const LineArgs &g, const LineInfo &info, float lam) {
    const f2_t d = f2_fma(f2_pack(lam, lam + 1.0f), f2_splat(-1.0f), f2_splat(info.ilf));
    const f2_t y = f2_mul(f2_fma(d, f2_splat(1.0f), f2_splat(info.frac)), f2_splat(g.lnr));
    const f2_t u = f2_mul(f2_fma(f2_mul(y, y), f2_fma(y, f2_splat(0.16666667f), f2_splat(0.5f)), y), f2_splat(g.uscale));
    return f2_mul(u, u);
}

// Reciprocals s_j = 1/U_j at the thread's points for the series forms: zero outside the window,
// below cut (the points left to the near-core kernels) and for lanes left to the box expansions.
template <int J>
__device__ __forceinline__ void far_series_s(const LineArgs &g, const LineInfo &info, int form, bool near, float lamf,
                                             int lam_thr, float cut, f2_t (&sp)[J]) {
    const bool full = form & kFormFull;
    float U[J];
    if ((form & 7) >= kFormEight) {
#pragma unroll
        for (int j = 0; j < J; j += 2) f2_unpack(point_u2(g, info, lamf + (float)j), U[j], U[j + 1]);
    } else {
        far_scaled_u2<J>(g, info, lamf, U);
    }
    const int di0 = lam_thr - (int)info.ilf;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const bool in = near && U[j] >= cut && (full || (di0 + j >= -g.W && di0 + j <= g.W));
        sp[j] = f2_splat(in ? rcp_approx(U[j]) : 0.0f);
    }
}

// acc += sum_n c_n s^(n+1) over the line's cells (N terms).
template <int J, int DP, int N>
__device__ __forceinline__ void far_fwd_series(const ulonglong2 *par, const f2_t (&sp)[J], f2_t (&acc)[DP][J]) {
#pragma unroll
    for (int dp = 0; dp < DP; ++dp) {
        const ulonglong2 *q = par + kNQF * dp;
        f2_t c[N + 1];
#pragma unroll
        for (int n = 0; n < N; n += 2) {
            const ulonglong2 v = q[1 + n / 2];
            c[n] = v.x;
            c[n + 1] = v.y;
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            f2_t h = c[N - 1];
#pragma unroll
            for (int n = N - 2; n >= 0; --n) h = f2_fma(sp[j], h, c[n]);
            acc[dp][j] = f2_fma(sp[j], h, acc[dp][j]);
        }
    }
}

// The reverse pass's sums of a line: S[0] for the strength, S[1] for van der Waals damping, and
// with FOUR S[2], S[3] for radiative and Stark damping.  Y: the damping sum of one depth pair, which
// FOUR shares among the families (without FOUR the family factor is in the coefficients and Y is S[1]).
template <bool FOUR>
struct FarSums {
    f2_t S[FOUR ? 4 : 2];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int k = 0; k < (FOUR ? 4 : 2); ++k) S[k] = 0ull;
    }
    __device__ __forceinline__ f2_t open() const { return FOUR ? 0ull : S[1]; }
    __device__ __forceinline__ void close(f2_t Y, const ulonglong2 *q) {   // q: the depth pair's quads
        if (FOUR) {
            const ulonglong2 g0 = q[kNQB], g1 = q[kNQB + 1];
            S[1] = f2_fma(g0.x, Y, S[1]);
            S[2 % (FOUR ? 4 : 2)] = f2_fma(g0.y, Y, S[2 % (FOUR ? 4 : 2)]);
            S[3 % (FOUR ? 4 : 2)] = f2_fma(g1.x, Y, S[3 % (FOUR ? 4 : 2)]);
        } else {
            S[1] = Y;
        }
    }
};
template <bool FOUR>
__host__ __device__ constexpr int far_nqb() {
    return FOUR ? kNQB4 : kNQB;
}

// S[0] += sum_n c_n X_n, Y += sum_n e_n X_n with X_n = sum_j G s_j^(n+1) per depth pair: one
// multiply-add per cell and term serves every gradient.
template <int J, int DP, int N, bool FOUR>
__device__ __forceinline__ void far_bwd_series(const ulonglong2 *par, const f2_t (&sp)[J], const f2_t (&gv)[DP][J],
                                               FarSums<FOUR> &R) {
    constexpr int NQ = far_nqb<FOUR>();
    constexpr int G = DP < 3 ? DP : 3;        // depth pairs taken together (registers)
#pragma unroll
    for (int d0 = 0; d0 < DP; d0 += G) {
        f2_t X[G][N];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            f2_t pw = sp[j];
#pragma unroll
            for (int n = 0; n < N; ++n) {
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    if (d0 + i >= DP) break;
                    X[i][n] = j == 0 ? f2_mul(gv[d0 + i][j], pw) : f2_fma(gv[d0 + i][j], pw, X[i][n]);
                }
                if (n + 1 < N) pw = f2_mul(pw, sp[j]);
            }
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
            if (d0 + i >= DP) break;
            const ulonglong2 *q = par + NQ * (d0 + i);
            f2_t Y = R.open();
#pragma unroll
            for (int n = 0; n < N; ++n) {
                const ulonglong2 c = q[1 + n / 2], e = q[1 + (kPolyN + n) / 2];
                R.S[0] = f2_fma((n & 1) ? c.y : c.x, X[i][n], R.S[0]);
                Y = f2_fma((n & 1) ? e.y : e.x, X[i][n], Y);
            }
            R.close(Y, q);
        }
    }
}

// Far-wing kernel (forward).  The cells of a line outside its core (far_form) and nearer than the box
// expansions' pairs are summed here; the cores' cells and the boxes' field are in knear already, which
// this kernel adds before applying stim.
template <int J, int DS, bool GATHER>
__device__ __forceinline__ void far_fwd_item(const LineArgs &g, const int st, const int tile, const int group,
                                             const int lo, const int hi, const int GW, const int LC,
                                             const WarpStage &ws, float *s_comp, const int4 ext) {
    static_assert(J == 2 || J == 4, "J must be 2 or 4");
    static_assert(DS % 2 == 0, "DS must be even (depth pairs)");
    constexpr int DP = DS / 2;          // depth pairs per warp
    constexpr int NQ = kNQF;
    const int T = 32 * J;
    const int DC = GW * DS;
    const int nthr = blockDim.x;
    const LineInfo *ginfo = g.finfo + (int64_t)group * g.nl;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d0 = group * DC;
    const int slab = group * GW + warp;
    const int t0 = tile * T;
    const float t0f = (float)t0, tendf = (float)(t0 + T - 1);
    const int lam_thr = t0 + lane * J;
    const float lamf = (float)lam_thr;

    const BoxView bv = box_view(g, st, slab, t0, T, lam_thr);

    f2_t acc[DP][J];
#pragma unroll
    for (int dp = 0; dp < DP; ++dp)
#pragma unroll
        for (int j = 0; j < J; ++j) acc[dp][j] = 0ull;
#pragma unroll
    for (int dd = 0; dd < DS; ++dd) {
        *comp_hi(s_comp, dd, tid, nthr) = make_float4(0.f, 0.f, 0.f, 0.f);
        *comp_lo(s_comp, dd, tid, nthr) = make_float4(0.f, 0.f, 0.f, 0.f);
    }

    warp_stage_depths<DS>(g, ws, d0 + warp * DS, lane);
    // chunks of LC lines; with GATHER (a centre test is set) of the lines this warp's slab
    // sweeps, so that lines whose slab the test rejects entirely are neither staged nor visited
    // one chunk of nl staged lines: the cells, then the fold into the compensated sums
    auto chunk = [&](const int nl) {
        const ulonglong2 *s_par = reinterpret_cast<const ulonglong2 *>(ws.par);
        const LineInfo *s_line = ws.info;
        int form = kFormSkip;          // of this lane's line of the current 32
        unsigned m_two = 0u;           // the two-term ones
        for (int li = 0; li < nl; ++li) {
            if ((li & 31) == 0) {
                const int lj = li + lane;
                form = lj < nl ? far_form(g, s_line[lj], t0f, tendf, slab, warp, bv) : kFormSkip;
                m_two = __ballot_sync(0xffffffffu, (form & 7) == kFormTwo);
            }
            const unsigned b = li & 31;
            const int fl = __shfl_sync(0xffffffffu, form, b);
            if (b < 31 && li + 1 < nl && ((m_two >> b) & 3u) == 3u) {
                // two consecutive two-term lines: their offsets and reciprocals are independent
                // chains, formed together; the sums take line li's terms, then line li + 1's
                const int fb = __shfl_sync(0xffffffffu, form, b + 1);
                f2_t spa[J], sqa[J], spb[J], sqb[J];
                far_reduced_s<J>(g, s_line[li], fl & kFormFull, box_near(g, bv, s_line[li], warp), lamf, lam_thr, spa, sqa);
                far_reduced_s<J>(g, s_line[li + 1], fb & kFormFull, box_near(g, bv, s_line[li + 1], warp), lamf, lam_thr,
                                 spb, sqb);
                const ulonglong2 *pa = s_par + (size_t)li * DP * NQ, *pb = pa + DP * NQ;
#pragma unroll
                for (int dp = 0; dp < DP; ++dp) {
                    const ulonglong2 qa = pa[NQ * dp + 1], qb = pb[NQ * dp + 1];
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        acc[dp][j] = f2_fma(sqa[j], qa.y, f2_fma(spa[j], qa.x, acc[dp][j]));
                        acc[dp][j] = f2_fma(sqb[j], qb.y, f2_fma(spb[j], qb.x, acc[dp][j]));
                    }
                }
                ++li;
                continue;
            }
            if ((fl & 7) == kFormSkip) continue;
            const LineInfo info = s_line[li];
            const ulonglong2 *par = s_par + (size_t)li * DP * NQ;
            const bool near = box_near(g, bv, info, warp);   // the lane's points are summed here
            if ((fl & 7) <= kFormWide) {
                f2_t sp[J];
                far_series_s<J>(g, info, fl, near, lamf, lam_thr,
                                far_cut(g, fl, info.sp, slab), sp);
                if ((fl & 7) >= kFormEight)
                    far_fwd_series<J, DP, 8>(par, sp, acc);
                else if ((fl & 7) == kFormFour)
                    far_fwd_series<J, DP, 4>(par, sp, acc);
                else if ((fl & 7) == kFormThree)
                    far_fwd_series<J, DP, 3>(par, sp, acc);
                else
                    far_fwd_series<J, DP, 2>(par, sp, acc);
            } else if ((fl & 7) == kFormLarge) {
                float U[J];
                far_scaled_u2<J>(g, info, lamf, U);
                f2_t u2[J];
#pragma unroll
                for (int j = 0; j < J; ++j) u2[j] = f2_splat(U[j]);
#pragma unroll
                for (int dp = 0; dp < DP; ++dp) {
                    // q0 = (K, a^2), q1 = (B1 K, B2' K^2): the polynomial in t with every
                    // coefficient times K, applied to r = t/K
                    const ulonglong2 q0 = par[NQ * dp], q1 = par[NQ * dp + 1];
                    f2_t B3, B4, B5;
                    far_b345(q0.y, q1.x, B3, B4, B5);
                    const f2_t B2 = f2_mul(q1.x, f2_splat(1.5f));
                    const f2_t ak = f2_mul(q0.y, q0.x);          // a^2 K
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        // r = 1/(U + a^2 K) = 4^-uexp/(u^2 + a^2/k^2), t = 1/(u^2 k^2 + a^2) = K r
                        const f2_t rr = f2_rcp(f2_fma(u2[j], f2_splat(1.0f), ak));
                        const f2_t r = near ? rr : 0ull;
                        const f2_t t = f2_mul(q0.x, r);
                        f2_t h = f2_fma(t, B5, B4);
                        h = f2_fma(t, h, B3);
                        h = f2_fma(t, h, B2);
                        h = f2_fma(t, h, q1.x);
                        acc[dp][j] = f2_fma(r, h, acc[dp][j]);
                    }
                }
            } else {
                // line near the tile or partly outside its window: far cells inside the window
                // only, classified near / far exactly as the near-core kernel does
                f2_t u2[J];
#pragma unroll
                for (int j = 0; j < J; ++j) u2[j] = f2_splat(offset_u((info.ilf - (lamf + (float)j)) + info.frac, g.lnr));
                const int il = (int)info.ilf;
                bool inwin[J];
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const int di = lam_thr + j - il;
                    inwin[j] = near && di >= -g.W && di <= g.W;
                }
                f2_t kp[DP];
                far_kpairs<DP>(g, info.sp, d0 + warp * DS, kp);
#pragma unroll
                for (int dp = 0; dp < DP; ++dp) {
                    const ulonglong2 q0 = par[NQ * dp], q1 = par[NQ * dp + 1];
                    // B1 = (B1 K) k^2 4^-uexp
                    const f2_t B1 = f2_mul(q1.x, f2_mul(f2_mul(kp[dp], kp[dp]), f2_splat(g.kunscale)));
                    f2_t B3, B4, B5;
                    far_b345(q0.y, B1, B3, B4, B5);
                    const f2_t B2 = f2_mul(B1, f2_splat(1.5f));
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const f2_t x = f2_mul(u2[j], kp[dp]);
                        const f2_t r2 = f2_fma(x, x, q0.y);
                        const f2_t t = f2_rcp(r2);
                        f2_t h = f2_fma(t, B5, B4);
                        h = f2_fma(t, h, B3);
                        h = f2_fma(t, h, B2);
                        h = f2_fma(t, h, B1);
                        const f2_t r = f2_fma(t, h, acc[dp][j]);
                        float r2a, r2b, ra, rb, aa, ab;
                        f2_unpack(r2, r2a, r2b);
                        f2_unpack(r, ra, rb);
                        f2_unpack(acc[dp][j], aa, ab);
                        aa = (inwin[j] && r2a >= kFar2) ? ra : aa;
                        ab = (inwin[j] && r2b >= kFar2) ? rb : ab;
                        acc[dp][j] = f2_pack(aa, ab);
                    }
                }
            }
        }
        // fold the chunk partials into the compensated sums (2Sum; the rounding
        // terms accumulate in this thread's shared-memory slots)
#pragma unroll
        for (int dp = 0; dp < DP; ++dp) {
            float pa[J], pb[J];
#pragma unroll
            for (int j = 0; j < J; ++j) {
                f2_unpack(acc[dp][j], pa[j], pb[j]);
                acc[dp][j] = 0ull;
            }
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                const int dd = 2 * dp + h2;
                float4 *ch = comp_hi(s_comp, dd, tid, nthr), *cl = comp_lo(s_comp, dd, tid, nthr);
                const float4 hsum = *ch, lsum = *cl;
                float hj[4] = {hsum.x, hsum.y, hsum.z, hsum.w};
                float lj[4] = {lsum.x, lsum.y, lsum.z, lsum.w};
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    float p = h2 ? pb[j] : pa[j], h = hj[j];
                    float s = h + p;
                    float bp = s - h;
                    float e = (h - (s - bp)) + (p - bp);
                    hj[j] = s;
                    lj[j] += e;
                }
                *ch = make_float4(hj[0], hj[1], hj[2], hj[3]);
                *cl = make_float4(lj[0], lj[1], lj[2], lj[3]);
            }
        }
    };
    auto listed = [&](const int nl) {
        warp_fill<NQ, DS>(g, ws, ginfo, 0, nl, d0 + warp * DS, lane, true);
        chunk(nl);
    };
    if (GATHER) {
        for (int cur = lo; cur < hi;) {
            const int nl = warp_gather(ws, ginfo, cur, hi, LC, warp, lane);
            if (nl == 0) break;
            listed(nl);
        }
    } else {
        const int nch = (hi - lo + LC - 1) / LC;
        for (int c = 0; c < nch; ++c) {
            const int nl = min(LC, hi - (lo + c * LC));
            warp_fill<NQ, DS>(g, ws, ginfo, lo + c * LC, nl, d0 + warp * DS, lane);
            chunk(nl);
        }
    }
    box_rings(g, bv, st, slab, box_group_n0(g, st, group, GW), t0, T, ext.w, ext.y, ws, LC, lane, listed);

    if (ext.y > 1) {
        // one of ext.y pieces of a split item (slots ext.x.., counter ext.z, piece ext.w):
        // store this piece's compensated sums; the piece that completes the item adds
        // all pieces' sums in piece order and finishes the cells below
        __shared__ int s_last;
        const size_t slot = (size_t)DS * nthr * 2;
        float4 *mine = g.fpart + (size_t)(ext.x + ext.w) * slot;
#pragma unroll
        for (int dd = 0; dd < DS; ++dd) {
            mine[((size_t)dd * nthr + tid) * 2] = *comp_hi(s_comp, dd, tid, nthr);
            mine[((size_t)dd * nthr + tid) * 2 + 1] = *comp_lo(s_comp, dd, tid, nthr);
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(g.fcnt + ext.z, 1) == ext.y - 1;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
#pragma unroll
        for (int dd = 0; dd < DS; ++dd) {
            float hj[4] = {0.f, 0.f, 0.f, 0.f}, lj[4] = {0.f, 0.f, 0.f, 0.f};
            for (int q = 0; q < ext.y; ++q) {
                const float4 *src = g.fpart + (size_t)(ext.x + q) * slot + ((size_t)dd * nthr + tid) * 2;
                const float4 h4 = __ldcg(src), l4 = __ldcg(src + 1);
                const float hq[4] = {h4.x, h4.y, h4.z, h4.w}, lq[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float h = hj[j], p = hq[j];
                    const float sum = h + p;
                    const float bp = sum - h;
                    const float e = (h - (sum - bp)) + (p - bp);
                    hj[j] = sum;
                    lj[j] += lq[j] + e;
                }
            }
            *comp_hi(s_comp, dd, tid, nthr) = make_float4(hj[0], hj[1], hj[2], hj[3]);
            *comp_lo(s_comp, dd, tid, nthr) = make_float4(lj[0], lj[1], lj[2], lj[3]);
        }
    }

    // epilogue: near-core sums, stimulated-emission factor at the sample frequency, vector store
#pragma unroll
    for (int dd = 0; dd < DS; ++dd) {
        int d = d0 + warp * DS + dd;
        if (d >= g.nd) continue;
        float c2T = __ldg(g.c2T + d);
        const float4 hsum = *comp_hi(s_comp, dd, tid, nthr), lsum = *comp_lo(s_comp, dd, tid, nthr);
        const float hj[4] = {hsum.x, hsum.y, hsum.z, hsum.w};
        const float lj[4] = {lsum.x, lsum.y, lsum.z, lsum.w};
        const float *nrow = g.knear + (int64_t)d * g.ld + lam_thr;
        float v[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            float lam = g.lam0cm * expf((float)(lam_thr + j) * g.lnr);
            float stim = -expm1f(-c2T / lam);
            float hi2 = hj[j], nj = nrow[j];
            float s = hi2 + nj;                    // 2Sum of the near-core sum into the total
            float bp = s - hi2;
            float e = (hi2 - (s - bp)) + (nj - bp);
            v[j] = stim * (s + (lj[j] + e));
        }
        float *row = g.kline + (int64_t)d * g.ld + lam_thr;
        if (J == 4)
            *reinterpret_cast<float4 *>(row) = make_float4(v[0], v[1 % J], v[2 % J], v[3 % J]);
        else
            *reinterpret_cast<float2 *>(row) = make_float2(v[0], v[1 % J]);
    }
}

// Shared memory of the far-wing kernels: each warp's stage (warp_stage_quads), then
// (forward) the compensated sums of every thread [DS][threads][8] or (backward) the
// per-line sums of the warps, double-buffered by chunk [2][LC][GW], and each warp's
// per-lane partial sums of a batch of kBwdBatch lines [kBwdBatch][32] (lane l of line k at
// column l ^ k, so that both the row writes and the column reads avoid bank conflicts).
template <int J, int DS, int MINB, bool GATHER>
__global__ void __launch_bounds__(128, MINB) k_line_fwd(LineArgs g, int GW, int LC) {
    extern __shared__ float4 smem4[];
    const int warp = threadIdx.x >> 5;
    const size_t wq = warp_stage_quads(LC, DS, kNQF);
    float4 *mine = smem4 + (size_t)warp * wq;
    const WarpStage ws = make_stage(mine, LC, DS, kNQF);
    float *s_comp = reinterpret_cast<float *>(smem4 + (size_t)GW * wq);
    for_each_item(g, [&](const LineArgs &v, int tile, int group, int lo, int hi, int it) {
        far_fwd_item<J, DS, GATHER>(v, g.items[it].x, tile, group, lo, hi, GW, LC, ws, s_comp, g.fext[it]);
    });
}

// One line's far-wing backward sums over a warp's J x DS cells (depth pairs):
// S[0] += G stim A H, Y += G stim A a6 dH/da.  Without MASK, w holds the scaled squared
// offsets U = 4^uexp u^2; with MASK, w holds the offsets u and kp the depth pairs' k, and
// only the far cells inside the window (inwin per lambda point) are kept.
template <int J, int DP, bool MASK, bool FOUR>
__device__ __forceinline__ void far_bwd_line(const LineArgs &g, const ulonglong2 *par, const f2_t (&w)[J],
                                             const f2_t (&gv)[DP][J], const bool near, const bool *inwin, const f2_t *kp,
                                             FarSums<FOUR> &R) {
    constexpr int NQ = far_nqb<FOUR>();
#pragma unroll
    for (int dp = 0; dp < DP; ++dp) {
        // (K, a^2) (B1 K, B2' K^2) (C1 K, C2' K^2); the other coefficients from a^2, B1 K and C1 K
        const ulonglong2 q0 = par[NQ * dp], q1 = par[NQ * dp + 1], q2 = par[NQ * dp + 1 + kPolyN / 2];
        f2_t Y = R.open();
        f2_t B1 = q1.x, C1 = q2.x;
        if (MASK) {
            // the masked cells use t = 1/|z|^2 itself: B1 = (B1 K) k^2 4^-uexp, C1 alike
            const f2_t kk = f2_mul(f2_mul(kp[dp], kp[dp]), f2_splat(g.kunscale));
            B1 = f2_mul(B1, kk);
            C1 = f2_mul(C1, kk);
        }
        f2_t B3, B4, B5, C3, C4, C5, C6;
        far_b345(q0.y, B1, B3, B4, B5);
        far_c3456(q0.y, C1, C3, C4, C5, C6);
        const f2_t B2 = f2_mul(B1, f2_splat(1.5f));
        const f2_t C2 = f2_mul(f2_fma(q0.y, f2_splat(-2.0f), f2_splat(1.5f)), C1);
        const f2_t ak = f2_mul(q0.y, q0.x);          // a^2 K
#pragma unroll
        for (int j = 0; j < J; ++j) {
            f2_t r2, t, m;
            if (MASK) {
                const f2_t x = f2_mul(w[j], kp[dp]);
                r2 = f2_fma(x, x, q0.y);
                t = f2_rcp(r2);
                m = t;
            } else {
                // r = 1/(U + a^2 K), t = K r; the coefficients carry K, so the sums take r
                const f2_t rr = f2_rcp(f2_fma(w[j], f2_splat(1.0f), ak));
                m = near ? rr : 0ull;
                t = f2_mul(q0.x, m);
            }
            f2_t h = f2_fma(t, B5, B4);
            h = f2_fma(t, h, B3);
            h = f2_fma(t, h, B2);
            h = f2_fma(t, h, B1);
            f2_t q = f2_fma(t, C6, C5);
            q = f2_fma(t, q, C4);
            q = f2_fma(t, q, C3);
            q = f2_fma(t, q, C2);
            q = f2_fma(t, q, C1);
            f2_t gt = f2_mul(gv[dp][j], m);
            if (MASK) {
                float r2a, r2b, ga, gb;
                f2_unpack(r2, r2a, r2b);
                f2_unpack(gt, ga, gb);
                ga = (inwin[j] && r2a >= kFar2) ? ga : 0.0f;
                gb = (inwin[j] && r2b >= kFar2) ? gb : 0.0f;
                gt = f2_pack(ga, gb);
            }
            R.S[0] = f2_fma(gt, h, R.S[0]);
            Y = f2_fma(gt, q, Y);
        }
        R.close(Y, par + NQ * dp);
    }
}

// Accumulator row of a line sum: strength, van der Waals, radiative, Stark.
__device__ __forceinline__ int64_t far_row(int q) { return q < 2 ? q : 2 * q - 1; }

// Far-wing kernel (backward): the per-line sums over the tile's far cells of
// G stim A H and G stim A a6 dH/da, reduced over the CTA and added to gacc.
template <int J, int DS, bool FOUR>
__device__ __forceinline__ void far_bwd_item(const LineArgs &g, const int st, const int tile, const int group,
                                             const int lo, const int hi, const int GW, const int LC,
                                             const WarpStage &ws, float2 *s_part, float2 *s_red2, unsigned &cc,
                                             const int4 ext) {
    static_assert(J == 2 || J == 4, "J must be 2 or 4");
    static_assert(DS % 2 == 0, "DS must be even (depth pairs)");
    constexpr int DP = DS / 2;
    constexpr int NQ = far_nqb<FOUR>();
    constexpr int NS = FOUR ? 2 : 1;          // pairs of sums
    const int T = 32 * J;
    const int DC = GW * DS;
    const int nthr = blockDim.x;
    const LineInfo *ginfo = g.finfo + (int64_t)group * g.nl;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d0 = group * DC;
    const int slab = group * GW + warp;
    const int t0 = tile * T;
    const float t0f = (float)t0, tendf = (float)(t0 + T - 1);
    const int lam_thr = t0 + lane * J;
    const float lamf = (float)lam_thr;

    // G * stim of the thread's cells as depth pairs; zero outside the grid
    f2_t gv[DP][J];
#pragma unroll
    for (int dp = 0; dp < DP; ++dp) {
        const int da = d0 + warp * DS + 2 * dp, db = da + 1;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const bool inl = lam_thr + j < g.nlam;
            const float ga = (da < g.nd && inl) ? g.Gt[(int64_t)da * g.ld + lam_thr + j] : 0.0f;
            const float gb = (db < g.nd && inl) ? g.Gt[(int64_t)db * g.ld + lam_thr + j] : 0.0f;
            gv[dp][j] = f2_pack(ga, gb);
        }
    }

    warp_stage_depths<DS>(g, ws, d0 + warp * DS, lane);
    const BoxView bv = box_view(g, st, slab, t0, T, lam_thr);
    // the staged lines of one chunk: the warp's sums 2h and 2h + 1 of slot k go to sink(k, h, a, b)
    auto put = [&](const int r, const FarSums<FOUR> &R) {
#pragma unroll
        for (int h = 0; h < NS; ++h)
            s_part[(h * kBwdBatch + r) * 32 + (lane ^ r)] =
                make_float2(f2_lo(R.S[2 * h]) + f2_hi(R.S[2 * h]), f2_lo(R.S[2 * h + 1]) + f2_hi(R.S[2 * h + 1]));
    };
    auto chunk = [&](const int nl, auto &&sink) {
        const ulonglong2 *s_par = reinterpret_cast<const ulonglong2 *>(ws.par);
        const LineInfo *s_line = ws.info;
        int form = kFormSkip;          // of this lane's line of the current 32
        unsigned m_two = 0u;           // the two-term ones
        for (int li = 0; li < nl;) {
            const unsigned b = li & 31;
            if (b == 0) {
                const int lj = li + lane;
                form = lj < nl ? far_form(g, s_line[lj], t0f, tendf, slab, warp, bv) : kFormSkip;
                m_two = __ballot_sync(0xffffffffu, (form & 7) == kFormTwo);
            }
            const int fl = __shfl_sync(0xffffffffu, form, b);
            if ((b & (kBwdBatch - 1)) != kBwdBatch - 1 && li + 1 < nl && ((m_two >> b) & 3u) == 3u) {
                // two consecutive two-term lines of one batch: independent offset and
                // reciprocal chains, formed together
                const int fb = __shfl_sync(0xffffffffu, form, b + 1);
                f2_t spa[J], sqa[J], spb[J], sqb[J];
                far_reduced_s<J>(g, s_line[li], fl & kFormFull, box_near(g, bv, s_line[li], warp), lamf, lam_thr, spa, sqa);
                far_reduced_s<J>(g, s_line[li + 1], fb & kFormFull, box_near(g, bv, s_line[li + 1], warp), lamf, lam_thr,
                                 spb, sqb);
                const ulonglong2 *pa = s_par + (size_t)li * DP * NQ;
                FarSums<FOUR> Ra, Rb;
                Ra.clear();
                Rb.clear();
                far_bwd_series<J, DP, 2, FOUR>(pa, spa, gv, Ra);
                far_bwd_series<J, DP, 2, FOUR>(pa + DP * NQ, spb, gv, Rb);
                const int r = b & (kBwdBatch - 1);
                put(r, Ra);
                put(r + 1, Rb);
                li += 2;
            } else {
                const LineInfo info = s_line[li];
                const ulonglong2 *par = s_par + (size_t)li * DP * NQ;
                FarSums<FOUR> R;
                R.clear();
                // (a slab whose every layer the centre test rejects keeps zero sums)
                if ((fl & 7) != kFormSkip) {
                    const bool near = box_near(g, bv, info, warp);   // the lane's points are summed here
                    if ((fl & 7) <= kFormWide) {
                        f2_t sp[J];
                        far_series_s<J>(g, info, fl, near, lamf, lam_thr,
                                        far_cut(g, fl, info.sp, slab), sp);
                        if ((fl & 7) >= kFormEight)
                            far_bwd_series<J, DP, 8, FOUR>(par, sp, gv, R);
                        else if ((fl & 7) == kFormFour)
                            far_bwd_series<J, DP, 4, FOUR>(par, sp, gv, R);
                        else if ((fl & 7) == kFormThree)
                            far_bwd_series<J, DP, 3, FOUR>(par, sp, gv, R);
                        else
                            far_bwd_series<J, DP, 2, FOUR>(par, sp, gv, R);
                    } else if ((fl & 7) == kFormLarge) {
                        float U[J];
                        far_scaled_u2<J>(g, info, lamf, U);
                        f2_t u2[J];
#pragma unroll
                        for (int j = 0; j < J; ++j) u2[j] = f2_splat(U[j]);
                        far_bwd_line<J, DP, false, FOUR>(g, par, u2, gv, near, nullptr, nullptr, R);
                    } else {
                        // line near the tile or partly outside its window: far cells inside the window only
                        f2_t u2[J];
#pragma unroll
                        for (int j = 0; j < J; ++j)
                            u2[j] = f2_splat(offset_u((info.ilf - (lamf + (float)j)) + info.frac, g.lnr));
                        bool inwin[J];
                        const int il = (int)info.ilf;
#pragma unroll
                        for (int j = 0; j < J; ++j) {
                            const int di = lam_thr + j - il;
                            inwin[j] = near && di >= -g.W && di <= g.W;
                        }
                        f2_t kp[DP];
                        far_kpairs<DP>(g, info.sp, d0 + warp * DS, kp);
                        far_bwd_line<J, DP, true, FOUR>(g, par, u2, gv, near, inwin, kp, R);
                    }
                }
                const int r = b & (kBwdBatch - 1);
                put(r, R);
                ++li;
            }
            if ((li & (kBwdBatch - 1)) == 0 || li >= nl) {
                // end of a batch of kBwdBatch lines: lanes 2r and 2r + 1 add the two halves of
                // line r's partial sums over the warp's lanes (row r holds lane j's at column
                // j ^ r), combine them and leave the warp's total for the CTA reduction
                __syncwarp();
                const int base = (li - 1) & ~(kBwdBatch - 1);
                const int r = lane >> 1, h = lane & 1;
#pragma unroll
                for (int q = 0; q < NS; ++q) {
                    float a1 = 0.0f, a2 = 0.0f;
                    if (base + r < nl) {
                        const float2 *row = s_part + (q * kBwdBatch + r) * 32;
#pragma unroll 8
                        for (int t = 0; t < 16; ++t) {
                            const float2 v = row[(16 * h + t) ^ r];
                            a1 += v.x;
                            a2 += v.y;
                        }
                    }
                    a1 += __shfl_xor_sync(0xffffffffu, a1, 1);
                    a2 += __shfl_xor_sync(0xffffffffu, a2, 1);
                    if (h == 0 && base + r < nl) sink(base + r, q, a1, a2);
                }
                __syncwarp();
            }
        }
    };
    const int nch = (hi - lo + LC - 1) / LC;
    for (int c = 0; c < nch; ++c) {
        const int c0 = lo + c * LC;
        const int nl = min(LC, hi - c0);
        // per-line sums of this chunk go to buffer cc & 1: its previous readers (the
        // reduction two chunks back) are past the CTA barrier of the previous chunk
        float2 *s_red = s_red2 + (size_t)((cc + c) & 1) * NS * LC * GW;
        warp_fill<NQ, DS>(g, ws, ginfo, c0, nl, d0 + warp * DS, lane);
        chunk(nl, [&](int k, int q, float a1, float a2) { s_red[(q * LC + k) * GW + warp] = make_float2(a1, a2); });
        __syncthreads();
        // thread k adds sum k % 2NS of line k / 2NS over the warps in FP32, in warp order, and
        // converts once for the FP64 accumulator: FP64 arithmetic runs at a small fraction
        // of the FP32 rate, and a chain of FP64 adds here would hold the CTA at the next barrier
        for (int k = tid; k < 2 * NS * nl; k += nthr) {
            const int li = k / (2 * NS), q = k % (2 * NS);
            const float *r = reinterpret_cast<const float *>(s_red + ((q >> 1) * LC + li) * GW) + (q & 1);
            float a = r[0];
            for (int w = 1; w < GW; ++w) a += r[2 * w];
            atomicAdd(g.gacc + far_row(q) * g.nl + c0 + li, (double)a);
        }
    }
    cc += nch;
    // lines beyond the near boxes: each warp gathers its slab's and adds their sums itself
    box_rings(g, bv, st, slab, box_group_n0(g, st, group, GW), t0, T, ext.w, ext.y, ws, LC, lane, [&](const int nl) {
        warp_fill<NQ, DS>(g, ws, ginfo, 0, nl, d0 + warp * DS, lane, true);
        chunk(nl, [&](int k, int q, float a1, float a2) {
            atomicAdd(g.gacc + far_row(2 * q) * g.nl + ws.idx[k], (double)a1);
            atomicAdd(g.gacc + far_row(2 * q + 1) * g.nl + ws.idx[k], (double)a2);
        });
    });
}

template <int J, int DS, int MINB, bool FOUR>
__global__ void __launch_bounds__(128, MINB) k_line_bwd(LineArgs g, int GW, int LC) {
    extern __shared__ float4 smem4[];
    const int warp = threadIdx.x >> 5;
    constexpr int NQ = far_nqb<FOUR>(), NS = FOUR ? 2 : 1;
    const size_t wq = warp_stage_quads(LC, DS, NQ);
    float4 *mine = smem4 + (size_t)warp * wq;
    const WarpStage ws = make_stage(mine, LC, DS, NQ);
    float2 *s_red2 = reinterpret_cast<float2 *>(smem4 + (size_t)GW * wq);
    float2 *s_part = s_red2 + (size_t)2 * NS * LC * GW + (size_t)warp * NS * kBwdBatch * 32;
    unsigned cc = 0;
    for_each_item(g, [&](const LineArgs &v, int tile, int group, int lo, int hi, int it) {
        far_bwd_item<J, DS, FOUR>(v, g.items[it].x, tile, group, lo, hi, GW, LC, ws, s_part, s_red2, cc, g.fext[it]);
    });
}

// Supported (lambda points per thread, depths per warp, minimum resident CTAs per SM).
#define PZ_TILE_LIST(X) \
    X(4, 6, 1) X(4, 6, 2) X(4, 6, 3) X(4, 6, 4) X(4, 8, 1) X(4, 8, 2) X(4, 8, 3) X(4, 12, 1) X(4, 12, 2) \
    X(2, 6, 4) X(2, 8, 2) X(2, 8, 3) X(2, 8, 4) X(2, 12, 1) X(2, 12, 2) X(2, 12, 3) X(4, 6, 5) X(4, 6, 6) X(2, 6, 6) X(2, 8, 5)

constexpr size_t kFarSmemMax = 200 * 1024;   // the opt-in size the far-wing kernels are given

// Persistent grid: as many CTAs as fit on the GPU at once, at most one per item.
template <class K>
static int persistent_grid(pz_ctx *c, K kernel, int threads, size_t smem, int n_items) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    int64_t n = (int64_t)per_sm * std::max(c->n_sm, 1);
    return (int)std::max<int64_t>(1, std::min<int64_t>(n, n_items));
}

// The far-wing reverse pass of the current tiling (pz_line_bwd.cu); LC lines per chunk.
cudaError_t launch_far_bwd(pz_ctx *c, const LineArgs &g, int LC, size_t smem, cudaStream_t s);
cudaError_t launch_far_bwd4(pz_ctx *c, const LineArgs &g, int LC, size_t smem, cudaStream_t s);

}  // namespace pz
