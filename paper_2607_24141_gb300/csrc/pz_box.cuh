// pz_box.cuh -- box expansions of the far wings (included by pz_line.cu).
//
// Far from a line's core its profile is a short series in p = 1/v^2,
//   H sqrt(pi)/A = a sum_n beta_n(a^2) p^(n+1),   dH/da sqrt(pi) = sum_n gamma_n(a^2) p^(n+1),
// and p depends on the line and the point only through their distance: p = kap f(x_l - i),
// f(D) = (eps/u)^2 with u = expm1(D ln r), eps = (B/2) ln r and kap = 1/(k eps)^2 per
// (species, layer).  Both kernels of the sum over lines are smooth over boxes of B grid
// points that are a few boxes apart, so the sum does not need a term per (line, point):
//   f(x - i) = sum_{k + j <= P(o)} C_kj(o) T_k(x^) T_j(i^)
// for a line in box s and a point in box t = s - o (T: Chebyshev polynomials, x^ and i^ the
// positions in their boxes scaled to [-1, 1]).  The powers of f follow from derivatives of f
// along x: u^-(m+1) = -(1/m)(d/dy + m) u^-m, y = D ln r, so
//   f^2 = (1/6)  (d + 3 eps)(d + 2 eps) f,   f^3 = (1/20) (d + 5 eps)(d + 4 eps) f^2,
//   f^4 = (1/42) (d + 7 eps)(d + 6 eps) f^3,  d = d/dx^,
// and applying them to T_k(x^) instead (W_qk below) leaves one kernel for all four terms.
//
// Forward:  k_box_moments   per source box and layer: M_k = sum_l sum_q w_q(l, d) W_qk(x^_l)
//           k_box_field     per target box: Phi_j = sum_o sum_k C_kj(o) M_k(t + o), then
//                           sum_j Phi_j T_j(i^) at its points
// Backward: k_box_gmoments  per target box: N_j = sum_i T_j(i^) G_i
//           k_box_grad      per source box: Psi_k = sum_o sum_j C_kj(o) N_j(s - o), then per line
//                           sum_d w_q sum_k W_qk Psi_k (and the same with the damping weights)
//
// Which pairs: all boxes |o| >= n_c whose points lie inside the window of every line of the
// source box (|o| <= omax = (W + 1)/B - 1).  n_c is the line's separation class at the slab
// of layers: at distance (n_c - 1) B every |v| is at least 20 (the widest species) and 9 a,
// where the dropped terms are at most 2.2e-8 of H and 2.1e-7 of dH/da (the first of them (a/v)^8 and
// 9 (a/v)^8, at |v| = 9 a; a tenth of that at a = v/12); n_0 >= 3 keeps the expansions' truncation
// below 1e-7.  Lines whose damping needs more than the widest class keep class 4 and are summed
// directly over their whole window.  A window ends inside at most two further boxes on each
// side; there f is almost constant over a box, a few k suffice, and the sharp end is kept by
// moments of every grid index of the boxes by itself, which the points add up in the order in
// which their windows reach the indices.
// Pairs nearer than n_c stay with the far-wing kernels, which skip exactly the pairs that
// are summed here (box_near).
//
// Cost per (point, layer): about 76 FMA for the boxes and 20 for the window ends at W = 1500,
// B = 32, whatever the number of lines, and about 60 per (line, layer), against 2-3 per (line,
// point, layer) for 3001 points of every line's window.
#pragma once

namespace pz {

constexpr int kBoxP = 13;                 // largest order: k + j <= 13 at the nearest box pair
constexpr int kBoxK = kBoxP + 1;          // moments per box
constexpr int kBoxRow = 16;               // row stride of the C tables (floats)
constexpr int kBoxSplit = kBoxQuarters;   // threads that share a (box, layer)

// Order of the expansion at box offset |o|: the worst error over the two boxes, relative to
// the pair's largest term, stays below 1e-7 at |o| = 3 and 4e-8 beyond (the corners; the mean
// over a box is some ten times smaller), evaluated for all four terms of H and dH/da.
__host__ __device__ __forceinline__ int box_order(int o) {
    return o >= 90 ? 3 : o >= 33 ? 4 : o >= 19 ? 5 : o >= 14 ? 6 : o >= 9 ? 7 : o >= 7 ? 8 : o == 6 ? 9 : o == 5 ? 10
                                                                                      : o == 4 ? 11 : 13;
}

// Chebyshev coefficients C_kj of f at every offset (side 0: o > 0, 1: o < 0), FP64 quadrature
// at 16 x 16 nodes, one block per (offset, side).  C[side][o][k][j], zero for k + j > P(o).
__global__ void k_box_tables(int B, double lnr, int omax, float *C) {
    constexpr int N = 16;
    __shared__ double f[N][N], g[N][N], Tn[N][N];
    const int o = blockIdx.x + 1, side = blockIdx.y;
    const int a = threadIdx.x / N, b = threadIdx.x % N;
    const double h = 0.5 * B, eps = h * lnr;
    const double xa = cospi((a + 0.5) / N), xb = cospi((b + 0.5) / N);
    const double u = expm1(((side ? -o : o) * (double)B + h * (xa - xb)) * lnr);
    f[a][b] = (eps / u) * (eps / u);
    Tn[a][b] = cospi(a * (b + 0.5) / N) * (a == 0 ? 1.0 : 2.0) / N;   // weight of node b in coefficient a
    __syncthreads();
    double s = 0.0;
    for (int n = 0; n < N; ++n) s += Tn[a][n] * f[n][b];
    g[a][b] = s;
    __syncthreads();
    s = 0.0;
    for (int n = 0; n < N; ++n) s += Tn[b][n] * g[a][n];
    if (a < kBoxK) C[(((size_t)side * (omax + 3) + o) * kBoxK + a) * kBoxRow + b] = (a + b <= box_order(o)) ? (float)s : 0.0f;
}

// Window-end tables: E[side][e][r][k] = sum_j C_kj(+-(omax + 1 + e)) T_j(i^_r), k <= KE - 1.
__global__ void k_box_edges(int B, int omax, int KE, const float *C, float *E) {
    const int k = threadIdx.x, r = blockIdx.x, e = blockIdx.y, side = blockIdx.z;
    if (k >= KE) return;
    const float *c = C + (((size_t)side * (omax + 3) + omax + 1 + e) * kBoxK + k) * kBoxRow;
    const float x = (r - 0.5f * (B - 1)) / (0.5f * B);
    float tm = 1.0f, t = x, s = c[0];
    for (int j = 1; j < kBoxK; ++j) {
        s = fmaf(c[j], t, s);
        const float n = fmaf(2.0f * x, t, -tm);
        tm = t;
        t = n;
    }
    E[(((size_t)side * 2 + e) * B + r) * KE + k] = s;
}

// First line of every quarter of a box: start[star][q] = first line of the star with i_l >= s_lo B + q B/4.
__global__ void k_box_start(int nq, int s_lo, int B, const int32_t *stars, const int32_t *il, const int64_t *off,
                            int64_t row, int32_t *start) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x, st = stars[blockIdx.y];
    if (b > nq) return;
    int64_t lo = off[st], hi = off[st + 1];
    const int64_t key = (int64_t)s_lo * B + (int64_t)b * (B / kBoxSplit);
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (il[mid] < key) lo = mid + 1; else hi = mid;
    }
    start[(int64_t)st * row + b] = (int32_t)lo;
}

struct BoxArgs {
    int B, omax, rem;             // box, widest whole offset, (W + 1) - (omax + 1) B
    int s_lo, nbox, ntb;          // first source box and source boxes of this launch, target boxes
    int box0, tgt0;               // place of s_lo among the star's boxes, first target box of this launch
    int DC, DS;                   // tiling of the line records (class bits)
    const int32_t *stars;         // stars of this launch
    float invh, ctr;              // 2/B, (B - 1)/2
    float kapscale;               // kap = K kapscale (K = 4^uexp/k^2)
    const float *A;               // [3][kBoxK][kBoxK]: W_qk = sum_j A[q - 2][k][j] T_j, q = 2..4
    const float *C, *E;           // expansion and window-end tables
    const int *nmin;              // [S][nslab][4]
    float *M, *PM, *N;            // moments [star][box][class][k][nd], those of each grid index [star][box][B][KE][nd],
                                  // moments of G [star][target box][k][nd]
};

// T_0..T_13 at x
__device__ __forceinline__ void box_cheb(float x, float (&T)[kBoxK]) {
    T[0] = 1.0f;
    T[1] = x;
#pragma unroll
    for (int k = 2; k < kBoxK; ++k) T[k] = fmaf(2.0f * x, T[k - 1], -T[k - 2]);
}

// W_1k..W_4k of a line at x^ (k = 0..13): T_k and its images under the operators of f^2, f^3, f^4
__device__ __forceinline__ void box_weights(const BoxArgs &b, float x, float4 *w) {
    float T[kBoxK];
    box_cheb(x, T);
#pragma unroll
    for (int k = 0; k < kBoxK; ++k) {
        float s2 = 0.0f, s3 = 0.0f, s4 = 0.0f;
#pragma unroll
        for (int j = 0; j <= k; ++j) {
            s2 = fmaf(__ldg(b.A + (0 * kBoxK + k) * kBoxK + j), T[j], s2);
            s3 = fmaf(__ldg(b.A + (1 * kBoxK + k) * kBoxK + j), T[j], s3);
            s4 = fmaf(__ldg(b.A + (2 * kBoxK + k) * kBoxK + j), T[j], s4);
        }
        w[k] = make_float4(T[k], s2, s3, s4);
    }
}

// Series weights of a (line, layer): A a/sqrt(pi) beta_n kap^(n+1) and, with D, A/sqrt(pi) gamma_n
// kap^(n+1)/(4 pi dnu_D) without the families' factors gb (van der Waals, radiative, Stark), with the
// prefactors of depth_params; dc = {beta_hi, beta_lo, n_e, n_pert}.
template <bool D>
__device__ __forceinline__ void box_series(const LineArgs &g, const BoxArgs &b, const LineScalars &L, int64_t l, int d,
                                           const float4 dc, float4 &w, float4 &c, float3 &gb) {
    const int id = L.sp * g.nd + d;
    const float invdv = __ldg(g.invdv + id);
    const float p = L.E * dc.x;
    const float r = fmaf(L.E, dc.x, -p) + L.E * dc.y;
    const float A = pair_kept(g.keep, l, d) ? L.Q * __ldg(g.R + id) * (expf(-p) * (1.0f - r)) : 0.0f;
    const float lw = L.lamcm * invdv * (float)(1.0 / (4.0 * kPI));
    const float g6n = L.g6 * dc.w;
    const float a = fmaf(L.g4, dc.z, L.grad + g6n) * lw;
    const float a2 = a * a;
    const float kap = __ldg(g.Ksd + id) * b.kapscale;
    const float B1 = A * a * kInvSqrtPiF * kap;
    const float k2 = kap * kap, k3 = k2 * kap;
    w.x = B1;
    w.y = B1 * kap * (1.5f - a2);
    w.z = B1 * k2 * fmaf(a2, a2 - 5.0f, 3.75f);
    w.w = B1 * k3 * fmaf(a2, fmaf(a2, 10.5f - a2, -26.25f), 13.125f);
    if (D) {
        gb = make_float3(g6n, L.grad, L.g4 * dc.z);
        const float C1 = A * lw * kInvSqrtPiF * kap;
        c.x = C1;
        c.y = C1 * kap * fmaf(-3.0f, a2, 1.5f);
        c.z = C1 * k2 * fmaf(a2, fmaf(5.0f, a2, -15.0f), 3.75f);
        c.w = C1 * k3 * fmaf(a2, fmaf(a2, fmaf(-7.0f, a2, 52.5f), -78.75f), 13.125f);
    }
}

__device__ __forceinline__ void two_sum(float &hi, float &lo, float p) {
    const float s = hi + p;
    const float bp = s - hi;
    lo += (hi - (s - bp)) + (p - bp);
    hi = s;
}

// Running sum of an expansion: the leading coefficients, which hold nearly all of the sum, are
// compensated.
constexpr int kBoxComp = 4;
struct BoxSum {
    float acc[kBoxK], hi[kBoxComp], lo[kBoxComp];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int k = 0; k < kBoxK; ++k) acc[k] = 0.0f;
#pragma unroll
        for (int k = 0; k < kBoxComp; ++k) hi[k] = lo[k] = 0.0f;
    }
    __device__ __forceinline__ void fold() {
#pragma unroll
        for (int k = 0; k < kBoxComp; ++k) {
            two_sum(hi[k], lo[k], acc[k]);
            acc[k] = 0.0f;
        }
    }
    __device__ __forceinline__ float get(int k) const { return k < kBoxComp ? hi[k] + (lo[k] + acc[k]) : acc[k]; }
};

__host__ __device__ constexpr int box_chunk(int NP) { return NP == 1 ? 32 : 16; }   // lines staged at a time and part
constexpr int kBoxBatch = 4;      // lines whose weights are formed together
template <int NP>
struct BoxStage {
    float4 w[NP][box_chunk(NP)][kBoxK];
    LineScalars l[NP][box_chunk(NP)];
    int q[NP][box_chunk(NP)];
};
template <int NP>
static size_t box_moment_smem(int nd) {
    return sizeof(BoxStage<NP>) + sizeof(float) * (size_t)NP * nd * 4 * kBoxK;
}

// Moments of one source box: thread = (part of the box's indices, layer), block = box (x) and star
// (y).  NP = 4 parts where the grid has few boxes: with one, the lines' chain of loads and sums leaves
// the chip waiting (12,000 lines in 165 boxes: forward lines 0.485 -> 0.420 ms); NP = 1 on longer grids,
// where the parts' shared memory leaves two boxes per SM (two stars on 10^5 lines: 2.50 ms, one part 2.40).
template <int KE, int NP>
__global__ void __launch_bounds__(NP * 128) k_box_moments(LineArgs gq, BoxArgs b) {
    constexpr int QP = kBoxSplit / NP, CH = box_chunk(NP);   // quarters per part, lines per chunk
    extern __shared__ float4 smem4[];
    BoxStage<NP> &sg = *reinterpret_cast<BoxStage<NP> *>(smem4);
    const int tid = threadIdx.x, box = blockIdx.x, sl = blockIdx.y, st = b.stars[sl];
    const LineArgs g = star_view(gq, st);
    const int nd = g.nd, part = tid / nd, d = tid - part * nd;
    const bool live = part < NP;
    float *s_cls = reinterpret_cast<float *>(&sg + 1);          // [part][3][kBoxK][nd]: lines of classes 1..3
    float *s_m = s_cls + NP * 3 * kBoxK * nd;            // [part][kBoxK][nd]: class 0
    const int32_t *start = gq.bstart + (int64_t)st * gq.brow + kBoxSplit * (b.box0 + box);
    const int i0 = (b.s_lo + box) * b.B;
    int most = 0;
#pragma unroll
    for (int q = 0; q < NP; ++q) most = max(most, start[(q + 1) * QP] - start[q * QP]);
    const int lo = live ? start[part * QP] : 0, hi = live ? start[(part + 1) * QP] : 0;
    const float4 dc = live ? make_float4(__ldg(g.beta_hi + d), __ldg(g.beta_lo + d), __ldg(g.ne + d), __ldg(g.npert + d))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    const int grp = live ? d / b.DC : 0, shift = 16 + 3 * (live ? (d % b.DC) / b.DS : 0);
    const LineInfo *info = gq.finfo + (int64_t)grp * gq.nl;
    BoxSum S;
    S.clear();
    float pm[KE];
#pragma unroll
    for (int k = 0; k < KE; ++k) pm[k] = 0.0f;
    for (int k = tid; k < NP * 3 * kBoxK * nd; k += blockDim.x) s_cls[k] = 0.0f;
    float *PM = b.PM + (((int64_t)sl * b.nbox + box) * b.B * KE) * nd + d;
    const int q0 = part * (b.B / NP), q1 = q0 + b.B / NP;
    int qcur = q0;
    for (int c = 0; c < most; c += CH) {
        __syncthreads();
        for (int k = tid; k < NP * CH; k += blockDim.x) {
            const int pt = k / CH, li = k % CH, l = start[pt * QP] + c + li;
            if (l < start[(pt + 1) * QP]) {
                sg.l[pt][li] = load_line(g, l);
                const float il = g.ilf[l];
                sg.q[pt][li] = (int)il - i0;
                box_weights(b, ((il - (float)i0) + g.frac[l] - b.ctr) * b.invh, sg.w[pt][li]);
            }
        }
        __syncthreads();
        const int c0 = lo + c, n = live ? min(CH, hi - c0) : 0;
        for (int lb = 0; lb < n; lb += kBoxBatch) {
            // the batch's weights first: their table loads are independent and overlap
            float4 w[kBoxBatch];
            int cls[kBoxBatch];
#pragma unroll
            for (int m = 0; m < kBoxBatch; ++m)
                cls[m] = lb + m < n ? (info[c0 + lb + m].amask >> shift) & 7 : kBoxClasses;
#pragma unroll
            for (int m = 0; m < kBoxBatch; ++m) {
                const int li = min(lb + m, n - 1);
                float4 cw;
                float3 gb;
                box_series<false>(g, b, sg.l[part][li], c0 + li, d, dc, w[m], cw, gb);
            }
#pragma unroll
            for (int m = 0; m < kBoxBatch; ++m) {
                if (lb + m >= n) break;
                // the sums of the grid indices before this line's are complete
                const int q = sg.q[part][lb + m];
                for (; qcur < q; ++qcur)
#pragma unroll
                    for (int k = 0; k < KE; ++k) {
                        PM[((int64_t)qcur * KE + k) * nd] = pm[k];
                        pm[k] = 0.0f;
                    }
                if (cls[m] >= kBoxClasses) continue;
                float v[kBoxK];
#pragma unroll
                for (int k = 0; k < kBoxK; ++k) {
                    const float4 W = sg.w[part][lb + m][k];
                    v[k] = fmaf(w[m].w, W.w, fmaf(w[m].z, W.z, fmaf(w[m].y, W.y, w[m].x * W.x)));
                    if (k < KE) pm[k] += v[k];
                }
                if (cls[m] == 0) {
#pragma unroll
                    for (int k = 0; k < kBoxK; ++k) S.acc[k] += v[k];
                } else {
                    float *sc = s_cls + ((part * 3 + cls[m] - 1) * kBoxK) * nd + d;
#pragma unroll
                    for (int k = 0; k < kBoxK; ++k) sc[k * nd] += v[k];
                }
            }
        }
        S.fold();
    }
    if (live) {
        for (; qcur < q1; ++qcur)
#pragma unroll
            for (int k = 0; k < KE; ++k) {
                PM[((int64_t)qcur * KE + k) * nd] = pm[k];
                pm[k] = 0.0f;
            }
#pragma unroll
        for (int k = 0; k < kBoxK; ++k) s_m[(part * kBoxK + k) * nd + d] = S.get(k);
    }
    __syncthreads();
    if (!live) return;
    // sets by class, each with the classes below it
    float *M = b.M + ((int64_t)sl * b.nbox + box) * kBoxClasses * kBoxK * nd + d;
    for (int k = part; k < kBoxK; k += NP) {
        float m = 0.0f;
#pragma unroll
        for (int q = 0; q < NP; ++q) m += s_m[(q * kBoxK + k) * nd + d];
        M[(int64_t)k * nd] = m;
        for (int c = 1; c < kBoxClasses; ++c) {
#pragma unroll
            for (int q = 0; q < NP; ++q) m += s_cls[((q * 3 + c - 1) * kBoxK + k) * nd + d];
            M[((int64_t)c * kBoxK + k) * nd] = m;
        }
    }
}

// One offset's share of an expansion: out[j] += sum_k C[k][j] in[k] (TRANS: out[k] += sum_j
// C[k][j] in[j]), k + j <= P.  The inputs are read from global memory, layer stride nd.
template <int P, bool TRANS>
__device__ __forceinline__ void box_translate(const float *C, const float *in, int64_t nd, float (&out)[kBoxK]) {
    float v[P + 1];
#pragma unroll
    for (int k = 0; k <= P; ++k) v[k] = in[k * nd];
    // small terms first: the largest products (k = 0) join last
#pragma unroll
    for (int k = P; k >= 0; --k) {
        float c[kBoxRow];
        const float4 *row = reinterpret_cast<const float4 *>(C + k * kBoxRow);
#pragma unroll
        for (int q = 0; q <= (P - k) / 4; ++q) {
            const float4 x = __ldg(row + q);
            c[4 * q] = x.x;
            c[4 * q + 1] = x.y;
            c[4 * q + 2] = x.z;
            c[4 * q + 3] = x.w;
        }
#pragma unroll
        for (int j = P - k; j >= 0; --j) {
            if (TRANS)
                out[k] = fmaf(c[j], v[j], out[k]);
            else
                out[j] = fmaf(c[j], v[k], out[j]);
        }
    }
}

template <bool TRANS>
__device__ __forceinline__ void box_translate_at(int P, const float *C, const float *in, int64_t nd,
                                                 float (&out)[kBoxK]) {
    switch (P) {
        case 3: box_translate<3, TRANS>(C, in, nd, out); break;
        case 4: box_translate<4, TRANS>(C, in, nd, out); break;
        case 5: box_translate<5, TRANS>(C, in, nd, out); break;
        case 6: box_translate<6, TRANS>(C, in, nd, out); break;
        case 7: box_translate<7, TRANS>(C, in, nd, out); break;
        case 8: box_translate<8, TRANS>(C, in, nd, out); break;
        case 9: box_translate<9, TRANS>(C, in, nd, out); break;
        case 10: box_translate<10, TRANS>(C, in, nd, out); break;
        case 11: box_translate<11, TRANS>(C, in, nd, out); break;
        default: box_translate<13, TRANS>(C, in, nd, out); break;
    }
}

// Window ends of target box t at one layer: the part of one of the boxes omax + 1 and omax + 2 on either
// side (end: side and box) that the windows of the target's points reach, into out[r row].  The
// indices are added in the order in which the windows reach them, so a line beyond a point's window
// leaves no rounding there however strong it is (a difference of prefixes left 6e-8 of the line).
template <int KE>
__device__ __forceinline__ void box_ends(const BoxArgs &b, const float *PM, int nd, int t, int end, float *out, int row) {
    const bool left = end >> 1;                // lines left of the points
    const int e = end & 1, B = b.B;
    const int s = t + (left ? -1 : 1) * (b.omax + 1 + e) - b.s_lo;
    for (int r = 0; r < B; ++r) out[r * row] = 0.0f;
    if (s < 0 || s >= b.nbox) return;
    const float *m = PM + (int64_t)s * B * KE * nd, *E = b.E + (size_t)end * B * KE;
    float P[KE];
#pragma unroll
    for (int k = 0; k < KE; ++k) P[k] = 0.0f;
    auto put = [&](int r) {
        float v = 0.0f;
#pragma unroll
        for (int k = 0; k < KE; ++k) v = fmaf(__ldg(E + r * KE + k), P[k], v);
        out[r * row] = v;
    };
    // point r reaches the indices q <= r + rem - 1 - e B of a box to its right, q >= r - rem + 1 + e B to its left
    const int off = e * B + 1 - b.rem;
#pragma unroll 4
    for (int j = 0; j < B; ++j) {
        const int q = left ? B - 1 - j : j;
#pragma unroll
        for (int k = 0; k < KE; ++k) P[k] += m[((int64_t)q * KE + k) * nd];
        const int r = left ? q - off : q + off;
        if (r >= 0 && r < B) put(r);
    }
    // points whose window holds the whole box
    if (left)
        for (int r = min(B - 1, -off - 1); r >= 0; --r) put(r);
    else
        for (int r = max(0, B + off); r < B; ++r) put(r);
}

// Far field of a target box, added to the near-core sums.  kBoxSplit threads share a layer: each
// takes every kBoxSplit-th offset, then every kBoxSplit-th point (one thread per layer left a
// single spectrum's few boxes waiting on the chain of table and moment loads).  Bound by the latency
// of those loads: 96 registers let two blocks of nine warps (72 layers) share an SM, where the 102
// of the free choice left one (two stars on 43,000 lines: forward lines 2.38 -> 2.19 ms; 72
// registers and three blocks spill and slow short grids, 0.419 -> 0.429 ms on 2,200 points).
static size_t box_field_smem(int B, int nd) {
    return sizeof(float) * kBoxSplit * ((size_t)kBoxK * nd + (size_t)B * (nd + 1));
}
template <int KE>
__global__ void __maxnreg__(96) k_box_field(LineArgs gq, BoxArgs b) {
    extern __shared__ float smem_f[];         // [kBoxSplit][kBoxK][nd], then [kBoxSplit][B][nd + 1]
    const int sl = blockIdx.y, st = b.stars[sl], t = b.tgt0 + blockIdx.x;
    const LineArgs g = star_view(gq, st);
    const int nd = g.nd, part = threadIdx.x / nd, d = threadIdx.x - part * nd;
    const bool live = part < kBoxSplit;
    const int row = nd + 1, pts = b.B * row;
    float *s_phi = smem_f, *s_out = smem_f + kBoxSplit * kBoxK * nd;   // s_out: window ends, then the field
    if (live) box_ends<KE>(b, b.PM + (int64_t)sl * b.nbox * b.B * KE * nd + d, nd, t, part, s_out + part * pts + d, row);
    if (live) {
        const int4 nm = *reinterpret_cast<const int4 *>(b.nmin + ((int64_t)st * gq.nslab + d / b.DS) * 4);
        const float *Mst = b.M + (int64_t)sl * b.nbox * kBoxClasses * kBoxK * nd + d;
        BoxSum S;
        S.clear();
        int n = 0;
        for (int o = b.omax - part; o >= 3; o -= kBoxSplit, ++n) {
            const int cls = o >= nm.w ? 3 : o >= nm.z ? 2 : o >= nm.y ? 1 : 0;
            if (o < nm.x) break;
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const int s = t + (side ? -o : o) - b.s_lo;
                if (s >= 0 && s < b.nbox)
                    box_translate_at<false>(box_order(o), b.C + ((size_t)side * (b.omax + 3) + o) * kBoxK * kBoxRow,
                                            Mst + ((int64_t)s * kBoxClasses + cls) * kBoxK * nd, nd, S.acc);
            }
            if ((n & 3) == 3 || o < 12) S.fold();
        }
#pragma unroll
        for (int j = 0; j < kBoxK; ++j) s_phi[(part * kBoxK + j) * nd + d] = S.get(j);
    }
    __syncthreads();
    if (live) {
        float phi[kBoxK];
#pragma unroll
        for (int j = 0; j < kBoxK; ++j) {
            phi[j] = s_phi[j * nd + d];
#pragma unroll
            for (int q = 1; q < kBoxSplit; ++q) phi[j] += s_phi[(q * kBoxK + j) * nd + d];
        }
        for (int r = part; r < b.B; r += kBoxSplit) {
            const float x = ((float)r - b.ctr) * b.invh;
            float *out = s_out + r * row + d;
            const float v = (out[0] + out[pts]) + (out[2 * pts] + out[3 * pts]);
            float T[kBoxK], s = 0.0f;
            box_cheb(x, T);
#pragma unroll
            for (int j = kBoxK - 1; j >= 0; --j) s = fmaf(phi[j], T[j], s);
            out[0] = v + s;
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < b.B * nd; k += blockDim.x) {
        const int dl = k / b.B, col = k - dl * b.B;
        const int64_t i = (int64_t)t * b.B + col;
        if (i < g.ld) g.knear[(int64_t)dl * g.ld + i] += s_out[col * row + dl];
    }
}

// Chebyshev moments of G stim over the points of a target box: thread = layer.
__global__ void __launch_bounds__(128) k_box_gmoments(LineArgs gq, BoxArgs b) {
    extern __shared__ float s_g[];            // [nd][B + 1]
    const int d = threadIdx.x, sl = blockIdx.y, st = b.stars[sl], t = blockIdx.x;
    const LineArgs g = star_view(gq, st);
    for (int k = threadIdx.x; k < b.B * g.nd; k += blockDim.x) {
        const int row = k / b.B, col = k - row * b.B;
        const int64_t i = (int64_t)t * b.B + col;
        s_g[row * (b.B + 1) + col] = i < g.nlam ? g.Gt[(int64_t)row * g.ld + i] : 0.0f;
    }
    __syncthreads();
    if (d >= g.nd) return;
    float n[kBoxK];
#pragma unroll
    for (int j = 0; j < kBoxK; ++j) n[j] = 0.0f;
    for (int r = 0; r < b.B; ++r) {
        float T[kBoxK];
        box_cheb(((float)r - b.ctr) * b.invh, T);
        const float v = s_g[d * (b.B + 1) + r];
#pragma unroll
        for (int j = 0; j < kBoxK; ++j) n[j] = fmaf(v, T[j], n[j]);
    }
    float *N = b.N + ((int64_t)sl * b.ntb + t) * kBoxK * g.nd + d;
#pragma unroll
    for (int j = 0; j < kBoxK; ++j) N[(int64_t)j * g.nd] = n[j];
}

constexpr int kBoxGradWarps = 8;
constexpr int kBoxGradSplit = 4;          // a warp's unit: 32 lines x a quarter of the layers

// row of the window-end sums of one layer: [KE][B + 1] floats, odd length
__host__ __device__ __forceinline__ int box_zrow(int B, int KE) { return (KE * (B + 1)) | 1; }
// nd: layers of the block
static size_t box_grad_smem(int B, int KE, int nd) {
    const size_t ends = (size_t)nd * box_zrow(B, KE) + (size_t)2 * nd * (B + 1), copies = (size_t)2 * kBoxClasses * kBoxK * nd;
    return sizeof(float) * ((size_t)kBoxClasses * kBoxK * nd + (ends > copies ? ends : copies));
}

// Block = box (x), star (y) and part of the layers (z; one part where the grid has boxes enough).
// Per-line sums of one source box over the boxes of its window: strength and van der Waals damping,
// FOUR: the radiative and Stark damping too.
template <int KE, bool FOUR>
__global__ void __launch_bounds__(32 * kBoxGradWarps) k_box_grad(LineArgs gq, BoxArgs b) {
    extern __shared__ float smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int box = blockIdx.x, sl = blockIdx.y, st = b.stars[sl];
    const LineArgs g = star_view(gq, st);
    const int32_t *start = gq.bstart + (int64_t)st * gq.brow + kBoxSplit * (b.box0 + box);
    const int lo = start[0], hi = start[kBoxSplit];
    if (lo >= hi) return;
    // the block's layers dz .. dz + nd
    const int nz = gridDim.z, dz = (int)blockIdx.z * g.nd / nz, nd = ((int)blockIdx.z + 1) * g.nd / nz - dz;
    const int64_t gnd = g.nd;
    const int zrow = box_zrow(b.B, KE);
    float *s_psi = smem;                                   // [class][k][nd]
    float *s_z = s_psi + (size_t)kBoxClasses * kBoxK * nd; // [nd][zrow]: [k][q]
    float *s_g = s_z + (size_t)nd * zrow;                  // [2][nd][B + 1]: G of two target boxes
    const int s = b.s_lo + box, i0 = s * b.B;
    // Psi_k: offsets from the widest in, a copy kept where a class begins; np threads share a layer,
    // each taking every np-th offset, their copies added in order afterwards
    const int np = min(3, 32 * kBoxGradWarps / nd), part = tid / nd, d = tid - part * nd;
    if (part < np) {
        const int4 nm = *reinterpret_cast<const int4 *>(b.nmin + ((int64_t)st * gq.nslab + (dz + d) / b.DS) * 4);
        const float *Nst = b.N + (int64_t)sl * b.ntb * kBoxK * gnd + dz + d;
        float *mine = part == 0 ? s_psi : s_z + (size_t)(part - 1) * kBoxClasses * kBoxK * nd;
        BoxSum S;
        S.clear();
        int o = b.omax - part, n = 0;
#pragma unroll
        for (int c = kBoxClasses - 1; c >= 0; --c) {
            const int nc = c == 3 ? nm.w : c == 2 ? nm.z : c == 1 ? nm.y : nm.x;
            for (; o >= nc; o -= np, ++n) {
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    const int t = s + (side ? o : -o);
                    if (t >= 0 && t < b.ntb)
                        box_translate_at<true>(box_order(o), b.C + ((size_t)side * (b.omax + 3) + o) * kBoxK * kBoxRow,
                                               Nst + (int64_t)t * kBoxK * gnd, gnd, S.acc);
                }
                if ((n & 3) == 3 || o < 12) S.fold();
            }
#pragma unroll
            for (int k = 0; k < kBoxK; ++k) mine[(c * kBoxK + k) * nd + d] = S.get(k);
        }
    }
    __syncthreads();
    for (int k = tid; k < kBoxClasses * kBoxK * nd; k += blockDim.x)
        for (int q = 1; q < np; ++q) s_psi[k] += s_z[(size_t)(q - 1) * kBoxClasses * kBoxK * nd + k];
    // window ends: Z_k(q) = sum of E_k G over the points that the window of a line at index q reaches
    for (int side = 0; side < 2; ++side) {
        __syncthreads();
        for (int k = tid; k < 2 * nd * b.B; k += blockDim.x) {
            const int e = k / (nd * b.B), kk = k - e * nd * b.B, row = kk / b.B, col = kk - row * b.B;
            const int t = side ? s + b.omax + 1 + e : s - b.omax - 1 - e;
            const int64_t i = (int64_t)t * b.B + col;
            s_g[(e * nd + row) * (b.B + 1) + col] = (t >= 0 && i < g.nlam) ? g.Gt[(int64_t)(dz + row) * g.ld + i] : 0.0f;
        }
        __syncthreads();
        // thread = (layer, moment): the points' G times E_k, running over the lines' indices q
        for (int u = tid; u < nd * KE; u += blockDim.x) {
            const int k = u / nd, dl = u - k * nd;
            const float *E0 = b.E + (size_t)side * 2 * b.B * KE + k, *E1 = E0 + (size_t)b.B * KE;
            const float *g0 = s_g + dl * (b.B + 1), *g1 = s_g + (nd + dl) * (b.B + 1);
            float *zr = s_z + dl * zrow + k * (b.B + 1);
            float z = 0.0f;
            if (side == 0) {
                // points left of the line, box s - omax - 1 - e: r >= q - rem + 1 + e B, q downwards
                int r0 = b.B - 1, r1 = b.B - 1;
                for (int q = b.B - 1; q >= 0; --q) {
                    for (; r0 >= max(q - b.rem + 1, 0); --r0) z = fmaf(__ldg(E0 + r0 * KE), g0[r0], z);
                    for (; r1 >= max(q - b.rem + 1 + b.B, 0); --r1) z = fmaf(__ldg(E1 + r1 * KE), g1[r1], z);
                    zr[q] = z;
                }
            } else {
                // points right of it, box s + omax + 1 + e: r <= q + rem - 1 - e B, q upwards
                int r0 = 0, r1 = 0;
                for (int q = 0; q < b.B; ++q) {
                    for (; r0 <= min(q + b.rem - 1, b.B - 1); ++r0) z = fmaf(__ldg(E0 + r0 * KE), g0[r0], z);
                    for (; r1 <= min(q + b.rem - 1 - b.B, b.B - 1); ++r1) z = fmaf(__ldg(E1 + r1 * KE), g1[r1], z);
                    zr[q] += z;
                }
            }
        }
    }
    __syncthreads();
    // lane = line; a unit is 32 lines at a quarter of the layers
    const int nch = (hi - lo + 31) / 32;
    for (int u = warp; u < nch * kBoxGradSplit; u += kBoxGradWarps) {
        const int l = lo + (u / kBoxGradSplit) * 32 + lane, part = u % kBoxGradSplit;
        if (l >= hi) continue;
        const LineScalars L = load_line(g, l);
        const float il = g.ilf[l];
        const int q = (int)il - i0;
        float4 W[kBoxK];
        box_weights(b, ((il - (float)i0) + g.frac[l] - b.ctr) * b.invh, W);
        float S1 = 0.0f, S2 = 0.0f, S3 = 0.0f, S4 = 0.0f;
        const int d1 = (part + 1) * nd / kBoxGradSplit;
        for (int dd = part * nd / kBoxGradSplit; dd < d1; ++dd) {
            const int da = dz + dd, grp = da / b.DC;
            const int cls = (gq.finfo[(int64_t)grp * gq.nl + l].amask >> (16 + 3 * ((da - grp * b.DC) / b.DS))) & 7;
            if (cls >= kBoxClasses) continue;
            float4 F = make_float4(0.f, 0.f, 0.f, 0.f);
            const float *psi = s_psi + cls * kBoxK * nd + dd, *z = s_z + dd * zrow + q;
#pragma unroll
            for (int k = kBoxK - 1; k >= 0; --k) {
                float v = psi[k * nd];
                if (k < KE) v += z[k * (b.B + 1)];
                F.x = fmaf(W[k].x, v, F.x);
                F.y = fmaf(W[k].y, v, F.y);
                F.z = fmaf(W[k].z, v, F.z);
                F.w = fmaf(W[k].w, v, F.w);
            }
            float4 w, c;
            float3 gb;
            box_series<true>(g, b, L, l, da,
                             make_float4(__ldg(g.beta_hi + da), __ldg(g.beta_lo + da), __ldg(g.ne + da), __ldg(g.npert + da)),
                             w, c, gb);
            S1 += fmaf(w.w, F.w, fmaf(w.z, F.z, fmaf(w.y, F.y, w.x * F.x)));
            const float Y = fmaf(c.w, F.w, fmaf(c.z, F.z, fmaf(c.y, F.y, c.x * F.x)));
            S2 = fmaf(gb.x, Y, S2);
            if (FOUR) {
                S3 = fmaf(gb.y, Y, S3);
                S4 = fmaf(gb.z, Y, S4);
            }
        }
        atomicAdd(gq.gacc + l, (double)S1);
        atomicAdd(gq.gacc + gq.nl + l, (double)S2);
        if (FOUR) {
            atomicAdd(gq.gacc + far_row(2) * gq.nl + l, (double)S3);
            atomicAdd(gq.gacc + far_row(3) * gq.nl + l, (double)S4);
        }
    }
}

}  // namespace pz
