// FP64 form: near-field entries and touching pairs at many frequencies by
// separated sums.
//
// An entry is sum_q w_q g(r_q) e^{-sigma_k r_q} over the point pairs q of two
// triangles (regular pairs 49 points, touching pairs up to 2 ng^4), and the
// FP64 near-field tensor holds it at every unique frequency k.  The distances of a
// regular pair span a short interval, r_q in [r0, r0 + 2D], r0 the smallest
// distance and D the sum of two triangle radii.  With u = (r - r0)/D - 1 in
// [-1, 1] and z = sigma D,
//     e^{-sigma r} = e^{-sigma r0} sum_m c_m(z) T_m(u),
// c_m the Chebyshev coefficients of e^{-z (u + 1)}, so that
//     entry(k) = e^{-sigma_k r0} sum_m c_m(z_k) M_m,   M_m = sum_q w_q g(r_q) T_m(u_q):
// the moments M_m are real, hold no frequency and are formed once per pair,
// and a frequency costs one complex exponential and m real x complex
// multiply-adds instead of one exponential per point pair.  The double-layer
// kernels (1 + sigma r) e^{-sigma r} = e^{-sigma r0} [(1 + sigma r0) + z (u + 1)] e^{-z(u+1)}
// take a second coefficient set for z (u + 1) e^{-z (u + 1)} on the same moments.
// Touching pairs have r in [0, 2D], D the longest edge, and two such sums, over
// [0, D/2] and [D/2, 2D]: most of a vertex pair's points lie at large r, where
// e^{-sigma r} may be small against its value 1 at r = 0, and one sum over the
// whole interval would round relative to that 1 (touching pairs of a
// 2640-triangle housing: 1.7e-14 of the sum of moduli instead of 6e-15).
//
// Accuracy: |c_m| <= 2 and the expanded function is at most 1 on the interval,
// 1 at the nearest point, so the sums lose little against the sum of the
// entry's moduli; the tail dropped is below 2^-57.  Measured against a 64-bit
// evaluation, all near-field entries of a strip: 5.8e-16 (direct sums: 5.6e-16) on
// the 1280-triangle sphere, 3.8e-16 (3.0e-16) on a 2640-triangle housing.
//
// What bounds it: the FP64 pipe (1/74 of the FP32 rate).  The direct sums take
// about 75 FP64 operations per point pair and frequency (square root and
// division shared by 4 frequencies); here a frequency takes 2 m + 80 and an
// entry's moments 49 x (30 + 3 m), m = 16..40.  1280-triangle sphere, 33
// frequencies: near field 93 -> 11 ms, touching pairs 34 -> 3.5 ms.
//
// The mixed form does not use them: its near field evaluates only the
// frequencies that Algorithm 1 selects (k_near_aca), a few of all.
#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.h"
#include "kernels.h"
#include "pair.cuh"

namespace {

constexpr int kNodes = 64;  // Chebyshev nodes of the coefficient sums

constexpr double kSepTol = 6.938893903907228e-18;  // 2^-57: coefficient tail dropped

// Coefficients of one frequency per block on r = left + half (u + 1): f = e^{-w},
// w = sigma r, and
//   kind 0: f;  kind 1: f and w f (two sets);  kind 2: (1 + w) f.
// by the discrete cosine sum over 64 Chebyshev nodes (aliasing c_{128 - m} is
// far below rounding for m < 64).  Written to the terms first .. first + P - 1
// of the layout near [i][set][stride] or touching [stride][n] (frequencies
// contiguous); pk[2 i] / pk[2 i + 1] = terms kept of the first / second
// interval, multiples of 4.
// A frequency index outside [0, nq) is left out.
__global__ void __launch_bounds__(kNodes) k_sep_coef(const double *sig, int nq, const int *klist, int n, double left,
                                                     double half, int P, int kind, int by_term, int stride, int first,
                                                     c64 *coef, int *pk) {
    __shared__ double ct[4 * kNodes];
    __shared__ c64 F[2][kNodes];
    __shared__ double mag[kNodes];
    const int i = blockIdx.x, j = threadIdx.x, k = klist[i];
    if (k < 0 || k >= nq) return;
    for (int e = j; e < 4 * kNodes; e += kNodes) ct[e] = cospi((double)e / (2 * kNodes));
    __syncthreads();
    const double r = fma(half, ct[2 * j + 1] + 1.0, left);  // u = cos(pi (j + 1/2) / 64)
    const double wr = sig[2 * k] * r, wi = sig[2 * k + 1] * r;
    const c64 f = expm_sr(wr, wi, 1.0);
    const c64 wf = {wr * f.x - wi * f.y, wr * f.y + wi * f.x};
    F[0][j] = kind == 2 ? f + wf : f;
    F[1][j] = wf;
    __syncthreads();
    const int nb = kind == 1 ? 2 : 1;
    double a = 0.0;
    if (j < P) {
        for (int b = 0; b < nb; ++b) {
            c64 c = {0.0, 0.0};
            for (int q = 0; q < kNodes; ++q) {
                const double t = ct[(j * (2 * q + 1)) & (4 * kNodes - 1)];
                c.x = fma(t, F[b][q].x, c.x);
                c.y = fma(t, F[b][q].y, c.y);
            }
            const double s = (j ? 2.0 : 1.0) / kNodes;
            c = c64{s * c.x, s * c.y};
            a += fabs(c.x) + fabs(c.y);
            const int64_t o = by_term ? (int64_t)(first + j) * n + i : ((int64_t)i * nb + b) * stride + first + j;
            coef[o] = c;
        }
    }
    mag[j] = a;
    __syncthreads();
    if (j == 0 && pk) {
        double tail = 0.0;
        int p = P;
        while (p > 1 && tail + mag[p - 1] <= kSepTol) tail += mag[--p];
        pk[2 * i + (first > 0)] = min(P, (p + 3) & ~3);
    }
}

// Difference d = y - x of test point a (registers) and a trial point, and |d|^2.
struct Point {
    double x, y, z, w;
};
TD_D Point load_point(const MeshDev &m, int o) { return Point{m.qx[o], m.qy[o], m.qz[o], m.qw[o]}; }
TD_D double diff2(const TestD &X, int a, const Point &p, double *d) {
    d[0] = p.x - X.x[a];
    d[1] = p.y - X.y[a];
    d[2] = p.z - X.z[a];
    return d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
}
// w / r (single layer) or w dn / r^3, and r
template <int OP>
TD_D double over_r(double w, double dn, double r2, double &r) {
    double ri;
    r = sqrt_inv(r2, ri);
    return OP == TD_SLP ? w * ri : w * dn * (ri * ri * ri);
}

// Adds the moments of test triangle X and trial triangle tj to M: P terms over
// [r0, r0 + 2D] (P1 = 0), or P1 terms over [r0, r0 + D/2] and P over the rest.
template <int OP, int P1, int P>
TD_D void add_moments(const TestD &X, const MeshDev &m, int tj, int loc, double r0, double D, double *M) {
    double nx = 0.0, ny = 0.0, nz = 0.0;  // signed kernel normal: -n_y (DLP), +n_x (ADLP)
    if (OP == TD_DLP) {
        nx = -m.n64[tj];
        ny = -m.n64[m.nt + tj];
        nz = -m.n64[2 * m.nt + tj];
    } else if (OP == TD_ADLP) {
        nx = X.nx;
        ny = X.ny;
        nz = X.nz;
    }
    const double inv1 = (P1 ? 4.0 : 1.0) / D, inv2 = (4.0 / 3.0) / D, cut = 0.5 * D;
#pragma unroll 1
    for (int b = 0; b < 7; ++b) {
        const Point p = load_point(m, b * m.nt + tj);
        const double wyb = p.w * (OP == TD_DLP ? bary7d(b, loc) : 1.0);
#pragma unroll
        for (int a = 0; a < 7; ++a) {
            double d[3], r;
            const double r2 = diff2(X, a, p, d);
            const double w = over_r<OP>(X.w[a] * wyb, d[0] * nx + d[1] * ny + d[2] * nz, r2, r);
            // T_{m+1} + T_m = 2 (1 + u) T_m - (T_m + T_{m-1}): keeps full accuracy at
            // u = -1, the nearest points, where e^{-sigma r} is largest
            const double t = r - r0;
            const bool inner = P1 > 0 && t < cut;
            const double v = P1 == 0 || inner ? t * inv1 : (t - cut) * inv2, v2 = v + v;
            const double wi = inner ? w : 0.0, wo = inner ? 0.0 : w;
            double tn = v - 1.0, dn = v;
            if (P1 > 0) {
                M[0] += wi;
                M[1] = fma(wi, tn, M[1]);
            }
            M[P1] += wo;
            M[P1 + 1] = fma(wo, tn, M[P1 + 1]);
#pragma unroll
            for (int q = 2; q < P; ++q) {
                dn = fma(v2, tn, -dn);
                tn = dn - tn;
                if (q < P1) M[q] = fma(wi, tn, M[q]);
                M[P1 + q] = fma(wo, tn, M[P1 + q]);
            }
        }
    }
}

// sum_m c[m] M[m] over the first p1 terms of the first interval and p2 of the
// second (multiples of 4; uniform); c in shared memory, 16-byte aligned
template <int P1, int P>
TD_D c64 term_sum(const c64 *c, const double *M, int p1, int p2) {
    c64 s = {0, 0}, s2 = {0, 0};
#pragma unroll
    for (int q = 0; q < P1 + P; q += 4) {
        if (P1 > 0 && q >= P1 ? q - P1 < p2 : q < p1) {
#pragma unroll
            for (int e = q; e < q + 4; e += 2) {
                const c64 a = c[e], b = c[e + 1];
                s.x = fma(a.x, M[e], s.x);
                s.y = fma(a.y, M[e], s.y);
                s2.x = fma(b.x, M[e + 1], s2.x);
                s2.y = fma(b.y, M[e + 1], s2.y);
            }
        }
    }
    return s + s2;
}

constexpr int kSepSmem = 40 * 1024;  // coefficients and frequencies in shared memory at a time
constexpr int kSlots = 12;           // touching slots of an entry kept (a longer list is searched again)

// near[noff[b] + (k nI + i) nJ + j] at the separated frequencies; one thread
// per entry, consecutive threads on consecutive columns (coalesced stores).
// `seg` frequencies have their coefficients in shared memory at a time; the
// moments of an entry are formed once per segment.
template <int OP, int P1, int P>
__global__ void __launch_bounds__(128) k_near_sep(MeshDev m, NearArgs a, SepSet s, const c64 *table, int seg) {
    constexpr int NB = OP == TD_SLP ? 1 : 2, NV = TD_P1_TRIAL(OP) ? 3 : 1, PT = P1 + P;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c64 *cf = reinterpret_cast<c64 *>(smem_raw);
    c64 *sg = cf + seg * NB * PT;
    int4 *kp = reinterpret_cast<int4 *>(sg + seg);  // frequency, terms of both intervals
    const int nf = a.nf;
    const double D = s.D;
    for (int k0 = 0; k0 < s.nsep; k0 += seg) {
        const int ns = min(seg, s.nsep - k0);
        __syncthreads();
        for (int e = threadIdx.x; e < ns * NB * PT; e += blockDim.x)
            cf[e] = s.coef[(int64_t)k0 * NB * PT + e];
        for (int e = threadIdx.x; e < ns; e += blockDim.x) {
            const int k = s.klist[k0 + e];
            kp[e] = make_int4(k, s.pk[2 * (k0 + e)], s.pk[2 * (k0 + e) + 1], 0);
            sg[e] = c64{a.sig[2 * k], a.sig[2 * k + 1]};
        }
        __syncthreads();
        for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < a.nentries;
             t += (int64_t)gridDim.x * blockDim.x) {
            int lo = 0, hi = a.nnear - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (a.eprefix[mid] <= t) lo = mid; else hi = mid - 1;
            }
            const int32_t *bl = a.blocks + 5 * a.near_ids[lo];
            const int nI = bl[1] - bl[0], nJ = bl[3] - bl[2];
            const int le = (int)(t - a.eprefix[lo]);
            const int i = le / nJ, j = le - i * nJ;
            const int row = a.perm_r[bl[0] + i], col = a.perm_c[bl[2] + j];
            c64 *dst = (c64 *)a.near + a.noff[lo] + le;
            const int64_t fstride = (int64_t)nI * nJ;
            // supports: touching ones keep their table slot, the others give the
            // smallest distance
            int slots[TD_P1_TRIAL(OP) ? kSlots : 1], nslot = 0;
            const int p0 = TD_P1_TRIAL(OP) ? m.v2t_ptr[col] : 0, p1 = TD_P1_TRIAL(OP) ? m.v2t_ptr[col + 1] : 1;
            TestD X;
            load_test(m, row, X);
            double r2m = -1.0;
            for (int p = p0; p < p1; ++p) {
                const int e = TD_P1_TRIAL(OP) ? m.v2t[p] : col;
                const int slot = touching_slot(m, row, e);
                if (slot >= 0) {
                    if (!TD_P1_TRIAL(OP)) slots[0] = slot;
                    else if (nslot < kSlots) slots[nslot] = slot * 3 + m.v2t_loc[p];
                    ++nslot;
                    continue;
                }
                double best = r2m < 0.0 ? 1e300 : r2m;
#pragma unroll 1
                for (int b = 0; b < 7; ++b) {
                    const Point pt = load_point(m, b * m.nt + e);
#pragma unroll
                    for (int q = 0; q < 7; ++q) {
                        double d[3];
                        best = fmin(best, diff2(X, q, pt, d));
                    }
                }
                r2m = best;
            }
            const bool reg = r2m >= 0.0;
            double r0 = 0.0;
            double M[PT];
#pragma unroll
            for (int q = 0; q < PT; ++q) M[q] = 0.0;
            if (reg) {
                over_r<TD_SLP>(1.0, 0.0, r2m, r0);
                for (int p = p0; p < p1; ++p) {
                    const int e = TD_P1_TRIAL(OP) ? m.v2t[p] : col;
                    if (TD_P1_TRIAL(OP) && nslot > 0 && touching_slot(m, row, e) >= 0) continue;
                    add_moments<OP, P1, P>(X, m, e, TD_P1_TRIAL(OP) ? m.v2t_loc[p] : 0, r0, D, M);
                }
                const double inv4pi = 1.0 / TD_FOUR_PI;
#pragma unroll
                for (int q = 0; q < PT; ++q) M[q] *= inv4pi;
            }
#pragma unroll 1
            for (int f = 0; f < ns; ++f) {
                const int4 kq = kp[f];
                const int k = kq.x;
                c64 v = {0, 0};
                if (reg) {
                    const c64 *c = cf + f * NB * PT;
                    v = term_sum<P1, P>(c, M, kq.y, kq.z);
                    if (OP != TD_SLP) {
                        const c64 sgm = sg[f];
                        const c64 o = {fma(sgm.x, r0, 1.0), sgm.y * r0};
                        v = o * v + term_sum<P1, P>(c + PT, M, kq.y, kq.z);
                    }
                    v = expm_sr(sg[f].x, sg[f].y, r0) * v;
                }
                if (nslot > 0) {
                    c64 sing = {0.0, 0.0};
                    if (!TD_P1_TRIAL(OP)) {
                        sing = table[(int64_t)slots[0] * nf + k];
                    } else if (nslot <= kSlots) {
                        for (int q = 0; q < nslot; ++q) {
                            const int sl = slots[q] / 3;
                            sing = sing + table[((int64_t)sl * nf + k) * NV + (slots[q] - 3 * sl)];
                        }
                    } else {
                        for (int p = p0; p < p1; ++p) {
                            const int sl = touching_slot(m, row, m.v2t[p]);
                            if (sl >= 0) sing = sing + table[((int64_t)sl * nf + k) * NV + m.v2t_loc[p]];
                        }
                    }
                    v = v + sing;
                }
                dst[k * fstride] = v;
            }
        }
    }
}

// ---- touching pairs -------------------------------------------------------------
// Reference points of the three classes (ss_ref), formed once per call.
__global__ void k_ss_rule(int ng, const double *gx, const double *gw, double *rule) {
    const int n1 = ss_npoints(1, ng), n2 = ss_npoints(2, ng), n3 = ss_npoints(3, ng);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n1 + n2 + n3; t += gridDim.x * blockDim.x) {
        const int cls = t < n1 ? 1 : t < n1 + n2 ? 2 : 3;
        const int q = cls == 1 ? t : cls == 2 ? t - n1 : t - n1 - n2, n = ss_npoints(cls, ng);
        double a[4], w, lam[3];
        ss_ref(cls, q, ng, gx, gw, a, w, lam);
        double *o = rule + ss_rule_off(cls, ng) + q;
        for (int e = 0; e < 4; ++e) o[(int64_t)e * n] = a[e];
        o[(int64_t)4 * n] = w;
        for (int e = 0; e < 3; ++e) o[(int64_t)(5 + e) * n] = lam[e];
    }
}

// A touching pair and its reference points; adds the lane's share of its moments
// (hat v of the trial triangle for P1 columns) to M (inner interval) and N.
struct SingPair {
    SingGeom G;
    SsEdges E;
    double nrm[3];  // signed kernel normal at d = y - x
    const double *rl;
    int nq;
};
template <int OP>
TD_D void sing_pair(const MeshDev &m, int ti, int tj, const double *rule, SingPair &S) {
    if (OP == TD_SLP && ti > tj) {
        const int t = ti;
        ti = tj;
        tj = t;
    }
    classify_pair(m, ti, tj, S.G);
    ss_edges(S.G, S.E);
    const double sn = OP == TD_DLP ? -1.0 : 1.0;
    const double *g = OP == TD_DLP ? S.G.ny : S.G.nx;
#pragma unroll
    for (int x = 0; x < 3; ++x) S.nrm[x] = sn * g[x];
    S.rl = rule + ss_rule_off(S.G.cls, m.ng);
    S.nq = OP != TD_SLP && S.G.cls == 3 ? 0 : ss_npoints(S.G.cls, m.ng);  // (flat panel: (x - y).n = 0)
}
template <int OP, int P1, int P2>
TD_D void sing_moments(const SingPair &S, int v, double D, double *M, double *N) {
    // intervals [0, D/2] (P1 terms) and [D/2, 2D] (P2 terms)
    const double cut = 0.5 * D, inv1 = 4.0 / D, inv2 = 4.0 / (3.0 * D);
    for (int q = threadIdx.x & 31; q < S.nq; q += 32) {
        double a[4], d[3], r;
#pragma unroll
        for (int e = 0; e < 4; ++e) a[e] = __ldg(S.rl + (int64_t)e * S.nq + q);
        ss_diff(S.G.cls, a, S.E, d);
        double w = over_r<OP>(__ldg(S.rl + (int64_t)4 * S.nq + q) * S.G.g, d[0] * S.nrm[0] + d[1] * S.nrm[1] + d[2] * S.nrm[2],
                              d[0] * d[0] + d[1] * d[1] + d[2] * d[2], r);
        if (TD_P1_TRIAL(OP)) w *= __ldg(S.rl + (int64_t)(5 + v) * S.nq + q);
        const bool inner = r < cut;
        const double v1 = inner ? r * inv1 : (r - cut) * inv2, v2 = v1 + v1;  // 1 + u
        const double wm = inner ? w : 0.0, wn = inner ? 0.0 : w;
        double tn = v1 - 1.0, dn = v1;  // as in add_moments
        M[0] += wm;
        M[1] = fma(wm, tn, M[1]);
        N[0] += wn;
        N[1] = fma(wn, tn, N[1]);
#pragma unroll
        for (int e = 2; e < P2; ++e) {
            dn = fma(v2, tn, -dn);
            tn = dn - tn;
            if (e < P1) M[e] = fma(wm, tn, M[e]);
            N[e] = fma(wn, tn, N[e]);
        }
    }
}
// sum_m c_m M_m of frequency i of n (all lanes hold the warp's sums)
template <int P1, int P2>
TD_D c64 sing_sum(const c64 *coef, int n, int i, const double *M, const double *N) {
    c64 a = {0.0, 0.0};
#pragma unroll
    for (int q = P1 + P2 - 1; q >= 0; --q) {  // outer interval first, large orders first
        const c64 c = coef[(int64_t)q * n + i];
        const double mq = q < P1 ? M[q < P1 ? q : 0] : N[q < P1 ? 0 : q - P1];
        a.x = fma(c.x, mq, a.x);
        a.y = fma(c.y, mq, a.y);
    }
    const double inv4pi = 1.0 / TD_FOUR_PI;
    return c64{a.x * inv4pi, a.y * inv4pi};
}

// Touching-pair table at the separated frequencies, one warp per pair: the
// lanes split the quadrature points, the moments are summed over the warp, and
// the lanes then take one frequency each.  P1 columns sweep the points once per
// hat (the moments of three hats do not fit in registers).
template <int OP, int P1, int P2>
__global__ void __launch_bounds__(128) k_sing_sep(MeshDev m, const int *pti, const int *ptj, int npairs,
                                                  const double *rule, SepSet s, int nf, c64 *table) {
    constexpr int NV = TD_P1_TRIAL(OP) ? 3 : 1;
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int p = warp; p < npairs; p += nwarps) {
        SingPair S;
        sing_pair<OP>(m, pti[p], ptj[p], rule, S);
        c64 *o = table + (int64_t)p * nf * NV;
#pragma unroll 1
        for (int v = 0; v < NV; ++v) {
            double M[P1], N[P2];
#pragma unroll
            for (int q = 0; q < P1; ++q) M[q] = 0.0;
#pragma unroll
            for (int q = 0; q < P2; ++q) N[q] = 0.0;
            sing_moments<OP, P1, P2>(S, v, s.D, M, N);
#pragma unroll
            for (int q = 0; q < P1; ++q) M[q] = warp_sum(M[q]);
#pragma unroll
            for (int q = 0; q < P2; ++q) N[q] = warp_sum(N[q]);
            for (int i = lane; i < s.nsep; i += 32)
                o[(int64_t)s.klist[i] * NV + (TD_P1_TRIAL(OP) ? S.G.loc[v] : 0)] = sing_sum<P1, P2>(s.coef, s.nsep, i, M, N);
        }
    }
}

// Touching part of tdbem_entries at many frequencies: adds it to the entries of
// out [nf][nr nc] that have one (either precision; the sums are FP64).  A warp
// looks at 32 entries and integrates the touching ones one after the other; all
// touching supports of a P1 column share the distance interval, so their moments
// are added before the frequencies are taken.  An invalid index was answered
// with NaN already.
template <class T, int OP, int P1, int P2>
__global__ void __launch_bounds__(128) k_entry_sing(MeshDev m, const double *rule, SepSet s, int nq, const int *rows,
                                                    int64_t nr, const int *cols, int64_t nc, cx<T> *out) {
    const int64_t nE = nr * nc, stride = (int64_t)gridDim.x * blockDim.x;
    const int ncols = TD_P1_TRIAL(OP) ? m.nv : m.nt, lane = threadIdx.x & 31;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < nE; base += stride) {
        const int64_t e = base + lane;
        int row = e < nE ? rows[e / nc] : -1, col = e < nE ? cols[e % nc] : -1;
        bool touch = false;
        if (row >= 0 && row < m.nt && col >= 0 && col < ncols) {
            if (!TD_P1_TRIAL(OP)) touch = touching_slot(m, row, col) >= 0;
            else
                for (int p = m.v2t_ptr[col]; p < m.v2t_ptr[col + 1] && !touch; ++p) touch = touching_slot(m, row, m.v2t[p]) >= 0;
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, touch); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int ti = __shfl_sync(0xffffffffu, row, src), tc = __shfl_sync(0xffffffffu, col, src);
            double M[P1], N[P2];
#pragma unroll
            for (int q = 0; q < P1; ++q) M[q] = 0.0;
#pragma unroll
            for (int q = 0; q < P2; ++q) N[q] = 0.0;
            const int p0 = TD_P1_TRIAL(OP) ? m.v2t_ptr[tc] : 0, p1 = TD_P1_TRIAL(OP) ? m.v2t_ptr[tc + 1] : 1;
#pragma unroll 1
            for (int p = p0; p < p1; ++p) {
                const int tj = TD_P1_TRIAL(OP) ? m.v2t[p] : tc, loc = TD_P1_TRIAL(OP) ? m.v2t_loc[p] : 0;
                if (TD_P1_TRIAL(OP) && touching_slot(m, ti, tj) < 0) continue;
                SingPair S;
                sing_pair<OP>(m, ti, tj, rule, S);
                sing_moments<OP, P1, P2>(S, S.G.loc[0] == loc ? 0 : S.G.loc[1] == loc ? 1 : 2, s.D, M, N);
            }
#pragma unroll
            for (int q = 0; q < P1; ++q) M[q] = warp_sum(M[q]);
#pragma unroll
            for (int q = 0; q < P2; ++q) N[q] = warp_sum(N[q]);
            for (int i = lane; i < s.nsep; i += 32) {
                const int k = s.klist[i];
                if (k < 0 || k >= nq) continue;
                const c64 a = sing_sum<P1, P2>(s.coef, s.nsep, i, M, N);
                cx<T> &o = out[(int64_t)i * nE + base + src];
                o = cx<T>{(T)((double)o.x + a.x), (T)((double)o.y + a.y)};
            }
        }
    }
}

// Kernel variants by |z| = |sigma| D.  A sum of P terms over an interval of
// half length h serves |sigma| h up to 1.15 (P = 16), 3.8 (24), 7.4 (32), 11.7 (40):
// the tail of the coefficients is at most 2 (|sigma| h / 2)^P / P! (purely
// imaginary sigma; less with a real part), bounded by 2^-56.  Two intervals
// have half lengths D/4 (P1 terms) and 3D/4 (P terms); one interval (P1 = 0)
// has D.  Touching pairs always take two.  Regular pairs take two for P1
// columns: the points nearest to the test triangle carry little of a hat
// function's weight, so one interval rounds relative to 1 where the sum is
// small (1280-triangle sphere, worst frequency: 8e-15 instead of 1e-15).
struct SepVariant {
    int P, P1;
    double zmax;
};
const SepVariant kOne[] = {{16, 0, 1.15}, {24, 0, 3.8}, {32, 0, 7.4}, {40, 0, 11.7}};
const SepVariant kTwo[] = {{24, 16, 4.6}, {40, 24, 15.2}};

const SepVariant *variant_for(int op, double z, bool touching) {
    const bool two = touching || TD_P1_TRIAL(op);
    const SepVariant *v = two ? kTwo : kOne;
    for (int i = 0; i < (two ? 2 : 4); ++i)
        if (z <= v[i].zmax) return v + i;
    return nullptr;
}

template <int OP, int P1, int P>
int launch_near(cudaStream_t st, const MeshDev &m, const NearArgs &a, const SepSet &s, const c64 *table, int num_sms) {
    constexpr int NB = OP == TD_SLP ? 1 : 2;
    const int per = (int)(NB * (P1 + P) * sizeof(c64) + sizeof(c64) + sizeof(int4));
    const int seg = std::min(s.nsep, std::max(1, kSepSmem / per));
    const int grid = (int)std::min<int64_t>((a.nentries + 127) / 128, (int64_t)num_sms * 16);
    k_near_sep<OP, P1, P><<<grid, 128, (size_t)seg * per, st>>>(m, a, s, table, seg);
    return (int)cudaGetLastError();
}
template <int OP>
int launch_near_p(cudaStream_t st, const MeshDev &m, const NearArgs &a, const SepSet &s, const c64 *table, int sms) {
    if constexpr (TD_P1_TRIAL(OP)) {
        if (s.P == 24) return launch_near<OP, 16, 24>(st, m, a, s, table, sms);
        return launch_near<OP, 24, 40>(st, m, a, s, table, sms);
    } else {
        switch (s.P) {
            case 16: return launch_near<OP, 0, 16>(st, m, a, s, table, sms);
            case 24: return launch_near<OP, 0, 24>(st, m, a, s, table, sms);
            case 32: return launch_near<OP, 0, 32>(st, m, a, s, table, sms);
            default: return launch_near<OP, 0, 40>(st, m, a, s, table, sms);
        }
    }
}

template <int OP>
int launch_sing(cudaStream_t st, const MeshDev &m, const int *pti, const int *ptj, int npairs, const double *rule,
                const SepSet &s, int nf, c64 *table, int num_sms) {
    const int grid = std::min((npairs + 3) / 4, num_sms * 16);
    if (s.P == 24) k_sing_sep<OP, 16, 24><<<grid, 128, 0, st>>>(m, pti, ptj, npairs, rule, s, nf, table);
    else k_sing_sep<OP, 24, 40><<<grid, 128, 0, st>>>(m, pti, ptj, npairs, rule, s, nf, table);
    return (int)cudaGetLastError();
}

}  // namespace

// Separated and direct frequencies of one call: a frequency whose |sigma| D is
// beyond the longest variant stays direct, and so does a single regular one
// (the moments cost about as much as one direct frequency; the sums of two
// frequencies already come cheaper: 2640-triangle housing, 2 frequencies).  The mixed
// form is direct throughout.
void td_sep_split(int op, int prec, const double *sigma, int nf, double D, bool touching, std::vector<int> &klist,
                  SepSet &s) {
    std::vector<int> dir;
    klist.clear();
    s = SepSet{};
    s.D = D;
    double zmax = 0.0;
    for (int k = 0; k < nf; ++k) {
        const double z = std::hypot(sigma[2 * k], sigma[2 * k + 1]) * D;
        if (prec == TDBEM_FP64 && D > 0.0 && variant_for(op, z, touching)) {
            klist.push_back(k);
            zmax = std::max(zmax, z);
        } else {
            dir.push_back(k);
        }
    }
    if ((int)klist.size() < (touching ? 1 : 2)) {
        klist.clear();
        dir.resize(nf);
        for (int k = 0; k < nf; ++k) dir[k] = k;
    }
    s.nsep = (int)klist.size();
    s.ndir = (int)dir.size();
    if (s.nsep) {
        const SepVariant *v = variant_for(op, zmax, touching);
        s.P = v->P;
        s.P1 = v->P1;
    }
    klist.insert(klist.end(), dir.begin(), dir.end());
}

size_t td_sep_coef_bytes(int op, const SepSet &s, bool touching) {
    return sizeof(c64) * s.nsep * (s.P + s.P1) * (op == TD_SLP || touching ? 1 : 2);
}

int td_launch_sep_coef(cudaStream_t st, int op, const double *sig, int nq, double c, const SepSet &s, bool touching) {
    if (s.nsep == 0) return 0;
    const int kind = op == TD_SLP ? 0 : touching ? 2 : 1;
    auto run = [&](double left, double half, int P, int first) {
        k_sep_coef<<<s.nsep, kNodes, 0, st>>>(sig, nq, s.klist, s.nsep, left / c, half / c, P, kind, touching, s.P1 + s.P, first,
                                              s.coef, touching ? nullptr : s.pk);
    };
    if (s.P1) {
        run(0.0, 0.25 * s.D, s.P1, 0);
        run(0.5 * s.D, 0.75 * s.D, s.P, s.P1);
    } else {
        run(0.0, s.D, s.P, 0);
    }
    return (int)cudaGetLastError();
}

int64_t td_ss_rule_size(int ng) { return ss_rule_off(3, ng) + (int64_t)8 * ss_npoints(3, ng); }

int td_launch_ss_rule(cudaStream_t st, int ng, const double *gx, const double *gw, double *rule) {
    const int n = ss_npoints(1, ng) + ss_npoints(2, ng) + ss_npoints(3, ng);
    k_ss_rule<<<std::min((n + 127) / 128, 1024), 128, 0, st>>>(ng, gx, gw, rule);
    return (int)cudaGetLastError();
}

int td_launch_near_sep(cudaStream_t st, const MeshDev &m, int op, const NearArgs &a, const SepSet &s, const c64 *table,
                       int num_sms) {
    if (a.nentries == 0 || s.nsep == 0) return 0;
    return op == TD_SLP   ? launch_near_p<TD_SLP>(st, m, a, s, table, num_sms)
           : op == TD_DLP ? launch_near_p<TD_DLP>(st, m, a, s, table, num_sms)
                          : launch_near_p<TD_ADLP>(st, m, a, s, table, num_sms);
}

int td_launch_sing_sep(cudaStream_t st, const MeshDev &m, int op, const int *pti, const int *ptj, int npairs,
                       const double *rule, const SepSet &s, int nf, c64 *table, int num_sms) {
    if (npairs == 0 || s.nsep == 0) return 0;
    return op == TD_SLP   ? launch_sing<TD_SLP>(st, m, pti, ptj, npairs, rule, s, nf, table, num_sms)
           : op == TD_DLP ? launch_sing<TD_DLP>(st, m, pti, ptj, npairs, rule, s, nf, table, num_sms)
                          : launch_sing<TD_ADLP>(st, m, pti, ptj, npairs, rule, s, nf, table, num_sms);
}

bool td_entry_sing_set(int op, double smax, double c, double D, int64_t nE, int64_t nf, SepSet &s) {
    s = SepSet{};
    const SepVariant *v = variant_for(op, smax / c * D, true);
    if (!v || !(D > 0.0) || nf < 3 || nf > 4096 || nE < 512) return false;
    s.nsep = (int)nf;
    s.P = v->P;
    s.P1 = v->P1;
    s.D = D;
    return true;
}

namespace {
template <class T, int OP>
int launch_entry_sing(cudaStream_t st, const MeshDev &m, const double *rule, const SepSet &s, int nq, const int *rows,
                      int64_t nr, const int *cols, int64_t nc, void *out, int num_sms) {
    const int grid = (int)std::min<int64_t>((nr * nc + 127) / 128, (int64_t)num_sms * 32);
    if (s.P == 24) k_entry_sing<T, OP, 16, 24><<<grid, 128, 0, st>>>(m, rule, s, nq, rows, nr, cols, nc, (cx<T> *)out);
    else k_entry_sing<T, OP, 24, 40><<<grid, 128, 0, st>>>(m, rule, s, nq, rows, nr, cols, nc, (cx<T> *)out);
    return (int)cudaGetLastError();
}
}  // namespace

int td_launch_entry_sing(cudaStream_t st, const MeshDev &m, int op, int prec, const double *rule, const SepSet &s, int nq,
                         const int *rows, int64_t nr, const int *cols, int64_t nc, void *out, int num_sms) {
    if (prec == TDBEM_FP64)
        return op == TD_SLP   ? launch_entry_sing<double, TD_SLP>(st, m, rule, s, nq, rows, nr, cols, nc, out, num_sms)
               : op == TD_DLP ? launch_entry_sing<double, TD_DLP>(st, m, rule, s, nq, rows, nr, cols, nc, out, num_sms)
                              : launch_entry_sing<double, TD_ADLP>(st, m, rule, s, nq, rows, nr, cols, nc, out, num_sms);
    return op == TD_SLP   ? launch_entry_sing<float, TD_SLP>(st, m, rule, s, nq, rows, nr, cols, nc, out, num_sms)
           : op == TD_DLP ? launch_entry_sing<float, TD_DLP>(st, m, rule, s, nq, rows, nr, cols, nc, out, num_sms)
                          : launch_entry_sing<float, TD_ADLP>(st, m, rule, s, nq, rows, nr, cols, nc, out, num_sms);
}
