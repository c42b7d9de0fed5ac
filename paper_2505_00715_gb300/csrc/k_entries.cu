// Entry kernels (Sec. 3; the ENTRY function of Algorithm 1):
//   k_entries_generic : arbitrary rows x cols x frequencies (C-ABI tdbem_entries)
//   (operators: single layer, double layer, adjoint double layer K')
//   k_sing_table      : touching pairs (Sauter-Schwab, FP64) at a list of
//                       frequencies, one warp per pair
//   k_near_entries    : every entry of a list of near-field blocks at a list of
//                       frequencies; regular pairs in the block precision with
//                       the quadrature geometry shared across frequencies,
//                       touching pairs read from the table.
// In the compression the FP64 form takes most frequencies by the separated sums
// of k_sep.cu, and the mixed form forms its near entries on demand (k_near_aca).
#include "internal.h"
#include "kernels.h"
#include "near.cuh"

namespace {

// ---- generic entries --------------------------------------------------------
// One point pair at FC frequencies: test point oa of the lane (its weight is
// left to the end of the sum), trial point ob with the trial hat; d = y - x.
// acc += w e^{-sigma r} / r (SLP) or w (1 + sigma r) e^{-sigma r} (d.n) / r^3 with
// the signed kernel normal n.
template <int OP, int FC>
TD_D void point_multi(const MeshDev &m, int oa, int ob, float hat, const float *n, const float *sr, const float *si,
                      c32 *acc) {
    const float4 xa = __ldg(&m.qp[2 * oa]), xl = __ldg(&m.qp[2 * oa + 1]);
    const float4 yb = __ldg(&m.qp[2 * ob]), yl = __ldg(&m.qp[2 * ob + 1]);
    const float dx = (yb.x - xa.x) + (yl.x - xl.x), dy = (yb.y - xa.y) + (yl.y - xl.y),
                dz = (yb.z - xa.z) + (yl.z - xl.z);
    const float r2 = dx * dx + dy * dy + dz * dz;
    const float rinv = rsqrtf(r2), r = r2 * rinv;
    float w = (TD_P1_TRIAL(OP) ? yb.w * hat : yb.w) * rinv;
    if (OP != TD_SLP) w *= (dx * n[0] + dy * n[1] + dz * n[2]) * rinv * rinv;
#pragma unroll
    for (int j = 0; j < FC; ++j) {
        const c32 e = expm_sr(sr[j], si[j], r);
        if (OP == TD_SLP) {
            acc[j].x = fmaf(w, e.x, acc[j].x);
            acc[j].y = fmaf(w, e.y, acc[j].y);
        } else {
            const float pr = fmaf(sr[j], r, 1.0f), pi = si[j] * r;
            acc[j].x = fmaf(w, pr * e.x - pi * e.y, acc[j].x);
            acc[j].y = fmaf(w, pr * e.y + pi * e.x, acc[j].y);
        }
    }
}
template <int OP, int FC>
TD_D void point_multi(const MeshDev &m, int oa, int ob, double hat, const double *n, const double *sr, const double *si,
                      c64 *acc) {
    const double dx = m.qx[ob] - m.qx[oa], dy = m.qy[ob] - m.qy[oa], dz = m.qz[ob] - m.qz[oa];
    double ri;
    const double r = sqrt_inv(dx * dx + dy * dy + dz * dz, ri);
    double w = (TD_P1_TRIAL(OP) ? m.qw[ob] * hat : m.qw[ob]) * ri;
    if (OP != TD_SLP) w *= (dx * n[0] + dy * n[1] + dz * n[2]) * ri * ri;
#pragma unroll
    for (int j = 0; j < FC; ++j) {
        const c64 e = expm_sr(sr[j], si[j], r);
        if (OP == TD_SLP) {
            acc[j].x += w * e.x;
            acc[j].y += w * e.y;
        } else {
            const double pr = 1.0 + sr[j] * r, pi = si[j] * r;
            acc[j].x += w * (pr * e.x - pi * e.y);
            acc[j].y += w * (pr * e.y + pi * e.x);
        }
    }
}
TD_D void tri_normal(const MeshDev &m, int t, float sign, float *n) {
    const float4 v = __ldg(&m.nrm4[t]);
    n[0] = sign * v.x;
    n[1] = sign * v.y;
    n[2] = sign * v.z;
}
TD_D void tri_normal(const MeshDev &m, int t, double sign, double *n) {
    for (int k = 0; k < 3; ++k) n[k] = sign * m.n64[(int64_t)k * m.nt + t];
}
TD_D float point_weight(const MeshDev &m, int o, float) { return m.qw32[o]; }
TD_D double point_weight(const MeshDev &m, int o, double) { return m.qw[o]; }
TD_D float hat7(int b, int loc, float) { return bary7f(b, loc); }
TD_D double hat7(int b, int loc, double) { return bary7d(b, loc); }

// out[f][r][c] = A[rows[r], cols[c]](s_{fidx[f]} / c), an item = one (row,
// column) at FC consecutive frequencies of the list.  Eight lanes per item: seven
// take one test point each against the seven trial points (regular pairs); with
// SING the touching pairs of a warp's four items are then integrated one after the
// other by all 32 lanes, which split the up to 2 ng^4 Sauter-Schwab points (FP64 in
// both forms), without it k_entry_sing adds them for all frequencies at once.  One
// thread per entry left a warp waiting for the lane with the touching pair, 1250
// points in a row at latency: 320 x 320 x 16 FP64 entries 269 -> 18.1 ms with SING, 10.5 with
// k_entry_sing; 67 x 1801 x 11 double-layer entries 119 -> 6.2 and 2.9 ms.  Bound:
// the FP64 pipe.
template <class T, int OP, int FC, bool SING>
__global__ void __launch_bounds__(128) k_entries_generic(MeshDev m, const double *s, double c, int nq, const int *rows,
                                                         int64_t nr, const int *cols, int64_t nc, const int *fidx,
                                                         int64_t nf, cx<T> *out) {
    const int64_t nE = nr * nc, items = nE * ((nf + FC - 1) / FC);
    const int ncols = TD_P1_TRIAL(OP) ? m.nv : m.nt;
    const int lane = threadIdx.x & 31, sub = lane & 7, grp = lane >> 3;
    const double inv4pi = 1.0 / TD_FOUR_PI;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 3;
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) >> 3; base < items; base += stride) {
        const bool valid = base + grp < items;
        const int64_t it = valid ? base + grp : 0;
        const int64_t e = it % nE, f0 = it / nE * FC;
        const int row = rows[e / nc], col = cols[e % nc];
        const bool ok = valid && row >= 0 && row < m.nt && col >= 0 && col < ncols;
        double sr[FC], si[FC];
        T tr[FC], ti[FC];
        bool fok[FC];
#pragma unroll
        for (int j = 0; j < FC; ++j) {
            const int k = f0 + j < nf ? fidx[f0 + j] : -1;
            fok[j] = k >= 0 && k < nq;
            sr[j] = fok[j] ? s[2 * k] / c : 0.0;
            si[j] = fok[j] ? s[2 * k + 1] / c : 0.0;
            tr[j] = (T)sr[j];
            ti[j] = (T)si[j];
        }
        cx<T> acc[FC];
        c64 sing[FC];
#pragma unroll
        for (int j = 0; j < FC; ++j) {
            acc[j] = cx<T>{0, 0};
            sing[j] = c64{0.0, 0.0};
        }
        const int p0 = ok && TD_P1_TRIAL(OP) ? m.v2t_ptr[col] : 0;
        const int ns = !ok ? 0 : TD_P1_TRIAL(OP) ? m.v2t_ptr[col + 1] - p0 : 1;
        const int nsw = __reduce_max_sync(0xffffffffu, ns);
        for (int q = 0; q < nsw; ++q) {
            const bool has = q < ns;
            const int tj = !has ? 0 : TD_P1_TRIAL(OP) ? m.v2t[p0 + q] : col;
            const int loc = has && TD_P1_TRIAL(OP) ? m.v2t_loc[p0 + q] : 0;
            const bool touch = has && touching_slot(m, row, tj) >= 0;
            if (has && !touch && sub < 7) {
                T n[3];
                if (OP != TD_SLP) tri_normal(m, OP == TD_DLP ? tj : row, OP == TD_DLP ? T(-1) : T(1), n);
                const int oa = sub * m.nt + row;
#pragma unroll 1
                for (int b = 0; b < 7; ++b)
                    point_multi<OP, FC>(m, oa, b * m.nt + tj, TD_P1_TRIAL(OP) ? hat7(b, loc, T(0)) : T(1), n, tr, ti, acc);
            }
            for (unsigned todo = SING ? __ballot_sync(0xffffffffu, touch && sub == 0) : 0u; todo; todo &= todo - 1) {
                const int src = __ffs(todo) - 1;
                int ta = __shfl_sync(0xffffffffu, row, src), tb = __shfl_sync(0xffffffffu, tj, src);
                const int lb = __shfl_sync(0xffffffffu, loc, src);
                double br[FC], bi[FC];
                c64 v[FC];
#pragma unroll
                for (int j = 0; j < FC; ++j) {
                    br[j] = __shfl_sync(0xffffffffu, sr[j], src);
                    bi[j] = __shfl_sync(0xffffffffu, si[j], src);
                    v[j] = c64{0.0, 0.0};
                }
                if (OP == TD_SLP && ta > tb) {
                    const int t = ta;
                    ta = tb;
                    tb = t;
                }
                SingGeom G;
                classify_pair(m, ta, tb, G);
                // (flat panel: (x - y).n = 0)
                const int np = OP != TD_SLP && G.cls == 3 ? 0 : ss_npoints(G.cls, m.ng);
                SsEdges E;
                ss_edges(G, E);
                const int hat = G.loc[0] == lb ? 0 : G.loc[1] == lb ? 1 : 2;
                for (int p = lane; p < np; p += 32) {
                    double a[4], w, lam[3], d[3];
                    ss_ref(G.cls, p, m.ng, m.gx, m.gw, a, w, lam);
                    ss_diff(G.cls, a, E, d);
                    const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
                    w *= G.g;
                    if (OP == TD_SLP) w /= r;
                    else w *= ss_dn<OP>(G, d) / (r * r * r);
                    if (TD_P1_TRIAL(OP)) w *= hat == 0 ? lam[0] : hat == 1 ? lam[1] : lam[2];
#pragma unroll
                    for (int j = 0; j < FC; ++j) {
                        const c64 x = expm_sr(br[j], bi[j], r);
                        if (OP == TD_SLP) {
                            v[j].x += w * x.x;
                            v[j].y += w * x.y;
                        } else {
                            const double pr = 1.0 + br[j] * r, pi = bi[j] * r;
                            v[j].x += w * (pr * x.x - pi * x.y);
                            v[j].y += w * (pr * x.y + pi * x.x);
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < FC; ++j) {
                    const c64 t = {warp_sum(v[j].x), warp_sum(v[j].y)};
                    if (grp == src >> 3) sing[j] = sing[j] + t;
                }
            }
        }
        const T wx = ok && sub < 7 ? point_weight(m, sub * m.nt + row, T(0)) : T(0);
#pragma unroll
        for (int j = 0; j < FC; ++j) {
            acc[j] = wx * acc[j];
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                acc[j].x += __shfl_xor_sync(0xffffffffu, acc[j].x, o);
                acc[j].y += __shfl_xor_sync(0xffffffffu, acc[j].y, o);
            }
            // an invalid index gives NaN without any table access
            if (valid && sub == 0 && f0 + j < nf)
                out[(f0 + j) * nE + e] = ok && fok[j] ? cx<T>{(T)(((double)acc[j].x + sing[j].x) * inv4pi),
                                                              (T)(((double)acc[j].y + sing[j].y) * inv4pi)}
                                                      : cx<T>{(T)NAN, (T)NAN};
        }
    }
}

// ---- touching-pair table ----------------------------------------------------
// table layout: [slot][nf][1 or 3 (P1 columns)] complex128, 1/(4 pi) applied.
// Both forms run the nd frequencies of klist, those that the separated sums
// (k_sep.cu) leave: |sigma| times the longest edge beyond their terms.
template <int OP, int FC>
__global__ void k_sing_table(MeshDev m, const int *pti, const int *ptj, int npairs,
                             const double *sig, int nf, const int *klist, int nd, c64 *table) {
    constexpr int NV = TD_P1_TRIAL(OP) ? 3 : 1;
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int p = warp; p < npairs; p += nwarps) {
        int ti = pti[p], tj = ptj[p];
        if (OP == TD_SLP && ti > tj) {
            int t = ti;
            ti = tj;
            tj = t;
        }
        SingGeom G;
        classify_pair(m, ti, tj, G);
        const int nq = ss_npoints(G.cls, m.ng);
        const bool zero = (OP != TD_SLP && G.cls == 3) || G.cls == 0;
        for (int f0 = 0; f0 < nd; f0 += FC) {
            c64 acc[FC][3];
#pragma unroll
            for (int j = 0; j < FC; ++j)
                for (int k = 0; k < 3; ++k) acc[j][k] = {0.0, 0.0};
            if (!zero) {
                for (int q = lane; q < nq; q += 32) {
                    double d[3], w, lam[3];
                    ss_point(G, q, m.ng, m.gx, m.gw, d, w, lam);
                    double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
                    double base, pre;
                    if (OP == TD_SLP) {
                        base = w / r;
                    } else {
                        base = w * ss_dn<OP>(G, d) / (r * r * r);
                    }
                    (void)pre;
#pragma unroll
                    for (int j = 0; j < FC; ++j) {
                        if (f0 + j < nd) {
                            const int kf = klist[f0 + j];
                            double sr = sig[2 * kf], si = sig[2 * kf + 1];
                            c64 e = expm_sr(sr, si, r);
                            if (OP == TD_SLP) {
                                acc[j][0].x += base * e.x;
                                acc[j][0].y += base * e.y;
                            } else {
                                double pr = 1.0 + sr * r, pi = si * r;
                                c64 v = {base * (pr * e.x - pi * e.y), base * (pr * e.y + pi * e.x)};
                                if (OP == TD_ADLP) {
                                    acc[j][0].x += v.x;
                                    acc[j][0].y += v.y;
                                } else {
#pragma unroll
                                    for (int k = 0; k < 3; ++k) {
                                        acc[j][k].x += lam[k] * v.x;
                                        acc[j][k].y += lam[k] * v.y;
                                    }
                                }
                            }
                        }
                    }
                }
            }
            const double inv4pi = 1.0 / TD_FOUR_PI;
#pragma unroll
            for (int j = 0; j < FC; ++j) {
                c64 outv[3];
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    outv[k] = {warp_sum(acc[j][k].x) * inv4pi, warp_sum(acc[j][k].y) * inv4pi};
                if (lane == 0 && f0 + j < nd) {
                    c64 *o = table + ((int64_t)p * nf + klist[f0 + j]) * NV;
                    if (!TD_P1_TRIAL(OP)) {
                        o[0] = zero ? c64{0.0, 0.0} : outv[0];
                    } else {
                        // parametrisation order -> mesh-local trial vertex
                        c64 z = {0.0, 0.0};
                        o[0] = o[1] = o[2] = z;
                        for (int k = 0; k < 3; ++k) o[G.loc[k]] = zero ? z : outv[k];
                    }
                }
            }
        }
    }
}

// Mixed form of the touching-pair table: the transformed coordinates, the
// Jacobian weights and the chunk sums in the table are FP64; the smooth
// factor e^{-sigma r} (SLP) or e^{-sigma r}(1 + sigma r) (DLP, ADLP) of
// every point and frequency runs on the FP32 special-function path
// (relative error about 3e-7), and each lane's partial sums over its points
// are FP32.  The points of a pair are taken in chunks of 32 P (P per lane,
// held in registers): the FP64 point geometry of a chunk is formed once and
// reused by every frequency, FC frequencies per pass; each pass's lane sums
// are reduced over the warp and added to the pair's table rows.  The reference
// points come from an array formed once per call (k_ss_rule): a point then takes
// 18 FP64 operations instead of about 100, and the chunk sums meet in shared memory
// (the table was read and written once per pass, a memory latency each).  30k
// housing: 65 -> 43 -> 33 ms; 5120-triangle sphere, double layer: 15.7 -> 6.4 ms.
// Bound by FP32 issue, 24 instructions per point and frequency, and by the FP64 pipe.
template <int OP, int FC>
__global__ void __launch_bounds__(128, 4) k_sing_table_mixed(MeshDev m, const int *pti, const int *ptj, int npairs, const double *rule,
                                   const double *sig, int nf, const int *klist, int nd, c64 *table) {
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    constexpr int NV = TD_P1_TRIAL(OP) ? 3 : 1;
    constexpr int P = TD_P1_TRIAL(OP) ? 8 : 16;  // points per lane and chunk
    // the warp's table rows, FP64 (dynamic: 4 warps x nd x NV)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *rows = reinterpret_cast<double *>(smem_raw) + (int64_t)(threadIdx.x >> 5) * nd * NV * 2;
    // s / c of every frequency in shared memory (nd <= nf <= 256, checked by the caller)
    __shared__ float2 s_sig[256];
    for (int k = threadIdx.x; k < nd; k += blockDim.x)
        s_sig[k] = make_float2((float)sig[2 * klist[k]], (float)sig[2 * klist[k] + 1]);
    __syncthreads();
    const double inv4pi = 1.0 / TD_FOUR_PI;
    for (int p = warp; p < npairs; p += nwarps) {
        int ti = pti[p], tj = ptj[p];
        if (OP == TD_SLP && ti > tj) {
            int t = ti;
            ti = tj;
            tj = t;
        }
        SingGeom G;
        classify_pair(m, ti, tj, G);
        const int nq = ss_npoints(G.cls, m.ng);
        const bool zero = (OP != TD_SLP && G.cls == 3) || G.cls == 0;
        c64 *o = table + (int64_t)p * nf * NV;
        if (zero) {
            for (int e = lane; e < nd * NV; e += 32) o[(int64_t)klist[e / NV] * NV + e % NV] = c64{0.0, 0.0};
            continue;
        }
        __syncwarp();
        for (int e = lane; e < nd * NV * 2; e += 32) rows[e] = 0.0;
        __syncwarp();
        SsEdges E;
        ss_edges(G, E);
        const double *rl = rule + ss_rule_off(G.cls, m.ng);
        for (int q0 = 0; q0 < nq; q0 += 32 * P) {
            // the transformed point and the difference x - y in FP64 (no
            // cancellation near the singularity); |d|^2 is exact to FP64
            // rounding, so the square root, the division and the rest run in
            // FP32 at FP32 relative accuracy
            float rf[P], bf[P], lf[P][NV];
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const int q = q0 + 32 * i + lane;
                rf[i] = 1.0f;
                bf[i] = 0.0f;
#pragma unroll
                for (int k = 0; k < NV; ++k) lf[i][k] = 0.0f;
                if (q < nq) {
                    double a[4], d[3];
#pragma unroll
                    for (int e = 0; e < 4; ++e) a[e] = __ldg(rl + (int64_t)e * nq + q);
                    const double w = __ldg(rl + (int64_t)4 * nq + q) * G.g;
                    ss_diff(G.cls, a, E, d);
                    const float r2 = (float)(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
                    const float rinv = rsqrtf(r2);
                    rf[i] = r2 * rinv;
                    bf[i] = OP == TD_SLP ? (float)w * rinv : (float)w * (float)ss_dn<OP>(G, d) * rinv * rinv * rinv;
#pragma unroll
                    for (int k = 0; k < NV; ++k) lf[i][k] = TD_P1_TRIAL(OP) ? (float)__ldg(rl + (int64_t)(5 + k) * nq + q) : 1.0f;
                }
            }
            for (int f0 = 0; f0 < nd; f0 += FC) {
                c32 acc[FC][NV];
#pragma unroll
                for (int j = 0; j < FC; ++j)
#pragma unroll
                    for (int k = 0; k < NV; ++k) acc[j][k] = {0.f, 0.f};
#pragma unroll
                for (int i = 0; i < P; ++i) {
#pragma unroll
                    for (int j = 0; j < FC; ++j) {
                        const float2 sgj = s_sig[min(f0 + j, nd - 1)];
                        const c32 e = expm_sr(sgj.x, sgj.y, rf[i]);
                        c32 v;
                        if (OP == TD_SLP) {
                            v = {bf[i] * e.x, bf[i] * e.y};
                        } else {
                            const float pr = fmaf(sgj.x, rf[i], 1.0f), pi = sgj.y * rf[i];
                            v = {bf[i] * (pr * e.x - pi * e.y), bf[i] * (pr * e.y + pi * e.x)};
                        }
#pragma unroll
                        for (int k = 0; k < NV; ++k) {
                            acc[j][k].x = fmaf(lf[i][k], v.x, acc[j][k].x);
                            acc[j][k].y = fmaf(lf[i][k], v.y, acc[j][k].y);
                        }
                    }
                }
                // lane sums over the warp in FP32 (NS sums, padded to a power of two), chunk
                // sums into the FP64 rows by the lanes that hold them
                constexpr int NS = FC * NV * 2, NP = NS <= 4 ? 4 : NS <= 8 ? 8 : NS <= 16 ? 16 : 32;
#pragma unroll
                for (int c0 = 0; c0 < NS; c0 += NP) {
                    float v[NP];
#pragma unroll
                    for (int q = 0; q < NP; ++q) {
                        const int t = c0 + q, j = t / (2 * NV), kk = t / 2 % NV;
                        v[q] = t >= NS ? 0.0f : t & 1 ? acc[j][kk].y : acc[j][kk].x;
                    }
                    const float sum = warp_sum_many<NP>(v, lane);
                    const int t = c0 + many_index<NP>(lane), j = t / (2 * NV);
                    if ((lane & (32 / NP - 1)) == 0 && t < NS && f0 + j < nd)
                        rows[(f0 + j) * NV * 2 + t % (2 * NV)] += (double)sum * inv4pi;
                }
            }
        }
        __syncwarp();
        for (int e = lane; e < nd * NV; e += 32) {
            const int v = e % NV;
            o[(int64_t)klist[e / NV] * NV + (TD_P1_TRIAL(OP) ? G.loc[v] : 0)] = c64{rows[2 * e], rows[2 * e + 1]};
        }
    }
}

// ---- near-field dense entries -------------------------------------------------
// FP64 version of pair_multi (near.cuh).
template <int OP, int FC>
TD_D void pair_multi(const TestD &X, const MeshDev &m, int tj, const double *sg, int nfc, c64 *acc, int loc) {
    double nx = 0.0, ny = 0.0, nz = 0.0;  // signed kernel normal, as in the FP32 version
    if (OP == TD_DLP) {
        nx = -m.n64[tj];
        ny = -m.n64[m.nt + tj];
        nz = -m.n64[2 * m.nt + tj];
    } else if (OP == TD_ADLP) {
        nx = X.nx;
        ny = X.ny;
        nz = X.nz;
    }
#pragma unroll 1
    for (int b = 0; b < 7; ++b) {
        const int ob = b * m.nt + tj;
        const double yx = m.qx[ob], yy = m.qy[ob], yz = m.qz[ob];
        const double wyb = m.qw[ob] * (OP == TD_DLP ? bary7d(b, loc) : 1.0);
#pragma unroll 1
        for (int a = 0; a < 7; ++a) {
            const double dx = yx - X.x[a], dy = yy - X.y[a], dz = yz - X.z[a];
            double ri;
            const double r = sqrt_inv(dx * dx + dy * dy + dz * dz, ri);
            double w = X.w[a] * wyb * ri;
            if (OP != TD_SLP) w *= (dx * nx + dy * ny + dz * nz) * ri * ri;
#pragma unroll
            for (int j = 0; j < FC; ++j) {
                if (j < nfc) {
                    const double sr = sg[2 * j], si = sg[2 * j + 1];
                    const c64 e = expm_sr(sr, si, r);
                    if (OP == TD_SLP) {
                        acc[j].x += w * e.x;
                        acc[j].y += w * e.y;
                    } else {
                        const double pr = 1.0 + sr * r, pi = si * r;
                        acc[j].x += w * (pr * e.x - pi * e.y);
                        acc[j].y += w * (pr * e.y + pi * e.x);
                    }
                }
            }
        }
    }
}

// near[noff[b] + (k * nI + i) * nJ + j] for every near block b (list nb_idx),
// the nd frequencies of klist (those that the separated sums of k_sep.cu leave).  Entry e of the flattened list belongs to the
// near block found by binary search in the prefix `eprefix` (entries per block).
template <class T, int OP, int FC>
__global__ void __launch_bounds__(128) k_near_entries(MeshDev m, NearArgs a, const int *klist, int nd, const c64 *table) {
    constexpr int NV = TD_P1_TRIAL(OP) ? 3 : 1;
    __shared__ T sg[2 * 256];
    const int nf = a.nf;  // <= 256 (checked by the caller)
    for (int i = threadIdx.x; i < 2 * nd; i += blockDim.x) sg[i] = (T)a.sig[2 * klist[i >> 1] + (i & 1)];
    __syncthreads();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < a.nentries;
         t += (int64_t)gridDim.x * blockDim.x) {
        // block lookup
        int lo = 0, hi = a.nnear - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (a.eprefix[mid] <= t) lo = mid; else hi = mid - 1;
        }
        const int nb = lo;
        const int32_t *bl = a.blocks + 5 * a.near_ids[nb];
        const int nI = bl[1] - bl[0], nJ = bl[3] - bl[2];
        const int64_t loc_e = t - a.eprefix[nb];
        const int i = (int)(loc_e / nJ), j = (int)(loc_e % nJ);
        const int row = a.perm_r[bl[0] + i], col = a.perm_c[bl[2] + j];
        cx<T> *dst = (cx<T> *)a.near + a.noff[nb] + (int64_t)i * nJ + j;
        const int64_t fstride = (int64_t)nI * nJ;
        typename Reg<T>::Test X;
        load_test(m, row, X);
        const int nsup = TD_P1_TRIAL(OP) ? m.v2t_ptr[col + 1] - m.v2t_ptr[col] : 1;
        for (int f0 = 0; f0 < nd; f0 += FC) {
            const int nfc = min(FC, nd - f0);
            cx<T> acc[FC];
#pragma unroll
            for (int jj = 0; jj < FC; ++jj) acc[jj] = {0, 0};
            c64 sing[FC];
#pragma unroll
            for (int jj = 0; jj < FC; ++jj) sing[jj] = {0.0, 0.0};
            for (int sidx = 0; sidx < nsup; ++sidx) {
                int e, l;
                if (!TD_P1_TRIAL(OP)) {
                    e = col;
                    l = 0;
                } else {
                    int p = m.v2t_ptr[col] + sidx;
                    e = m.v2t[p];
                    l = m.v2t_loc[p];
                }
                int slot = touching_slot(m, row, e);
                if (slot >= 0) {
#pragma unroll
                    for (int jj = 0; jj < FC; ++jj)
                        if (jj < nfc) sing[jj] = sing[jj] + table[((int64_t)slot * nf + klist[f0 + jj]) * NV + l];
                } else {
                    pair_multi<OP, FC>(X, m, e, sg + 2 * f0, nfc, acc, l);
                }
            }
            const T inv4pi = (T)(1.0 / TD_FOUR_PI);
#pragma unroll
            for (int jj = 0; jj < FC; ++jj)
                if (jj < nfc)
                    dst[klist[f0 + jj] * fstride] =
                        cx<T>{(T)(acc[jj].x * inv4pi + (T)sing[jj].x), (T)(acc[jj].y * inv4pi + (T)sing[jj].y)};
        }
    }
}

}  // namespace

// ---- launchers ----------------------------------------------------------------
namespace {
// Four frequencies share the point geometry where that leaves enough items to
// fill the GPU (four per warp, 16 warps per SM); fewer items run one frequency each.
template <class T, int OP>
int launch_generic(cudaStream_t st, const MeshDev &m, const double *s, double c, int nq, const int *rows, int64_t nr,
                   const int *cols, int64_t nc, const int *fidx, int64_t nf, void *out, int num_sms, bool regular_only) {
    const int64_t nE = nr * nc;
    const bool four = nf >= 3 && nE * ((nf + 3) / 4) >= (int64_t)num_sms * 64;
    const int64_t items = nE * (four ? (nf + 3) / 4 : nf);
    const int grid = (int)std::min<int64_t>((items + 15) / 16, (int64_t)num_sms * 64);
    auto run = [&](auto kernel) { kernel<<<grid, 128, 0, st>>>(m, s, c, nq, rows, nr, cols, nc, fidx, nf, (cx<T> *)out); };
    if (regular_only) run(four ? k_entries_generic<T, OP, 4, false> : k_entries_generic<T, OP, 1, false>);
    else run(four ? k_entries_generic<T, OP, 4, true> : k_entries_generic<T, OP, 1, true>);
    return (int)cudaGetLastError();
}
}  // namespace

int td_launch_entries(cudaStream_t st, const MeshDev &m, int op, int prec, const double *s, double c, int nq,
                      const int *rows, int64_t nr, const int *cols, int64_t nc, const int *fidx,
                      int64_t nf, void *out, int num_sms, bool regular_only) {
    if (nr * nc * nf == 0) return 0;
    const bool ro = regular_only;
    if (prec == TDBEM_FP64)
        return op == TD_SLP   ? launch_generic<double, TD_SLP>(st, m, s, c, nq, rows, nr, cols, nc, fidx, nf, out, num_sms, ro)
               : op == TD_DLP ? launch_generic<double, TD_DLP>(st, m, s, c, nq, rows, nr, cols, nc, fidx, nf, out, num_sms, ro)
                              : launch_generic<double, TD_ADLP>(st, m, s, c, nq, rows, nr, cols, nc, fidx, nf, out, num_sms, ro);
    return op == TD_SLP   ? launch_generic<float, TD_SLP>(st, m, s, c, nq, rows, nr, cols, nc, fidx, nf, out, num_sms, ro)
           : op == TD_DLP ? launch_generic<float, TD_DLP>(st, m, s, c, nq, rows, nr, cols, nc, fidx, nf, out, num_sms, ro)
                          : launch_generic<float, TD_ADLP>(st, m, s, c, nq, rows, nr, cols, nc, fidx, nf, out, num_sms, ro);
}

// Frequencies per pass of the mixed-form kernels, selected by the tuning
// variant (0 = default): touching-pair table (single layer / double layer /
// adjoint double layer: one value per pair and frequency like the single
// layer) and near-field tensor.
constexpr int kSingFcSlp[3] = {4, 8, 16};
constexpr int kSingFcDlp[3] = {2, 4, 8};
constexpr int kNearFc[3] = {8, 4, 16};
int td_sing_fc(int op, int variant) { return op == TD_DLP ? kSingFcDlp[variant % 3] : kSingFcSlp[variant % 3]; }
int td_near_fc(int variant) { return kNearFc[variant % 3]; }

int td_launch_sing_table(cudaStream_t st, const MeshDev &m, int op, int prec, const int *pti, const int *ptj,
                         int npairs, const double *rule, const double *sig, int nf, const int *klist, int nd,
                         c64 *table, int num_sms, int variant) {
    if (npairs == 0 || nd == 0) return 0;
    if (nf > 256) return (int)cudaErrorInvalidValue;  // the frequencies are staged in shared memory
    int grid = std::min((npairs + 3) / 4, num_sms * 8);
    if (prec == TDBEM_MIXED) {
        const int v = variant % 3;
        const size_t sm = sizeof(c64) * 4 * nd * (op == TD_DLP ? 3 : 1);
        cudaError_t e = cudaSuccess;
        auto run = [&](auto kernel) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
            if (e == cudaSuccess) kernel<<<grid, 128, sm, st>>>(m, pti, ptj, npairs, rule, sig, nf, klist, nd, table);
        };
        if (op == TD_SLP)
            run(v == 1 ? k_sing_table_mixed<TD_SLP, 8> : v == 2 ? k_sing_table_mixed<TD_SLP, 16> : k_sing_table_mixed<TD_SLP, 4>);
        else if (op == TD_DLP)
            run(v == 1 ? k_sing_table_mixed<TD_DLP, 4> : v == 2 ? k_sing_table_mixed<TD_DLP, 8> : k_sing_table_mixed<TD_DLP, 2>);
        else
            run(v == 1 ? k_sing_table_mixed<TD_ADLP, 8> : v == 2 ? k_sing_table_mixed<TD_ADLP, 16> : k_sing_table_mixed<TD_ADLP, 4>);
        return e != cudaSuccess ? (int)e : (int)cudaGetLastError();
    }
    if (op == TD_SLP)
        k_sing_table<TD_SLP, 8><<<grid, 128, 0, st>>>(m, pti, ptj, npairs, sig, nf, klist, nd, table);
    else if (op == TD_DLP)
        k_sing_table<TD_DLP, 4><<<grid, 128, 0, st>>>(m, pti, ptj, npairs, sig, nf, klist, nd, table);
    else
        k_sing_table<TD_ADLP, 4><<<grid, 128, 0, st>>>(m, pti, ptj, npairs, sig, nf, klist, nd, table);
    return (int)cudaGetLastError();
}

int td_launch_near_entries(cudaStream_t st, const MeshDev &m, int op, int prec, const NearArgs &a, const int *klist,
                           int nd, const c64 *table, int num_sms, int variant) {
    if (a.nentries == 0 || nd == 0) return 0;
    int grid = (int)std::min<int64_t>((a.nentries + 127) / 128, (int64_t)num_sms * 16);
    if (prec == TDBEM_FP64) {
        if (op == TD_SLP) k_near_entries<double, TD_SLP, 4><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
        else if (op == TD_DLP) k_near_entries<double, TD_DLP, 4><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
        else k_near_entries<double, TD_ADLP, 4><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
    } else {
        const int v = variant % 3;
        if (op == TD_SLP) {
            if (v == 1) k_near_entries<float, TD_SLP, 4><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
            else if (v == 2) k_near_entries<float, TD_SLP, 16><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
            else k_near_entries<float, TD_SLP, 8><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
        } else if (op == TD_DLP) {
            if (v == 1) k_near_entries<float, TD_DLP, 4><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
            else if (v == 2) k_near_entries<float, TD_DLP, 16><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
            else k_near_entries<float, TD_DLP, 8><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
        } else {
            if (v == 1) k_near_entries<float, TD_ADLP, 4><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
            else if (v == 2) k_near_entries<float, TD_ADLP, 16><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
            else k_near_entries<float, TD_ADLP, 8><<<grid, 128, 0, st>>>(m, a, klist, nd, table);
        }
    }
    return (int)cudaGetLastError();
}
