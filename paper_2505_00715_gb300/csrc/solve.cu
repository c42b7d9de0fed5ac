// Per-frequency solve on the compressed tensor and persistence of tensors
// and models.
//
// tdbem_solve: restarted GMRES (Arnoldi with classical Gram-Schmidt applied
// twice, Givens rotations) for A(s_l) x = b, one Krylov space per right-hand side, all
// right-hand sides advanced together so that every operator application is
// one call of the single-frequency apply (y = sum_d f_d[l] H_d x, eq. product
// at one frequency).  Inner products are accumulated in FP64.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "internal.h"
#include "kernels.h"
#include "mlp.h"

namespace {

// red[c] = sum over the threads c, c + n, c + 2 n, ... < act of red, by halves (a thread
// per column adding 64 values in a row was a fifth of k_dots)
template <class R>
TD_D void column_sums(R *red, int act, int n) {
    const int g = threadIdx.x / n;
    for (int G = act / n; G > 1;) {
        const int half = (G + 1) / 2;
        __syncthreads();
        if (g < G - half) red[threadIdx.x] = red[threadIdx.x] + red[threadIdx.x + half * n];
        G = half;
    }
    __syncthreads();
}

// out[i n + c] += sum_r conj(V_i[r][c]) w[r][c] for the vectors V_i, i = blockIdx.y
// (FP64 accumulation; n <= 64 columns).  A thread keeps to one column: the
// block's active threads are a multiple of n.
template <class T>
__global__ void __launch_bounds__(256) k_dots(const cx<T> *V, const cx<T> *w, int64_t M, int n, c64 *out) {
    __shared__ c64 red[256];
    const int act = 256 / n * n, tid = threadIdx.x;
    const int64_t total = M * n;
    const cx<T> *v = V + (int64_t)blockIdx.y * total;
    double re = 0.0, im = 0.0;
    if (tid < act)
        for (int64_t e = (int64_t)blockIdx.x * act + tid; e < total; e += (int64_t)gridDim.x * act) {
            const cx<T> x = v[e], y = w[e];
            re += (double)x.x * y.x + (double)x.y * y.y;
            im += (double)x.x * y.y - (double)x.y * y.x;
        }
    red[tid] = c64{re, im};
    column_sums(red, act, n);
    if (tid < n) {
        const c64 s = red[tid];
        c64 *o = out + (int64_t)blockIdx.y * n + tid;
        atomicAdd(&o->x, s.x);
        atomicAdd(&o->y, s.y);
    }
}

// y[r][c] += sign sum_{i < k} V_i[r][c] h[i n + c]; norm2 (nullable): += |y|^2 per column
template <class T>
__global__ void __launch_bounds__(256) k_combine(cx<T> *y, const cx<T> *V, const c64 *h, int k, double sign, int64_t M,
                                                 int n, double *norm2) {
    __shared__ double red[256];
    const int act = 256 / n * n, tid = threadIdx.x, c = tid % n;
    const int64_t total = M * n;
    double s2 = 0.0;
    if (tid < act)
        for (int64_t e = (int64_t)blockIdx.x * act + tid; e < total; e += (int64_t)gridDim.x * act) {
            cx<T> s = {0, 0};
            for (int i = 0; i < k; ++i) {
                const c64 hv = h[i * n + c];
                cfma(s, cx<T>{(T)hv.x, (T)hv.y}, V[(int64_t)i * total + e]);
            }
            cx<T> v = y[e];
            v = cx<T>{v.x + (T)sign * s.x, v.y + (T)sign * s.y};
            y[e] = v;
            s2 += (double)v.x * v.x + (double)v.y * v.y;
        }
    if (!norm2) return;
    red[tid] = s2;
    column_sums(red, act, n);
    if (tid < n) atomicAdd(&norm2[tid], red[tid]);
}

// y[r][c] = x[r][c] / sqrt(norm2[c]) (0 where the norm is 0)
template <class T>
__global__ void __launch_bounds__(256) k_normalise(cx<T> *y, const cx<T> *x, const double *norm2, int64_t M, int n) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < M * n; e += (int64_t)gridDim.x * blockDim.x) {
        const double s = norm2[e % n];
        const T f = s > 0.0 ? (T)(1.0 / sqrt(s)) : (T)0;
        const cx<T> v = x[e];
        y[e] = cx<T>{f * v.x, f * v.y};
    }
}

// r = b - w with its squared column norms added to norm2
template <class T>
__global__ void __launch_bounds__(256) k_residual(cx<T> *r, const cx<T> *b, const cx<T> *w, int64_t M, int n, double *norm2) {
    __shared__ double red[256];
    const int act = 256 / n * n, tid = threadIdx.x;
    const int64_t total = M * n;
    double s2 = 0.0;
    if (tid < act)
        for (int64_t e = (int64_t)blockIdx.x * act + tid; e < total; e += (int64_t)gridDim.x * act) {
            cx<T> v = b[e];
            if (w) v = v - w[e];
            r[e] = v;
            s2 += (double)v.x * v.x + (double)v.y * v.y;
        }
    red[tid] = s2;
    column_sums(red, act, n);
    if (tid < n) atomicAdd(&norm2[tid], red[tid]);
}

// Restarted GMRES.  Arnoldi by classical Gram-Schmidt applied twice (two passes of
// all inner products and one combination each, orthogonal to working precision like
// the modified form) so that a step is one product, six launches and one wait for
// the host's rotations, where modified Gram-Schmidt waited for the host after
// every inner product: 5120-triangle sphere, 4 right-hand sides, 19 steps: 212 waits,
// 15.1 -> 10.9 ms by the single-frequency apply of k_apply_one, -> 5.8 ms by this,
// -> 4.0 ms by later forms of that apply, -> 3.6 ms by one copy of a step's sums and
// their reduction by halves.
template <class T>
int gmres(tdbem_tensor *t, int fidx, const cx<T> *b, int n, cx<T> *x, double tol, int maxit, int m, int *iters,
          double *relres) {
    tdbem_ctx *ctx = t->ctx;
    cudaStream_t st = ctx->stream;
    const int64_t M = t->nrows, Mn = M * n;
    using C = std::complex<double>;
    // one allocation: V [m + 1] | w | r, then FP64 sums [2 (m + 1)][n] complex | norm2 [n]
    const size_t vb = (sizeof(cx<T>) * Mn * (m + 3) + 255) & ~(size_t)255;
    const size_t nh = (size_t)(m + 1) * n, hb = sizeof(c64) * 2 * nh + sizeof(double) * n;
    char *mem = nullptr;
    if (cudaMalloc((void **)&mem, vb + hb) != cudaSuccess) {
        cudaGetLastError();
        return TDBEM_ERR_OOM;
    }
    cx<T> *V = (cx<T> *)mem, *w = V + (int64_t)(m + 1) * Mn, *r = w + Mn;
    c64 *h1 = (c64 *)(mem + vb);
    double *norm2 = (double *)(h1 + 2 * nh);
    std::vector<C> hh(2 * nh + (n + 1) / 2);
    std::vector<double> hn(n);
    const int act = 256 / n * n;
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((Mn + act - 1) / act, (int64_t)ctx->num_sms * 2));
    auto ok = [&](cudaError_t e) { return e == cudaSuccess ? TDBEM_OK : TDBEM_ERR_CUDA; };
    // r = b - A x (A x left out at x = 0), its column norms to hn
    auto residual = [&](bool zero) {
        int rc = TDBEM_OK;
        if (!zero && (rc = tdbem_apply_freq(t, fidx, x, n, w))) return rc;
        cudaMemsetAsync(norm2, 0, sizeof(double) * n, st);
        k_residual<T><<<g, 256, 0, st>>>(r, b, zero ? nullptr : w, M, n, norm2);
        cudaMemcpyAsync(hn.data(), norm2, sizeof(double) * n, cudaMemcpyDeviceToHost, st);
        return ok(cudaStreamSynchronize(st));
    };
    int rc = TDBEM_OK, it = 0;
    cudaMemsetAsync(x, 0, sizeof(cx<T>) * Mn, st);
    std::vector<double> bnorm(n), res(n, 1.0), beta(n);
    bool done = false;
    for (bool first = true; !done && it < maxit; first = false) {
        if ((rc = residual(first))) break;
        if (first)
            for (int c = 0; c < n; ++c) bnorm[c] = std::sqrt(std::max(hn[c], 1e-300));
        done = true;
        for (int c = 0; c < n; ++c) {
            beta[c] = std::sqrt(std::max(hn[c], 0.0));
            res[c] = beta[c] / bnorm[c];
            if (res[c] > tol) done = false;
        }
        if (done) break;
        // V0 = r / beta
        k_normalise<T><<<g, 256, 0, st>>>(V, r, norm2, M, n);
        std::vector<std::vector<C>> H(n, std::vector<C>((m + 1) * m, C(0, 0)));
        std::vector<std::vector<C>> cs(n, std::vector<C>(m)), sn(n, std::vector<C>(m));
        std::vector<std::vector<C>> g0(n, std::vector<C>(m + 1, C(0, 0)));
        for (int c = 0; c < n; ++c) g0[c][0] = beta[c];
        int j = 0;
        for (; j < m && it < maxit; ++j, ++it) {
            cx<T> *Vj = V + (int64_t)j * Mn, *Vn = V + (int64_t)(j + 1) * Mn;
            if ((rc = tdbem_apply_freq(t, fidx, Vj, n, w))) break;
            // the step's sums h1 [j + 1][n] | h2 [j + 1][n] | squared norms [n], read back by one copy
            const size_t nj = (size_t)(j + 1) * n, sb = sizeof(c64) * 2 * nj + sizeof(double) * n;
            c64 *h2 = h1 + nj;
            double *nw = (double *)(h2 + nj);
            cudaMemsetAsync(h1, 0, sb, st);
            const dim3 gd(std::max(1u, std::min(g, 2u * (unsigned)ctx->num_sms / (unsigned)(j + 1) + 1u)), j + 1);
            k_dots<T><<<gd, 256, 0, st>>>(V, w, M, n, h1);
            k_combine<T><<<g, 256, 0, st>>>(w, V, h1, j + 1, -1.0, M, n, nullptr);
            k_dots<T><<<gd, 256, 0, st>>>(V, w, M, n, h2);
            k_combine<T><<<g, 256, 0, st>>>(w, V, h2, j + 1, -1.0, M, n, nw);
            k_normalise<T><<<g, 256, 0, st>>>(Vn, w, nw, M, n);
            cudaMemcpyAsync(hh.data(), h1, sb, cudaMemcpyDeviceToHost, st);
            if ((rc = ok(cudaStreamSynchronize(st)))) break;
            const double *hw = reinterpret_cast<const double *>(hh.data() + 2 * nj);
            bool all = true;
            for (int c = 0; c < n; ++c) {
                for (int i = 0; i <= j; ++i) H[c][i * m + j] = hh[i * n + c] + hh[nj + i * n + c];
                const double h = std::sqrt(std::max(hw[c], 0.0));
                H[c][(j + 1) * m + j] = h;
                // Givens rotations on column j
                for (int i = 0; i < j; ++i) {
                    const C a = H[c][i * m + j], bb = H[c][(i + 1) * m + j];
                    H[c][i * m + j] = std::conj(cs[c][i]) * a + std::conj(sn[c][i]) * bb;
                    H[c][(i + 1) * m + j] = -sn[c][i] * a + cs[c][i] * bb;
                }
                const C a = H[c][j * m + j], bb = H[c][(j + 1) * m + j];
                const double den = std::sqrt(std::norm(a) + std::norm(bb));
                if (den > 0) {
                    cs[c][j] = a / den;
                    sn[c][j] = bb / den;
                } else {
                    cs[c][j] = 1.0;
                    sn[c][j] = 0.0;
                }
                H[c][j * m + j] = std::conj(cs[c][j]) * a + std::conj(sn[c][j]) * bb;
                H[c][(j + 1) * m + j] = 0.0;
                const C gj = g0[c][j];
                g0[c][j] = std::conj(cs[c][j]) * gj;
                g0[c][j + 1] = -sn[c][j] * gj;
                res[c] = std::abs(g0[c][j + 1]) / bnorm[c];
                if (res[c] > tol) all = false;
            }
            if (all) {
                ++j;
                ++it;
                break;
            }
        }
        if (rc) break;
        // x += V y with H y = g (upper triangular, per column)
        const int kk = j;
        for (int c = 0; c < n; ++c) {
            std::vector<C> yv(kk);
            for (int i = kk - 1; i >= 0; --i) {
                C s = g0[c][i];
                for (int l = i + 1; l < kk; ++l) s -= H[c][i * m + l] * yv[l];
                yv[i] = std::abs(H[c][i * m + i]) > 0 ? s / H[c][i * m + i] : C(0, 0);
            }
            for (int i = 0; i < kk; ++i) hh[i * n + c] = yv[i];
        }
        cudaMemcpyAsync(h1, hh.data(), sizeof(c64) * (size_t)kk * n, cudaMemcpyHostToDevice, st);
        k_combine<T><<<g, 256, 0, st>>>(x, V, h1, kk, 1.0, M, n, nullptr);
        if ((rc = ok(cudaStreamSynchronize(st)))) break;  // hh is reused
    }
    if (!rc && !done) {
        // explicit final residual (when the loop ended by the true residual
        // test, res holds the explicit residuals of the final x already; a
        // second product would differ from it by the rounding of the apply)
        if (!(rc = residual(it == 0)))
            for (int c = 0; c < n; ++c) res[c] = std::sqrt(std::max(hn[c], 0.0)) / bnorm[c];
    }
    cudaStreamSynchronize(st);
    cudaFree(mem);
    if (iters) *iters = it;
    if (relres)
        for (int c = 0; c < n; ++c) relres[c] = res[c];
    if (rc) return rc;
    for (int c = 0; c < n; ++c)
        if (!(res[c] <= tol * 1.0000001)) return TDBEM_ERR_NOT_CONVERGED;
    return TDBEM_OK;
}

// ---- binary files ------------------------------------------------------------
const char kTensorMagic[8] = {'T', 'D', 'B', 'E', 'M', 'T', '0', '1'};
const char kModelMagic[8] = {'T', 'D', 'B', 'E', 'M', 'M', '0', '1'};

bool wr(FILE *f, const void *p, size_t n) { return n == 0 || fwrite(p, 1, n, f) == n; }
bool rd(FILE *f, void *p, size_t n) { return n == 0 || fread(p, 1, n, f) == n; }

template <class V>
bool wr_dev(FILE *f, const V *d, size_t count) {
    std::vector<V> h(count);
    if (count && cudaMemcpy(h.data(), d, sizeof(V) * count, cudaMemcpyDeviceToHost) != cudaSuccess) return false;
    return wr(f, h.data(), sizeof(V) * count);
}
template <class V>
bool rd_dev(FILE *f, V *d, size_t count) {
    std::vector<V> h(count);
    if (!rd(f, h.data(), sizeof(V) * count)) return false;
    return count == 0 || cudaMemcpy(d, h.data(), sizeof(V) * count, cudaMemcpyHostToDevice) == cudaSuccess;
}

}  // namespace

extern "C" int tdbem_solve(tdbem_tensor_t t, int32_t fidx, const void *b, int32_t nrhs, void *x, double tol,
                           int32_t maxit, int32_t restart, int32_t *iters, double *relres) {
    if (!t) return TDBEM_ERR_ARG;
    tdbem_ctx *ctx = t->ctx;
    cudaGetLastError();
    if (t->nrows != t->ncols) return td_fail(ctx, TDBEM_ERR_ARG, "tdbem_solve needs a square operator (SLP)");
    if (!b || !x || nrhs < 1 || nrhs > 64 || fidx < 0 || fidx >= t->NQ || !(tol > 0.0) || maxit < 1)
        return td_fail(ctx, TDBEM_ERR_ARG, "tdbem_solve: bad arguments");
    const int m = restart > 0 ? std::min(restart, 200) : 30;
    int rc = t->prec == TDBEM_FP64 ? gmres<double>(t, fidx, (const c64 *)b, nrhs, (c64 *)x, tol, maxit, m, iters, relres)
                                   : gmres<float>(t, fidx, (const c32 *)b, nrhs, (c32 *)x, tol, maxit, m, iters, relres);
    if (rc == TDBEM_ERR_NOT_CONVERGED) return td_fail(ctx, rc, "GMRES did not reach the tolerance in %d iterations", maxit);
    if (rc) return td_fail(ctx, rc, "tdbem_solve failed");
    return TDBEM_OK;
}

extern "C" int tdbem_tensor_save(tdbem_tensor_t t, const char *path) {
    if (!t || !path) return TDBEM_ERR_ARG;
    tdbem_ctx *ctx = t->ctx;
    TD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    FILE *f = fopen(path, "wb");
    if (!f) return td_fail(ctx, TDBEM_ERR_ARG, "cannot open %s for writing", path);
    int64_t used = 0;
    cudaMemcpy(&used, t->dface_used, sizeof(int64_t), cudaMemcpyDeviceToHost);
    const size_t es = t->prec == TDBEM_FP64 ? sizeof(c64) : sizeof(c32);
    const int32_t hdr_i[8] = {t->op, t->prec, t->ng, t->Nu, t->NQ, t->kcap, t->max_near_rows, 0};
    const int64_t hdr_l[4] = {t->nrows, t->ncols, t->nblocks, used};
    bool ok = wr(f, kTensorMagic, 8) && wr(f, hdr_i, sizeof hdr_i) && wr(f, hdr_l, sizeof hdr_l) && wr(f, &t->c, sizeof(double)) &&
              wr(f, &t->stats, sizeof t->stats) && wr(f, t->blocks.data(), sizeof(int32_t) * 5 * t->nblocks) &&
              wr(f, t->rank.data(), sizeof(int32_t) * t->nblocks) && wr(f, t->frank_sum.data(), sizeof(int32_t) * t->nblocks) &&
              wr_dev(f, t->dperm_r, t->nrows) && wr_dev(f, t->dperm_c, t->ncols) && wr_dev(f, t->dinv_r, t->nrows) &&
              wr_dev(f, t->dinv_c, t->ncols) && wr_dev(f, t->drank, t->nblocks) && wr_dev(f, t->dkpiv, t->nblocks * t->Nu) &&
              wr_dev(f, t->dfrank, t->nblocks * t->Nu) && wr_dev(f, t->dfoff, t->nblocks * t->Nu) &&
              wr_dev(f, t->dpartner, t->NQ) && wr_dev(f, (const char *)t->dfib, es * t->nblocks * t->Nu * t->Nu) &&
              wr_dev(f, (const char *)t->dface, es * used);
    fclose(f);
    return ok ? TDBEM_OK : td_fail(ctx, TDBEM_ERR_CUDA, "writing %s failed", path);
}

extern "C" int tdbem_tensor_info(tdbem_tensor_t t, int32_t *op, int32_t *prec, int64_t *nrows, int64_t *ncols,
                                 int32_t *NQ, int32_t *Nu) {
    if (!t) return TDBEM_ERR_ARG;
    if (op) *op = t->op;
    if (prec) *prec = t->prec;
    if (nrows) *nrows = t->nrows;
    if (ncols) *ncols = t->ncols;
    if (NQ) *NQ = t->NQ;
    if (Nu) *Nu = t->Nu;
    return TDBEM_OK;
}

extern "C" int tdbem_tensor_load(tdbem_ctx_t ctx, const char *path, tdbem_tensor_t *out) {
    if (!ctx || !path || !out) return TDBEM_ERR_ARG;
    *out = nullptr;
    FILE *f = fopen(path, "rb");
    if (!f) return td_fail(ctx, TDBEM_ERR_ARG, "cannot open %s", path);
    char magic[8];
    int32_t hi[8];
    int64_t hl[4];
    tdbem_tensor *t = new (std::nothrow) tdbem_tensor();
    bool ok = t && rd(f, magic, 8) && !memcmp(magic, kTensorMagic, 8) && rd(f, hi, sizeof hi) && rd(f, hl, sizeof hl);
    if (!ok) {
        fclose(f);
        delete t;
        return td_fail(ctx, TDBEM_ERR_ARG, "%s is not a tensor file of this version", path);
    }
    // sizes must be plausible and account for the file's length exactly
    {
        const int64_t nb = hl[2], nr = hl[0], nc = hl[1], used = hl[3];
        const int Nu = hi[3], NQ = hi[4];
        const bool sane = (hi[0] == TDBEM_SLP || hi[0] == TDBEM_DLP || hi[0] == TDBEM_ADLP) && (hi[1] == TDBEM_FP64 || hi[1] == TDBEM_MIXED) &&
                          Nu >= 1 && Nu <= 256 && NQ >= Nu && NQ <= (1 << 20) && nb >= 1 && nb < (1LL << 31) &&
                          nr >= 1 && nr < (1LL << 31) && nc >= 1 && nc < (1LL << 31) && used >= 0 && used < (1LL << 40);
        const long here = ftell(f);
        const int64_t es = hi[1] == TDBEM_FP64 ? 16 : 8;
        const int64_t expect = here + 8 + (int64_t)sizeof(tdbem_stats) + 4 * (7 * nb) + 4 * (2 * nr + 2 * nc) +
                               4 * nb * (1 + 2 * (int64_t)Nu) + 8 * nb * Nu + 4 * (int64_t)NQ +
                               es * (nb * Nu * Nu + used);
        bool size_ok = false;
        if (sane && here > 0 && fseek(f, 0, SEEK_END) == 0) {
            size_ok = ftell(f) == expect;
            fseek(f, here, SEEK_SET);
        }
        if (!sane || !size_ok) {
            fclose(f);
            delete t;
            return td_fail(ctx, TDBEM_ERR_ARG, "%s: header sizes do not match the file", path);
        }
    }
    t->ctx = ctx;
    t->op = hi[0];
    t->prec = hi[1];
    t->ng = hi[2];
    t->Nu = hi[3];
    t->NQ = hi[4];
    t->kcap = hi[5];
    t->max_near_rows = hi[6];
    t->nrows = hl[0];
    t->ncols = hl[1];
    t->nblocks = hl[2];
    const int64_t used = hl[3], nb = t->nblocks;
    const size_t es = t->prec == TDBEM_FP64 ? sizeof(c64) : sizeof(c32);
    t->blocks.resize(5 * nb);
    t->rank.resize(nb);
    t->frank_sum.resize(nb);
    auto alloc = [&](void **p, size_t bytes) {
        if (cudaMalloc(p, std::max<size_t>(bytes, 1)) != cudaSuccess) return false;
        t->owned.push_back(*p);
        return true;
    };
    ok = rd(f, &t->c, sizeof(double)) && rd(f, &t->stats, sizeof t->stats) &&
         rd(f, t->blocks.data(), sizeof(int32_t) * 5 * nb) && rd(f, t->rank.data(), sizeof(int32_t) * nb) &&
         rd(f, t->frank_sum.data(), sizeof(int32_t) * nb) && alloc((void **)&t->dblocks, sizeof(int32_t) * 5 * nb) &&
         alloc((void **)&t->dperm_r, sizeof(int32_t) * t->nrows) && alloc((void **)&t->dperm_c, sizeof(int32_t) * t->ncols) &&
         alloc((void **)&t->dinv_r, sizeof(int32_t) * t->nrows) && alloc((void **)&t->dinv_c, sizeof(int32_t) * t->ncols) &&
         alloc((void **)&t->drank, sizeof(int32_t) * nb) && alloc((void **)&t->dkpiv, sizeof(int32_t) * nb * t->Nu) &&
         alloc((void **)&t->dfrank, sizeof(int32_t) * nb * t->Nu) && alloc((void **)&t->dfoff, sizeof(int64_t) * nb * t->Nu) &&
         alloc((void **)&t->dpartner, sizeof(int32_t) * (t->NQ + 1)) && alloc(&t->dfib, es * nb * t->Nu * t->Nu) &&
         alloc(&t->dface, es * used) && alloc((void **)&t->dface_used, sizeof(int64_t) * 2) &&
         cudaMemcpy(t->dblocks, t->blocks.data(), sizeof(int32_t) * 5 * nb, cudaMemcpyHostToDevice) == cudaSuccess &&
         rd_dev(f, t->dperm_r, t->nrows) && rd_dev(f, t->dperm_c, t->ncols) && rd_dev(f, t->dinv_r, t->nrows) &&
         rd_dev(f, t->dinv_c, t->ncols) && rd_dev(f, t->drank, nb) && rd_dev(f, t->dkpiv, nb * t->Nu) &&
         rd_dev(f, t->dfrank, nb * t->Nu) && rd_dev(f, t->dfoff, nb * t->Nu) && rd_dev(f, t->dpartner, t->NQ) &&
         rd_dev(f, (char *)t->dfib, es * nb * t->Nu * t->Nu) && rd_dev(f, (char *)t->dface, es * used) &&
         cudaMemcpy(t->dface_used, &used, sizeof(int64_t), cudaMemcpyHostToDevice) == cudaSuccess;
    fclose(f);
    if (!ok) {
        cudaGetLastError();
        for (void *p : t->owned) cudaFree(p);
        delete t;
        return td_fail(ctx, TDBEM_ERR_ARG, "reading %s failed", path);
    }
    t->face_cap = used;
    if (const int rc = td_upload_order(t)) {
        for (void *p : t->owned) cudaFree(p);
        delete t;
        return rc;
    }
    *out = t;
    return TDBEM_OK;
}

extern "C" int tdbem_model_save(tdbem_model_t m, const char *path) {
    if (!m || !path) return TDBEM_ERR_ARG;
    std::vector<float> p(TD_MLP_NPARAMS);
    int rc = tdbem_model_get_params(m, p.data());
    if (rc) return rc;
    FILE *f = fopen(path, "wb");
    if (!f) return TDBEM_ERR_ARG;
    const int32_t n = TD_MLP_NPARAMS;
    const bool ok = wr(f, kModelMagic, 8) && wr(f, &n, sizeof n) && wr(f, p.data(), sizeof(float) * n);
    fclose(f);
    return ok ? TDBEM_OK : TDBEM_ERR_ARG;
}

extern "C" int tdbem_model_load(tdbem_ctx_t ctx, const char *path, tdbem_model_t *out) {
    if (!ctx || !path || !out) return TDBEM_ERR_ARG;
    *out = nullptr;
    FILE *f = fopen(path, "rb");
    if (!f) return td_fail(ctx, TDBEM_ERR_ARG, "cannot open %s", path);
    char magic[8];
    int32_t n = 0;
    std::vector<float> p(TD_MLP_NPARAMS);
    const bool ok = rd(f, magic, 8) && !memcmp(magic, kModelMagic, 8) && rd(f, &n, sizeof n) && n == TD_MLP_NPARAMS &&
                    rd(f, p.data(), sizeof(float) * n);
    fclose(f);
    if (!ok) return td_fail(ctx, TDBEM_ERR_ARG, "%s is not a model file of this version", path);
    int rc = tdbem_model_create(ctx, 0, out);
    if (rc) return rc;
    return tdbem_model_set_params(*out, p.data());
}
