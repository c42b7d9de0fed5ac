// Compressed multi-frequency apply (eq. product):
//   y = sum_{l < NQ} A(s_l) W_l = sum_b sum_d [ H_d z1_d + conj(H_d) z2_d ]_I,
//   z1_d = sum_{l: s_l = s_u}       f_d[u] W_l[J],
//   z2_d = sum_{l: s_l = conj(s_u)} conj(f_d[u]) W_l[J],
// using A(conj s) = conj A(s) for the conjugate half of the frequency set.
// Far faces H_d = U_d V_d^T are applied as U_d (V_d^T z1) + conj(U_d) (V_d^H z2).
// One CTA per block: the block's W columns are streamed tile by tile (TJ
// columns, all NQ frequencies) through shared memory, the frequency
// contraction of every term is done on the tile, then contracted with the
// face (near) or V (far); results are added to y with atomics.
#include <algorithm>

#include "internal.h"
#include "kernels.h"

namespace {

TD_D void atomic_add_c(c64 *p, c64 v) {
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}
TD_D void atomic_add_c(c32 *p, c32 v) { atomicAdd(reinterpret_cast<float2 *>(p), make_float2(v.x, v.y)); }

// FP64 weighted apply.  Dynamic shared memory layout (complex units):
//   Wt [NQ][TJ][nrhs] | z [RC][2][TJ][nrhs] | acc: near [nI][nrhs] or far [sumk][2][nrhs]
__global__ void __launch_bounds__(256) k_apply(ApplyArgs a, TensorOut o, int TJ, int RC) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c64 *sm = reinterpret_cast<c64 *>(smem_raw);
    const int NQ = a.NQ;
    const int nrhs = a.nrhs, Nu = a.Nu;
    const c64 *W = (const c64 *)a.W;
    c64 *y = (c64 *)a.y;
    const c64 *fib = (const c64 *)o.fib;
    const c64 *pool = (const c64 *)o.face;
    c64 *Wt = sm;
    c64 *z = Wt + (int64_t)NQ * TJ * nrhs;
    c64 *acc = z + (int64_t)RC * 2 * TJ * nrhs;
    c64 *fq_s = acc + a.acc_max;                                   // [RC][NQ]
    int *sg_s = reinterpret_cast<int *>(fq_s + (int64_t)RC * NQ);    // [NQ]
    const int tid = threadIdx.x;
    for (int b = blockIdx.x; b < a.nb; b += gridDim.x) {
        const int *bl = a.blocks + 5 * b;
        const int nI = bl[1] - bl[0], nJ = bl[3] - bl[2];
        const bool far = bl[4] != 0;
        const int r = o.rank[b];
        const int64_t tb = (int64_t)b * Nu;
        for (int d0 = 0; d0 < r; d0 += RC) {
            const int rc = min(RC, r - d0);
            // accumulator size for this chunk
            int sumk = 0;
            if (far)
                for (int d = d0; d < d0 + rc; ++d) sumk += o.frank[tb + d];
            const int nacc = far ? sumk * 2 * nrhs : nI * nrhs;
            for (int e = tid; e < nacc; e += blockDim.x) acc[e] = {0, 0};
            // fibre value per point of the frequency list (conjugated for the
            // conjugate half) and the half it belongs to
            for (int e = tid; e < rc * NQ; e += blockDim.x) {
                const int q = e % NQ, dd = e / NQ;
                const int mp = a.qmap[q];
                const c64 fv = fib[(tb + d0 + dd) * Nu + (mp > 0 ? mp - 1 : -mp - 1)];
                fq_s[e] = mp > 0 ? fv : cconj(fv);
                if (dd == 0) sg_s[q] = mp > 0 ? 1 : -1;
            }
            for (int j0 = 0; j0 < nJ; j0 += TJ) {
                const int tj = min(TJ, nJ - j0);
                __syncthreads();
                for (int e = tid; e < NQ * tj * nrhs; e += blockDim.x) {
                    const int c = e % nrhs, jj = (e / nrhs) % tj, q = e / (nrhs * tj);
                    const int64_t col = a.perm_c[bl[2] + j0 + jj];
                    Wt[((int64_t)q * TJ + jj) * nrhs + c] = W[((int64_t)q * a.ncols + col) * nrhs + c];
                }
                __syncthreads();
                // frequency contraction of the tile for the chunk's terms; the
                // per-point fibre coefficients were staged in shared memory
                for (int e = tid; e < rc * tj * nrhs; e += blockDim.x) {
                    const int c = e % nrhs, jj = (e / nrhs) % tj, dd = e / (nrhs * tj);
                    const c64 *fq = fq_s + (int64_t)dd * NQ;
                    c64 z1 = {0, 0}, z2 = {0, 0};
#pragma unroll 4
                    for (int q = 0; q < NQ; ++q) {
                        const c64 w = Wt[((int64_t)q * TJ + jj) * nrhs + c];
                        if (sg_s[q] > 0) cfma(z1, fq[q], w);
                        else cfma(z2, fq[q], w);
                    }
                    z[(((int64_t)dd * 2 + 0) * TJ + jj) * nrhs + c] = z1;
                    z[(((int64_t)dd * 2 + 1) * TJ + jj) * nrhs + c] = z2;
                }
                __syncthreads();
                if (!far) {
                    for (int e = tid; e < nI * nrhs; e += blockDim.x) {
                        const int c = e % nrhs, i = e / nrhs;
                        c64 s = acc[e];
                        for (int dd = 0; dd < rc; ++dd) {
                            const c64 *H = pool + o.foff[tb + d0 + dd] + (int64_t)i * nJ + j0;
                            for (int jj = 0; jj < tj; ++jj) {
                                const c64 h = H[jj];
                                cfma(s, h, z[(((int64_t)dd * 2 + 0) * TJ + jj) * nrhs + c]);
                                cfma(s, cconj(h), z[(((int64_t)dd * 2 + 1) * TJ + jj) * nrhs + c]);
                            }
                        }
                        acc[e] = s;
                    }
                } else {
                    // acc[(tau, p, c)] += sum_j V[tau][j] z_p[j][c]  (p = 1 uses conj V)
                    for (int e = tid; e < sumk * nrhs; e += blockDim.x) {
                        const int c = e % nrhs;
                        int t = e / nrhs, dd = 0;
                        while (t >= o.frank[tb + d0 + dd]) {
                            t -= o.frank[tb + d0 + dd];
                            ++dd;
                        }
                        const int kd = o.frank[tb + d0 + dd];
                        const c64 *V = pool + o.foff[tb + d0 + dd] + (int64_t)kd * nI + (int64_t)t * nJ + j0;
                        c64 s1 = acc[(e / nrhs) * 2 * nrhs + c], s2 = acc[(e / nrhs) * 2 * nrhs + nrhs + c];
                        for (int jj = 0; jj < tj; ++jj) {
                            const c64 v = V[jj];
                            cfma(s1, v, z[(((int64_t)dd * 2 + 0) * TJ + jj) * nrhs + c]);
                            cfma(s2, cconj(v), z[(((int64_t)dd * 2 + 1) * TJ + jj) * nrhs + c]);
                        }
                        acc[(e / nrhs) * 2 * nrhs + c] = s1;
                        acc[(e / nrhs) * 2 * nrhs + nrhs + c] = s2;
                    }
                }
            }
            __syncthreads();
            if (!far) {
                for (int e = tid; e < nI * nrhs; e += blockDim.x) {
                    const int c = e % nrhs, i = e / nrhs;
                    atomic_add_c(y + (int64_t)a.perm_r[bl[0] + i] * nrhs + c, acc[e]);
                }
            } else {
                for (int e = tid; e < nI * nrhs; e += blockDim.x) {
                    const int c = e % nrhs, i = e / nrhs;
                    c64 s = {0, 0};
                    int base = 0;
                    for (int dd = 0; dd < rc; ++dd) {
                        const int kd = o.frank[tb + d0 + dd];
                        const c64 *U = pool + o.foff[tb + d0 + dd];
                        for (int t = 0; t < kd; ++t) {
                            const c64 u = U[(int64_t)t * nI + i];
                            cfma(s, u, acc[(int64_t)(base + t) * 2 * nrhs + c]);
                            cfma(s, cconj(u), acc[(int64_t)(base + t) * 2 * nrhs + nrhs + c]);
                        }
                        base += kd;
                    }
                    atomic_add_c(y + (int64_t)a.perm_r[bl[0] + i] * nrhs + c, s);
                }
            }
            __syncthreads();
        }
    }
}

// y += A(s_f) x at one point of the list: sum_d f_d[f] H_d x, one CTA per block.
// Both kinds of block multiply a tile A of rows with x in shared memory, the threads
// (row, part of the columns), the parts' sums meeting in shared memory:
//   near: A = sum_d f_d H_d, combined as it is read (contiguous loads, all lanes
//         busy for any width), rows of y;
//   far:  A = rows of the V_d (asynchronous copies), t = f_d (V_d x) kept in shared
//         memory; then rows of y from U, threads along i (coalesced), CTAs of
//         short blocks splitting the factor rows over thread groups.
// CC right-hand sides per pass over the faces.  A conjugate point takes conj(x)
// and conjugates its result.  Bound: HBM (every face read once per pass) for long
// blocks, the chain of dependent loads and the instructions for short ones.
// 5120-triangle sphere, 4 right-hand sides (14,488 blocks of 1800 values): 400 us by
// the general kernel -> 193 us with a warp per row (a reduction per row, lanes idle in
// rows of 20 to 40 values) -> 134 us, 103 with the largest blocks first; 30k housing,
// 8 frequencies, 1 right-hand side (142M stored values): 1043 -> 340 -> 274, 244 us.
constexpr int kOneT = 128, kOneD = 32;  // factor rows, terms in shared memory at a time
constexpr int kOneBytes = 12288;                     // the tile A

TD_D void copy_async(c32 *dst, const c32 *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
TD_D void copy_async(c64 *dst, const c64 *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

template <class T, int CC>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 8 : 5) k_apply_one(ApplyArgs a, TensorOut o, int c0) {
    constexpr int kH = kOneBytes / (int)sizeof(cx<T>), kOneJ = CC == 4 ? 128 : 256;  // tile, columns of x
    constexpr int kDQ = sizeof(T) == 8 ? 1 : CC == 1 ? 3 : 2, kUQ = CC == 1 ? 8 : 4;  // terms of a near tile, loads of U in flight
    __shared__ alignas(16) cx<T> h[kH];
    __shared__ alignas(16) cx<T> xs[kOneJ][CC];
    __shared__ alignas(16) cx<T> ts[kOneT][CC];
    __shared__ alignas(16) cx<T> red[128][CC];
    __shared__ cx<T> fs[kOneD];
    __shared__ long long off[kOneD], rowoff[kOneT];
    __shared__ int pre[kOneD + 1], rowd[kOneT];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, b = a.order[blockIdx.x];
    const int64_t tb = (int64_t)b * a.Nu;
    const int mp = a.qmap[a.single_f];
    const bool cj = mp < 0;
    const int u = (cj ? -mp : mp) - 1;
    // the first terms' data, before the number of terms is known
    cx<T> pf = {0, 0};
    long long po = 0;
    int pk = 0;
    if (tid < min(kOneD, a.Nu)) {
        pf = ((const cx<T> *)o.fib)[(tb + tid) * a.Nu + u];
        po = o.foff[tb + tid];
        pk = o.frank[tb + tid];
    }
    const int rb = o.rank[b];
    const int *bl = a.blocks + 5 * b;
    const int nI = bl[1] - bl[0], nJ = bl[3] - bl[2], nrhs = a.nrhs;
    const bool far = bl[4] != 0;
    const int nc = min(CC, nrhs - c0);
    const int *perm = a.perm_r + bl[0];
    const cx<T> *x = (const cx<T> *)a.W, *pool = (const cx<T> *)o.face;
    cx<T> *y = (cx<T> *)a.y;
    int loaded = -1;  // first column of the x tile in shared memory
    auto load_x = [&](int j0, int tj) {  // (the caller synchronises before the tile is read)
        if (loaded == j0) return;
        if (loaded >= 0) __syncthreads();
        loaded = j0;
        for (int e = tid; e < tj * CC; e += 128) {
            const int j = e / CC, c = e - j * CC;
            cx<T> v = {0, 0};
            if (c < nc) v = x[(int64_t)a.perm_c[bl[2] + j0 + j] * nrhs + c0 + c];
            xs[j][c] = cj ? cconj(v) : v;
        }
    };
    // the product of the tile's ti rows with the x tile, by parts of the columns, to red;
    // one thread per (row, column) then takes the sum of the parts
    auto product = [&](int ti, int tj, int ld, auto take) {
        const int P = 128 / ti, part = tid / ti, row = tid - part * ti;
        cx<T> acc[CC];
#pragma unroll
        for (int c = 0; c < CC; ++c) acc[c] = cx<T>{0, 0};
        if (part < P) {
            const cx<T> *hr = h + row * ld;
#pragma unroll (CC == 4 ? 2 : 4)
            for (int j = part; j < tj; j += P) {
                const cx<T> v = hr[j];
#pragma unroll
                for (int c = 0; c < CC; ++c) cfma(acc[c], v, xs[j][c]);
            }
        }
#pragma unroll
        for (int c = 0; c < CC; ++c) red[tid][c] = acc[c];
        __syncthreads();
        for (int e = tid; e < ti * CC; e += 128) {
            const int i = e / CC, c = e - i * CC;
            cx<T> s = red[i][c];
            for (int q = 1; q < P; ++q) s = s + red[q * ti + i][c];
            take(i, c, s);
        }
    };
    for (int d0 = 0; d0 < rb; d0 += kOneD) {
        const int r = min(kOneD, rb - d0);
        if (d0 > 0) {
            __syncthreads();
            if (tid < r) {
                pf = ((const cx<T> *)o.fib)[(tb + d0 + tid) * a.Nu + u];
                po = o.foff[tb + d0 + tid];
                pk = o.frank[tb + d0 + tid];
            }
        }
        if (tid < r) {
            fs[tid] = pf;
            off[tid] = po;
        }
        if (wid == 0) {  // inclusive prefix of the face ranks
            int k = far && lane < r ? pk : 0;
            for (int s = 1; s < 32; s <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, k, s);
                if (lane >= s) k += v;
            }
            if (lane == 0) pre[0] = 0;
            pre[lane + 1] = k;
        }
        load_x(0, min(kOneJ, nJ));
        __syncthreads();
        if (!far) {
            for (int j0 = 0; j0 < nJ; j0 += kOneJ) {
                const int tj = min(kOneJ, nJ - j0), ld = tj | 1, rows = min(128, kH / ld);
                const float inv = 1.0f / (float)tj;
                load_x(j0, tj);
                for (int i0 = 0; i0 < nI; i0 += rows) {
                    const int ti = min(rows, nI - i0), n = ti * tj;
                    const cx<T> *hb = pool + (int64_t)i0 * nJ + j0;
                    for (int e0 = tid; e0 < n; e0 += 4 * 128) {
                        int src[4], dst[4];
                        cx<T> acc[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            // (row: exact, e0 < 2^11 and tj <= 256)
                            const int e = e0 + 128 * q, i = (int)(((float)e + 0.5f) * inv), j = e - i * tj;
                            src[q] = e < n ? i * nJ + j : -1;
                            dst[q] = i * ld + j;
                            acc[q] = cx<T>{0, 0};
                        }
                        for (int d = 0; d < r; d += kDQ) {
                            cx<T> v[kDQ][4] = {};
#pragma unroll
                            for (int s = 0; s < kDQ; ++s)
                                if (d + s < r) {
                                    const cx<T> *p = hb + off[d + s];
#pragma unroll
                                    for (int q = 0; q < 4; ++q)
                                        if (src[q] >= 0) v[s][q] = p[src[q]];
                                }
#pragma unroll
                            for (int s = 0; s < kDQ; ++s)
                                if (d + s < r) {
#pragma unroll
                                    for (int q = 0; q < 4; ++q) cfma(acc[q], fs[d + s], v[s][q]);
                                }
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (src[q] >= 0) h[dst[q]] = acc[q];
                    }
                    const int yr = tid < ti * CC ? perm[i0 + tid / CC] : 0;
                    __syncthreads();
                    product(ti, tj, ld, [&](int i, int c, cx<T> s) {
                        const int row = i == tid / CC ? yr : perm[i0 + i];
                        if (c < nc) atomic_add_c(y + (int64_t)row * nrhs + c0 + c, cj ? cconj(s) : s);
                    });
                }
            }
            continue;
        }
        const int R = pre[r];
        for (int r0 = 0; r0 < R; r0 += kOneT) {
            const int rc = min(kOneT, R - r0);
            if (tid < rc) {
                int d = 0;
                while (r0 + tid >= pre[d + 1]) ++d;
                rowd[tid] = d;
                rowoff[tid] = off[d] + (int64_t)(pre[d + 1] - pre[d]) * nI + (int64_t)(r0 + tid - pre[d]) * nJ;
            }
            __syncthreads();
            for (int j0 = 0; j0 < nJ; j0 += kOneJ) {
                const int tj = min(kOneJ, nJ - j0), ld = tj | 1, rows = min(128, kH / ld);
                const float inv = 1.0f / (float)tj;
                load_x(j0, tj);
                for (int i0 = 0; i0 < rc; i0 += rows) {
                    const int ti = min(rows, rc - i0), n = ti * tj;
#pragma unroll 4
                    for (int e = tid; e < n; e += 128) {
                        const int i = (int)(((float)e + 0.5f) * inv), j = e - i * tj;
                        copy_async(h + i * ld + j, pool + rowoff[i0 + i] + j0 + j);
                    }
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    __syncthreads();
                    product(ti, tj, ld, [&](int i, int c, cx<T> s) {
                        const cx<T> v = fs[rowd[i0 + i]] * s;
                        ts[i0 + i][c] = j0 == 0 ? v : ts[i0 + i][c] + v;
                    });
                }
            }
            __syncthreads();
            // rows of y: groups of gi threads along i, each a part of the factor rows
            const int gi = nI >= 128 ? 128 : (nI + 31) & ~31, G = 128 / gi;
            const int g = tid / gi;
            cx<T> own[CC];
            int yrow = 0;
            if (g < G) {
                const int per = (rc + G - 1) / G, tA = min(rc, g * per), tB = min(rc, tA + per);
                for (int i = tid - g * gi; i < nI && (tA < tB || G > 1); i += gi) {
                    if (g == 0) yrow = perm[i];
                    cx<T> acc[CC];
#pragma unroll
                    for (int c = 0; c < CC; ++c) acc[c] = cx<T>{0, 0};
                    for (int t = tA; t < tB;) {
                        const int d = rowd[t];
                        // a run of factor rows of one term is contiguous
                        const int te = min(tB, pre[d + 1] - r0), n = te - t;
                        const cx<T> *ub = pool + off[d] + (int64_t)(r0 + t - pre[d]) * nI + i;
                        int q = 0;
                        for (; q + kUQ <= n; q += kUQ) {
                            cx<T> uv[kUQ];
#pragma unroll
                            for (int e = 0; e < kUQ; ++e) uv[e] = ub[(int64_t)(q + e) * nI];
#pragma unroll
                            for (int e = 0; e < kUQ; ++e)
#pragma unroll
                                for (int c = 0; c < CC; ++c) cfma(acc[c], uv[e], ts[t + q + e][c]);
                        }
                        for (; q < n; ++q) {
                            const cx<T> uv = ub[(int64_t)q * nI];
#pragma unroll
                            for (int c = 0; c < CC; ++c) cfma(acc[c], uv, ts[t + q][c]);
                        }
                        t = te;
                    }
                    if (G == 1) {
#pragma unroll
                        for (int c = 0; c < CC; ++c)
                            if (c < nc) atomic_add_c(y + (int64_t)yrow * nrhs + c0 + c, cj ? cconj(acc[c]) : acc[c]);
                    }
#pragma unroll
                    for (int c = 0; c < CC; ++c) {
                        own[c] = acc[c];
                        if (g > 0) red[tid - gi][c] = acc[c];  // (G > 1: one i per thread)
                    }
                }
            }
            __syncthreads();
            if (G > 1) {  // the groups' sums meet: one atomic add per output
                if (g == 0 && tid < nI) {
                    for (int q = 1; q < G; ++q)
#pragma unroll
                        for (int c = 0; c < CC; ++c) own[c] = own[c] + red[(q - 1) * gi + tid][c];
#pragma unroll
                    for (int c = 0; c < CC; ++c)
                        if (c < nc) atomic_add_c(y + (int64_t)yrow * nrhs + c0 + c, cj ? cconj(own[c]) : own[c]);
                }
                __syncthreads();
            }
        }
    }
}

// Second phase of the tensor-core apply.  The frequency contraction
// z_(b,d,p) = sum_l f_d(l) W_l[J] is already in Z (k_zgemm.cu); Z rows of a
// block are (term d, half p) at zbase[b] + p zpstride[b] + d nJ nrhs.  Both face
// stages are small complex GEMMs out[m][(p, c)] = sum_k A_p[m][k] B[k][(p, c)]
// with A_1 = conj(A_0) for the conjugate half:
//   stage 0 (one CTA per far term):  T_p = V_d^T z_p, m = tau < k_d, k = j < |J|,
//            written to T;
//   stage 1 (one CTA per block):      y_I += sum_d U_d T_(d,1) + conj(U_d) T_(d,2)
//            (far; k = (d, tau)) or y_I += sum_d H_d z_(d,1) + conj(H_d) z_(d,2)
//            (near; k = (d, j)); both halves summed before one atomic add per
//            output.
// The k of all terms run through one chunked loop (no padding per term): each
// k has a descriptor (A column, B row), chunks of 32 are brought to shared memory
// by asynchronous copies in two stages.  Four warps of 4 x (4 or 8 or 2) register
// tiles, 16 rows each: M <= 16 rows take one row tile with k split over the four
// warps, M <= 32 two and two, else four row tiles; the warps' sums meet in shared
// memory.  conj(a) b is formed as conj(a conj(b)): the sign goes on b when it is
// loaded and on the result, not on every product.  Fixed tiles of 64 rows spent
// three quarters of stage 0 on padding (k_d is 16 on average): 30k housing, 16
// right-hand sides: both stages 23.2 -> 11.5 ms.  Bound: FP32 FMA.
constexpr int kFK = 32, kFA = kFK + 2;  // k per chunk; A row stride (16-byte reads of 4 rows conflict-free)
constexpr int kFY = 4;                  // CTAs that share a large block's row tiles (stage 1)

struct FaceK {
    const c32 *A, *B;  // column k of A (row stride per job), row k of B (half 0)
    int64_t sB;        // offset of the half-1 row
};
template <int CQ>
struct FaceSmem {
    static constexpr int NC = 8 * CQ;
    c32 A[2][64][kFA];
    c32 B[2][kFK][NC];
    FaceK kd[2][kFK];
};

TD_D void cp_async(void *dst, const void *src, int bytes, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (bytes == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(valid ? 8 : 0) : "memory");
}

template <int CQ>
__global__ void __launch_bounds__(128) k_apply_faces(ApplyZArgs a, TensorOut o, int stage, int col0) {
    using Smem = FaceSmem<CQ>;
    constexpr int NC = Smem::NC;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem &S = *reinterpret_cast<Smem *>(smem_raw);
    const int nrhs = a.nrhs, Nu = a.Nu, ncol = min(NC, a.rpt * nrhs - col0);
    const c32 *pool = (const c32 *)o.face;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, tx = lane & 7, ry = lane >> 3;
    // columns 2 tx + 16 h + {0, 1} of this thread: sign of the conjugate half
    float sgn[CQ];
#pragma unroll
    for (int q = 0; q < CQ; ++q) sgn[q] = col0 + 2 * tx + 16 * (q >> 1) + (q & 1) >= nrhs ? -1.0f : 1.0f;
    // 16-byte copies of B rows: two columns of one half
    const bool wide = (nrhs & 1) == 0 && (ncol & 1) == 0;
    int b, d0, d1;
    if (stage == 0) {
        const int2 bd = a.ftab[blockIdx.x];
        b = bd.x;
        d0 = bd.y;
        d1 = bd.y + 1;
    } else {
        b = a.order[blockIdx.x];
        d0 = 0;
        d1 = o.rank[b];
        if (d1 == 0 || a.zbase[b] < 0) return;
    }
    const int *bl = a.blocks + 5 * b;
    const int nI = bl[1] - bl[0], nJ = bl[3] - bl[2];
    const bool far = bl[4] != 0, ucol = stage == 1 && far;
    const int64_t tb = (int64_t)b * Nu, L = (int64_t)nJ * nrhs;
    const int M = stage == 0 ? o.frank[tb + d0] : nI;
    const int64_t sA = ucol ? 1 : nJ;  // row stride of A
    if ((int)blockIdx.y * 64 >= M) return;
    for (int e = tid; e < 2 * kFK * NC; e += 128) (&S.B[0][0][0])[e] = c32{0.f, 0.f};  // columns beyond ncol stay 0
    int K = 0;
    if (ucol)
        for (int d = 0; d < d1; ++d) K += o.frank[tb + d];
    else
        K = (d1 - d0) * nJ;
    // descriptor of k; its term is found from the last one's (k ascends)
    int dk = d0, kbase = 0;  // threads < 32
    auto describe = [&](int chunk) {
        const int k = chunk * kFK + tid;
        if (tid >= kFK || k >= K) return;
        FaceK f;
        if (ucol) {
            int kd = o.frank[tb + dk];
            while (k - kbase >= kd) {
                kbase += kd;
                kd = o.frank[tb + ++dk];
            }
            const int t = k - kbase;
            f.A = pool + o.foff[tb + dk] + (int64_t)t * nI;
            f.B = a.T + a.toff[tb + dk] + (int64_t)t * nrhs;
            f.sB = (int64_t)kd * nrhs;
        } else {
            const int d = d0 + k / nJ, j = k - (k / nJ) * nJ;
            f.A = pool + o.foff[tb + d] + (stage == 0 ? (int64_t)M * nI : 0) + j;
            f.B = a.Z + a.zbase[b] + (int64_t)d * L + (int64_t)j * nrhs;
            f.sB = a.zpstride[b];
        }
        S.kd[chunk & 1][tid] = f;
    };
    const int nchunk = (K + kFK - 1) / kFK;
    for (int m0 = blockIdx.y * 64; m0 < M; m0 += 64 * gridDim.y) {
        const int mc = min(64, M - m0);
        const int WR = mc <= 16 ? 1 : mc <= 32 ? 2 : 4, WK = 4 / WR, R = 16 * WR;
        const int wr = wid % WR, wk = wid / WR;
        auto stage_in = [&](int chunk) {
            const int buf = chunk & 1, kc = min(kFK, K - chunk * kFK);
            for (int e = tid; e < R * kFK; e += 128) {
                // consecutive lanes take consecutive addresses: rows of U, columns of V and H
                const int m = ucol ? e % R : e / kFK, k = ucol ? e / R : e % kFK;
                const bool ok = k < kc && m < mc;
                cp_async(&S.A[buf][m][k], ok ? S.kd[buf][k].A + (int64_t)(m0 + m) * sA : pool, 8, ok);
            }
            const int per = wide ? 2 : 1, nn = (ncol + per - 1) / per;
            for (int e = tid; e < kFK * nn; e += 128) {
                const int k = e / nn, n = (e - k * nn) * per, g = col0 + n, p = g >= nrhs ? 1 : 0;
                const bool ok = k < kc;
                cp_async(&S.B[buf][k][n], ok ? S.kd[buf][k].B + p * S.kd[buf][k].sB + g - p * nrhs : pool, 8 * per, ok);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        c32 acc[4][CQ];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int q = 0; q < CQ; ++q) acc[x][q] = c32{0.f, 0.f};
        __syncthreads();  // shared memory is free
        dk = d0;
        kbase = 0;
        describe(0);
        describe(1);
        __syncthreads();
        if (nchunk > 0) stage_in(0);
        for (int ch = 0; ch < nchunk; ++ch) {
            if (ch + 1 < nchunk) {
                stage_in(ch + 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            const int buf = ch & 1, k1 = (wk + 1) * (kFK / WK);
#pragma unroll 2
            for (int k = wk * (kFK / WK); k < k1; k += 2) {
                float4 av[4];  // rows 16 wr + ry + 4 x at k and k + 1
#pragma unroll
                for (int x = 0; x < 4; ++x) av[x] = *reinterpret_cast<const float4 *>(&S.A[buf][16 * wr + ry + 4 * x][k]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    c32 bv[CQ];
#pragma unroll
                    for (int q = 0; q < CQ; q += 2) {
                        const float4 v = *reinterpret_cast<const float4 *>(&S.B[buf][k + h][2 * tx + 8 * q]);
                        bv[q] = c32{v.x, v.y * sgn[q]};
                        bv[q + 1] = c32{v.z, v.w * sgn[q + 1]};
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const c32 ax = h == 0 ? c32{av[x].x, av[x].y} : c32{av[x].z, av[x].w};
#pragma unroll
                        for (int q = 0; q < CQ; ++q) cfma(acc[x][q], ax, bv[q]);
                    }
                }
            }
            describe(ch + 2);
            __syncthreads();  // the stage is refilled, its descriptors replaced
        }
        // ---- the warps' sums meet in shared memory [wk][R][NC], in the place of A
        c32 *red = &S.A[0][0][0];
        static_assert(sizeof(S.A) >= 4 * 16 * NC * sizeof(c32), "the sums fit in A's stages");
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int q = 0; q < CQ; ++q)
                red[((wk * R) + 16 * wr + ry + 4 * x) * NC + 2 * tx + 16 * (q >> 1) + (q & 1)] =
                    c32{acc[x][q].x, acc[x][q].y * sgn[q]};
        __syncthreads();
        if (stage == 0) {
            c32 *Tout = a.T + a.toff[tb + d0];
            for (int e = tid; e < mc * ncol; e += 128) {
                const int m = e / ncol, n = e - m * ncol, g = col0 + n, p = g >= nrhs ? 1 : 0;
                c32 v = red[m * NC + n];
                for (int w = 1; w < WK; ++w) v = v + red[(w * R + m) * NC + n];
                Tout[((int64_t)p * M + m0 + m) * nrhs + g - p * nrhs] = v;
            }
        } else {
            // columns of both halves in this pass are summed first
            const int lo = min(ncol, max(0, nrhs - col0));  // half-0 columns of the pass
            const bool both = col0 == 0 && ncol == 2 * nrhs;
            const int no = both ? nrhs : ncol;
            for (int e = tid; e < mc * no; e += 128) {
                const int m = e / no, n = e - m * no;
                c32 v = {0.f, 0.f};
                for (int w = 0; w < WK; ++w) {
                    v = v + red[(w * R + m) * NC + n];
                    if (both) v = v + red[(w * R + m) * NC + n + nrhs];
                }
                const int c = n < lo ? col0 + n : col0 + n - nrhs;
                atomic_add_c(a.y + (int64_t)a.perm_r[bl[0] + m0 + m] * nrhs + c, v);
            }
        }
    }
}

template <class T>
__global__ void k_tensor_entries(TensorOut o, const int *blocks, int nb, int64_t nrows, int64_t ncols,
                                 int nq, const int *inv_r, const int *inv_c, const int *qmap,
                                 const int *rows, const int *cols, const int *fidx, int64_t count,
                                 cx<T> *out) {
    const cx<T> *fib = (const cx<T> *)o.fib;
    const cx<T> *pool = (const cx<T> *)o.face;
    const int Nu = o.Nu;
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < count;
         n += (int64_t)gridDim.x * blockDim.x) {
        if (rows[n] < 0 || rows[n] >= nrows || cols[n] < 0 || cols[n] >= ncols || fidx[n] < 0 || fidx[n] >= nq) {
            out[n] = cx<T>{(T)NAN, (T)NAN};  // invalid index: no access, NaN result
            continue;
        }
        const int pi = inv_r[rows[n]], pj = inv_c[cols[n]];
        const int mp = qmap[fidx[n]];
        const int u = mp > 0 ? mp - 1 : -mp - 1;
        cx<T> v = {0, 0};
        for (int b = 0; b < nb; ++b) {
            const int *bl = blocks + 5 * b;
            if (pi < bl[0] || pi >= bl[1] || pj < bl[2] || pj >= bl[3]) continue;
            const int nI = bl[1] - bl[0], nJ = bl[3] - bl[2];
            const int i = pi - bl[0], j = pj - bl[2];
            const int64_t tb = (int64_t)b * Nu;
            for (int d = 0; d < o.rank[b]; ++d) {
                const cx<T> *F = pool + o.foff[tb + d];
                cx<T> h = {0, 0};
                const int kd = o.frank[tb + d];
                if (kd < 0)
                    h = F[(int64_t)i * nJ + j];
                else
                    for (int t = 0; t < kd; ++t) cfma(h, F[(int64_t)t * nI + i], F[(int64_t)kd * nI + (int64_t)t * nJ + j]);
                cfma(v, h, fib[(tb + d) * Nu + u]);
            }
            break;
        }
        out[n] = mp > 0 ? v : cconj(v);
    }
}

}  // namespace

// One right-hand side, two or up to four per pass over the faces.
template <class T>
static int launch_one(cudaStream_t st, const ApplyArgs &a, const TensorOut &o) {
    for (int c = 0; c < a.nrhs;) {
        const int left = a.nrhs - c;
        if (left >= 3) k_apply_one<T, 4><<<a.nb, 128, 0, st>>>(a, o, c);
        else if (left == 2) k_apply_one<T, 2><<<a.nb, 128, 0, st>>>(a, o, c);
        else k_apply_one<T, 1><<<a.nb, 128, 0, st>>>(a, o, c);
        c += left >= 3 ? std::min(4, left) : left;
    }
    return (int)cudaGetLastError();
}

int td_launch_apply(cudaStream_t st, int prec, const ApplyArgs &a, const TensorOut &o, int num_sms) {
    if (a.nb == 0) return 0;
    if (a.single_f >= 0)
        return prec == TDBEM_FP64 ? launch_one<double>(st, a, o) : launch_one<float>(st, a, o);
    if (prec != TDBEM_FP64) return (int)cudaErrorInvalidValue;  // the mixed form runs on the tensor cores
    const int NQ = a.NQ;
    const size_t es = sizeof(c64);
    const int budget = 160 * 1024;
    // W tile: NQ x TJ x nrhs; z: RC x 2 x TJ x nrhs; acc: max(nI, 2*sumk) x nrhs
    int TJ = (int)std::max<int64_t>(1, std::min<int64_t>(32, (budget / 2) / ((int64_t)NQ * a.nrhs * es)));
    const int RC = 4;
    const int64_t acc_max = (int64_t)std::max(2 * RC * a.kcap, a.max_near_rows) * a.nrhs;
    auto smem = [&](int tj) {
        return ((int64_t)NQ * tj * a.nrhs + (int64_t)RC * 2 * tj * a.nrhs + acc_max + (int64_t)RC * NQ) * es +
               sizeof(int) * NQ;
    };
    size_t sm = smem(TJ);
    while (sm > (size_t)(200 * 1024) && TJ > 1) {
        TJ /= 2;
        sm = smem(TJ);
    }
    ApplyArgs aa = a;
    aa.acc_max = acc_max;
    if (sm > (size_t)(220 * 1024)) return (int)cudaErrorInvalidConfiguration;
    const int grid = std::min(a.nb, num_sms * 4);
    const cudaError_t e = cudaFuncSetAttribute(k_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return (int)e;
    k_apply<<<grid, 256, sm, st>>>(aa, o, TJ, RC);
    return (int)cudaGetLastError();
}

template <int CQ>
static int launch_faces(cudaStream_t st, const ApplyZArgs &a, const TensorOut &o, int stage, int col0) {
    const size_t sm = sizeof(FaceSmem<CQ>);
    cudaError_t e = cudaFuncSetAttribute(k_apply_faces<CQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return (int)e;
    const dim3 grid(stage == 0 ? a.nft : a.nb, stage == 0 ? 1 : kFY);
    k_apply_faces<CQ><<<grid, 128, sm, st>>>(a, o, stage, col0);
    return (int)cudaGetLastError();
}

int td_launch_apply_z(cudaStream_t st, const ApplyZArgs &a, const TensorOut &o, int num_sms) {
    // 16, 32 or 64 columns (half, right-hand side) per pass over the faces
    const int ncol = a.rpt * a.nrhs;
    int e = 0;
    for (int stage = 0; stage < 2 && !e; ++stage) {
        if ((stage == 0 ? a.nft : a.nb) == 0) continue;
        for (int c = 0; c < ncol && !e;) {
            const int left = ncol - c;
            e = left <= 16 ? launch_faces<2>(st, a, o, stage, c)
                : left <= 32 ? launch_faces<4>(st, a, o, stage, c) : launch_faces<8>(st, a, o, stage, c);
            c += left <= 16 ? 16 : left <= 32 ? 32 : 64;
        }
    }
    return e;
}

int td_launch_tensor_entries(cudaStream_t st, int prec, const TensorOut &o, const int *blocks,
                             int nb, int64_t nrows, int64_t ncols, int nq, const int *inv_r,
                             const int *inv_c, const int *qmap,
                             const int *rows, const int *cols, const int *fidx, int64_t count,
                             void *out) {
    if (count == 0) return 0;
    const int grid = (int)std::min<int64_t>((count + 127) / 128, 4096);
    if (prec == TDBEM_FP64)
        k_tensor_entries<double><<<grid, 128, 0, st>>>(o, blocks, nb, nrows, ncols, nq, inv_r, inv_c, qmap, rows, cols, fidx, count, (c64 *)out);
    else
        k_tensor_entries<float><<<grid, 128, 0, st>>>(o, blocks, nb, nrows, ncols, nq, inv_r, inv_c, qmap, rows, cols, fidx, count, (c32 *)out);
    return (int)cudaGetLastError();
}
