// Rank-predictor MLP: 6 features -> 64 -> 64 -> 16 rank bins, GELU hidden
// activations (x Phi(x), erf form), softmax cross-entropy, Adam.
//
// Parameter layout (FP32 master copy, same order for gradients):
//   W1[64][6] b1[64] W2[64][64] b2[64] W3[16][64] b3[16]
// Inference uses a BF16 copy of the weights with FP32 accumulation; training
// runs forward and backward in FP32 from the master copy.  Weights live in
// shared memory; inference takes one thread per sample, training tiles of 32
// samples per CTA.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "mlp.h"

namespace cg = cooperative_groups;

namespace {

constexpr int NIN = 6, NH = 64, NOUT = 16;
constexpr int OW1 = 0, OB1 = OW1 + NH * NIN, OW2 = OB1 + NH, OB2 = OW2 + NH * NH, OW3 = OB2 + NH,
              OB3 = OW3 + NOUT * NH, NP = OB3 + NOUT;
static_assert(NP == TD_MLP_NPARAMS, "parameter count");

TD_D float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__global__ void k_to_bf16(const float *p, __nv_bfloat16 *q, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) q[i] = __float2bfloat16(p[i]);
}

// Forward pass of one sample from weights in shared memory; returns the arg-max bin.
TD_D int mlp_forward_bin(const float *w, const float *in, float *logits) {
    float h1[NH], h2[NH];
    for (int o = 0; o < NH; ++o) {
        float a = w[OB1 + o];
#pragma unroll
        for (int i = 0; i < NIN; ++i) a = fmaf(w[OW1 + o * NIN + i], in[i], a);
        h1[o] = gelu(a);
    }
    for (int o = 0; o < NH; ++o) {
        float a = w[OB2 + o];
        for (int i = 0; i < NH; ++i) a = fmaf(w[OW2 + o * NH + i], h1[i], a);
        h2[o] = gelu(a);
    }
    int best = 0;
    float bv = -INFINITY;
    for (int o = 0; o < NOUT; ++o) {
        float a = w[OB3 + o];
        for (int i = 0; i < NH; ++i) a = fmaf(w[OW3 + o * NH + i], h2[i], a);
        if (logits) logits[o] = a;
        if (a > bv) {
            bv = a;
            best = o;
        }
    }
    return best;
}

// lower edges of the rank bins (the first ACA steps the compressor may run unchecked)
__constant__ int c_bin_lower[NOUT] = {1, 2, 3, 4, 5, 7, 9, 11, 13, 17, 21, 25, 33, 41, 49, 65};

// Presizing of the far blocks: sample s = (far block q, unique frequency u);
// the two frequency features are formed here from the block distance and
// s/c.  Writes the predicted first trip count kp to kpred[far[q] Nu + u],
// adds min(kp, kcap) to ks[q] (the block's predicted face ranks summed over
// the frequencies) and len[q] kp^2 to cost[q].
__global__ void __launch_bounds__(128) k_mlp_presize(const __nv_bfloat16 *P, const float *bfeat, const float *ffeat,
                                                     int nfar, int Nu, const int *far, const int *len, int kcap,
                                                     int *kpred, int *ks, float *cost) {
    __shared__ float w[NP];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) w[i] = __bfloat162float(P[i]);
    __syncthreads();
    const int64_t n = (int64_t)nfar * Nu;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        const int q = (int)(s / Nu), u = (int)(s - (s / Nu) * Nu);
        const float *b = bfeat + (int64_t)q * 5;
        float in[NIN] = {b[0], b[1], b[2], b[3], log1pf(fmaxf(0.f, ffeat[2 * u]) * b[4]),
                         log1pf(ffeat[2 * u + 1] * b[4])};
        const int kp = c_bin_lower[mlp_forward_bin(w, in, nullptr)];
        kpred[(int64_t)far[q] * Nu + u] = kp;
        atomicAdd(&ks[q], min(kp, kcap));
        atomicAdd(&cost[q], (float)len[q] * (float)kp * (float)kp);
    }
}

// Inference: bins[n] = argmax logits (BF16 weights, FP32 accumulation).
__global__ void __launch_bounds__(128) k_mlp_predict(const __nv_bfloat16 *P, const float *x, int64_t n,
                                                     int *bins, float *logits) {
    __shared__ float w[NP];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) w[i] = __bfloat162float(P[i]);
    __syncthreads();
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        float in[NIN], h1[NH], h2[NH];
#pragma unroll
        for (int i = 0; i < NIN; ++i) in[i] = x[s * NIN + i];
        for (int o = 0; o < NH; ++o) {
            float a = w[OB1 + o];
#pragma unroll
            for (int i = 0; i < NIN; ++i) a = fmaf(w[OW1 + o * NIN + i], in[i], a);
            h1[o] = gelu(a);
        }
        for (int o = 0; o < NH; ++o) {
            float a = w[OB2 + o];
            for (int i = 0; i < NH; ++i) a = fmaf(w[OW2 + o * NH + i], h1[i], a);
            h2[o] = gelu(a);
        }
        int best = 0;
        float bv = -INFINITY;
        for (int o = 0; o < NOUT; ++o) {
            float a = w[OB3 + o];
            for (int i = 0; i < NH; ++i) a = fmaf(w[OW3 + o * NH + i], h2[i], a);
            if (logits) logits[s * NOUT + o] = a;
            if (a > bv) {
                bv = a;
                best = o;
            }
        }
        if (bins) bins[s] = best;
    }
}

// Mean softmax cross-entropy and its gradient (FP32).  grad and loss must be
// zeroed by the caller; every CTA adds its sums once at the end.
//
// A CTA takes tiles of 32 samples through both passes with the weights and the
// tile's activations in shared memory ([feature][sample], rows of kGS).  The
// layers put one sample on each lane and eight outputs in registers: the weights
// are broadcasts, W2 kept in both orders so that the eight weights of a step
// are contiguous.  The weight gradients are outer products over the 32 samples,
// 4 x 4 outputs per thread (W2), kept in registers over the CTA's tiles.  One
// thread per sample with a warp sum per weight took 5648 x 5 shuffles a warp:
// 4096 samples 989 -> 21 us.  Clusters of 8 CTAs add their sums pairwise through
// distributed shared memory before the atomic adds: 128 partial sums added in any
// order had twice the rounding of the first form (relative gradient error 1.7e-7
// against 0.92e-7 at 4096 samples, 2.6e-7 against 3.3e-7 at 65536); so it is
// 0.73e-7 and 0.92e-7, for 30 us.  Bound at that size: latency, one tile per SM.
constexpr int kGT = 256, kGS = 36, kGC = 8;
struct GradSmem {
    float w2[NH * NH], w2t[NH * NH], w3[NOUT * NH], w3t[NH * NOUT], w1[NH * NIN], b1[NH], b2[NH], b3[NOUT];
    float in[NIN][kGS], h1[NH][kGS], g1[NH][kGS], h2[NH][kGS], g2[NH][kGS], d3[NOUT][kGS];
};

// GELU and its derivative
TD_D void gelu_both(float x, float &h, float &g) {
    const float c = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
    h = x * c;
    g = c + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// a[q] += sum_k x[k][lane] w[k ld + q], q < 8 (w 16-byte aligned)
template <int K>
TD_D void layer8(const float (*x)[kGS], const float *w, int ld, int lane, float *a) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float v = x[k][lane];
        const float4 p = *reinterpret_cast<const float4 *>(w + k * ld), q = *reinterpret_cast<const float4 *>(w + k * ld + 4);
        a[0] = fmaf(p.x, v, a[0]);
        a[1] = fmaf(p.y, v, a[1]);
        a[2] = fmaf(p.z, v, a[2]);
        a[3] = fmaf(p.w, v, a[3]);
        a[4] = fmaf(q.x, v, a[4]);
        a[5] = fmaf(q.y, v, a[5]);
        a[6] = fmaf(q.z, v, a[6]);
        a[7] = fmaf(q.w, v, a[7]);
    }
}
// sum over the 32 samples of two rows
TD_D float row_dot(const float *x, const float *y, float a) {
    float4 t = {0.0f, 0.0f, 0.0f, 0.0f};  // four chains: half the rounding of one
#pragma unroll
    for (int s = 0; s < 32; s += 4) {
        const float4 p = *reinterpret_cast<const float4 *>(x + s), q = *reinterpret_cast<const float4 *>(y + s);
        t = float4{fmaf(p.x, q.x, t.x), fmaf(p.y, q.y, t.y), fmaf(p.z, q.z, t.z), fmaf(p.w, q.w, t.w)};
    }
    return a + ((t.x + t.y) + (t.z + t.w));
}
TD_D float row_sum(const float *x, float a) {
#pragma unroll
    for (int s = 0; s < 32; s += 4) {
        const float4 p = *reinterpret_cast<const float4 *>(x + s);
        a += (p.x + p.y) + (p.z + p.w);
    }
    return a;
}

__global__ void __cluster_dims__(kGC) __launch_bounds__(kGT) k_mlp_grad(const float *P, const float *x, const int *label, int64_t n,
                                                  float *grad, float *loss) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem &S = *reinterpret_cast<GradSmem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, tx = tid & 15, ty = tid >> 4;
    for (int i = tid; i < NH * NH; i += kGT) {
        const float v = P[OW2 + i];
        S.w2[i] = v;
        S.w2t[(i % NH) * NH + i / NH] = v;
    }
    for (int i = tid; i < NOUT * NH; i += kGT) {
        const float v = P[OW3 + i];
        S.w3[i] = v;
        S.w3t[(i % NH) * NOUT + i / NH] = v;
    }
    for (int i = tid; i < NH * NIN; i += kGT) S.w1[i] = P[OW1 + i];
    for (int i = tid; i < NH; i += kGT) {
        S.b1[i] = P[OB1 + i];
        S.b2[i] = P[OB2 + i];
    }
    if (tid < NOUT) S.b3[tid] = P[OB3 + tid];
    float a2[4][4] = {}, a3[4] = {}, a1[2] = {}, ab = 0.0f, lsum = 0.0f;
    const float inv_n = 1.0f / (float)n;
    const int64_t tiles = (n + 31) / 32;
    const int o8 = wid * 8;  // this warp's eight outputs of a 64-wide layer
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t s0 = t * 32;
        const bool valid = s0 + lane < n;
        __syncthreads();  // weights loaded; the previous tile's sums are done
        if (tid < 32 * NIN) {
            const int i = tid % NIN, q = tid / NIN;
            S.in[i][q] = s0 + q < n ? x[s0 * NIN + tid] : 0.0f;
        }
        __syncthreads();
        // ---- forward
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float a = S.b1[o8 + q];
#pragma unroll
            for (int i = 0; i < NIN; ++i) a = fmaf(S.w1[(o8 + q) * NIN + i], S.in[i][lane], a);
            gelu_both(a, S.h1[o8 + q][lane], S.g1[o8 + q][lane]);
        }
        __syncthreads();
        {
            float a[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) a[q] = S.b2[o8 + q];
            layer8<NH>(S.h1, S.w2t + o8, NH, lane, a);
#pragma unroll
            for (int q = 0; q < 8; ++q) gelu_both(a[q], S.h2[o8 + q][lane], S.g2[o8 + q][lane]);
        }
        __syncthreads();
        {
            const int o = wid * 2;
            float a0 = S.b3[o], a1q = S.b3[o + 1];
#pragma unroll 8
            for (int i = 0; i < NH; ++i) {
                const float v = S.h2[i][lane];
                const float2 w = *reinterpret_cast<const float2 *>(&S.w3t[i * NOUT + o]);
                a0 = fmaf(w.x, v, a0);
                a1q = fmaf(w.y, v, a1q);
            }
            S.d3[o][lane] = a0;
            S.d3[o + 1][lane] = a1q;
        }
        __syncthreads();
        // ---- softmax cross-entropy: d loss / d logits = (softmax - onehot) / n
        {
            float lg[NOUT], mx = -INFINITY, se = 0.0f;
#pragma unroll
            for (int o = 0; o < NOUT; ++o) {
                lg[o] = S.d3[o][lane];
                mx = fmaxf(mx, lg[o]);
            }
#pragma unroll
            for (int o = 0; o < NOUT; ++o) se += expf(lg[o] - mx);
            const int lab = valid ? label[s0 + lane] : 0;
            const float l0 = S.d3[2 * wid][lane], l1 = S.d3[2 * wid + 1][lane];
            if (wid == 0 && valid) lsum += (logf(se) + mx - S.d3[lab][lane]) * inv_n;
            __syncthreads();
            S.d3[2 * wid][lane] = valid ? (expf(l0 - mx) / se - (2 * wid == lab ? 1.0f : 0.0f)) * inv_n : 0.0f;
            S.d3[2 * wid + 1][lane] = valid ? (expf(l1 - mx) / se - (2 * wid + 1 == lab ? 1.0f : 0.0f)) * inv_n : 0.0f;
        }
        __syncthreads();
        // ---- backward: g2 <- d2 = (W3^T d3) gelu'(z2), g1 <- d1 = (W2^T d2) gelu'(z1)
        {
            float a[8] = {};
            layer8<NOUT>(S.d3, S.w3 + o8, NH, lane, a);
#pragma unroll
            for (int q = 0; q < 8; ++q) S.g2[o8 + q][lane] *= a[q];
        }
        __syncthreads();
        {
            float a[8] = {};
            layer8<NH>(S.g2, S.w2 + o8, NH, lane, a);
#pragma unroll
            for (int q = 0; q < 8; ++q) S.g1[o8 + q][lane] *= a[q];
        }
        __syncthreads();
        // ---- gradients over the tile's samples
        float t2[4][4][2] = {};
#pragma unroll 2
        for (int q = 0; q < 32; q += 4) {
            float4 d[4], h[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                d[e] = *reinterpret_cast<const float4 *>(&S.g2[ty + 16 * e][q]);
                h[e] = *reinterpret_cast<const float4 *>(&S.h1[tx + 16 * e][q]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    t2[e][f][0] = fmaf(d[e].x, h[f].x, fmaf(d[e].y, h[f].y, t2[e][f][0]));
                    t2[e][f][1] = fmaf(d[e].z, h[f].z, fmaf(d[e].w, h[f].w, t2[e][f][1]));
                }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f) a2[e][f] += t2[e][f][0] + t2[e][f][1];
#pragma unroll
        for (int f = 0; f < 4; ++f) a3[f] = row_dot(S.d3[ty], S.h2[tx + 16 * f], a3[f]);
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const int e = tid + kGT * f;
            if (e < NH * NIN) a1[f] = row_dot(S.g1[e / NIN], S.in[e % NIN], a1[f]);
        }
        if (tid < NH) ab = row_sum(S.g1[tid], ab);
        else if (tid < 2 * NH) ab = row_sum(S.g2[tid - NH], ab);
        else if (tid < 2 * NH + NOUT) ab = row_sum(S.d3[tid - 2 * NH], ab);
    }
    // the cluster's sums meet in shared memory, then one atomic add per parameter
    __syncthreads();  // the last tile's sums are done
    float *R = reinterpret_cast<float *>(smem_raw);  // [NP] gradient, then the loss
#pragma unroll
    for (int e = 0; e < 4; ++e) {
#pragma unroll
        for (int f = 0; f < 4; ++f) R[OW2 + (ty + 16 * e) * NH + tx + 16 * f] = a2[e][f];
        R[OW3 + ty * NH + tx + 16 * e] = a3[e];
    }
#pragma unroll
    for (int f = 0; f < 2; ++f)
        if (tid + kGT * f < NH * NIN) R[OW1 + tid + kGT * f] = a1[f];
    if (tid < NH) R[OB1 + tid] = ab;
    else if (tid < 2 * NH) R[OB2 + tid - NH] = ab;
    else if (tid < 2 * NH + NOUT) R[OB3 + tid - 2 * NH] = ab;
    if (wid == 0) {
        lsum = warp_sum(lsum);
        if (lane == 0) R[NP] = lsum;
    }
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    // each CTA takes its share of the parameters (and the loss), four per thread
    constexpr int per = (NP + 1 + 4 * kGC - 1) / (4 * kGC) * 4;
    static_assert(sizeof(GradSmem) >= sizeof(float) * per * kGC && per <= 4 * kGT, "shares of the sums");
    if (4 * tid < per) {
        const int i = (int)cl.block_rank() * per + 4 * tid;
        float4 v[kGC];
#pragma unroll
        for (int q = 0; q < kGC; ++q) v[q] = *reinterpret_cast<const float4 *>(cl.map_shared_rank(R, q) + i);
#pragma unroll
        for (int s = kGC / 2; s > 0; s >>= 1)
#pragma unroll
            for (int q = 0; q < s; ++q)
                v[q] = float4{v[q].x + v[q + s].x, v[q].y + v[q + s].y, v[q].z + v[q + s].z, v[q].w + v[q + s].w};
        const float o[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (i + e <= NP) atomicAdd(i + e < NP ? grad + i + e : loss, o[e]);
    }
    cl.sync();  // (the others' reads of this CTA's shared memory)
}

// Adam: m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// p -= lr (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps).
__global__ void k_adam(float *P, const float *G, float *m, float *v, int n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = G[i];
    const float mi = b1 * m[i] + (1.0f - b1) * g;
    const float vi = b2 * v[i] + (1.0f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Seeded initialisation (counter-based hash -> uniform in [-a, a] with a =
// sqrt(6 / fan_in) per layer, biases zero).
TD_D uint32_t mix32(uint64_t z) {
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return (uint32_t)((z ^ (z >> 31)) >> 32);
}
__global__ void k_mlp_init(float *P, uint64_t seed) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NP) return;
    float fan = 0.0f;
    if (i < OB1) fan = NIN;
    else if (i >= OW2 && i < OB2) fan = NH;
    else if (i >= OW3 && i < OB3) fan = NH;
    if (fan == 0.0f) {
        P[i] = 0.0f;
        return;
    }
    const float u = (mix32(seed * 1000003ull + (uint64_t)i) + 0.5f) * (1.0f / 4294967296.0f);
    P[i] = (2.0f * u - 1.0f) * sqrtf(6.0f / fan);
}

}  // namespace

int td_mlp_init(cudaStream_t st, float *P, uint64_t seed) {
    k_mlp_init<<<(NP + 255) / 256, 256, 0, st>>>(P, seed);
    return (int)cudaGetLastError();
}

int td_mlp_to_bf16(cudaStream_t st, const float *P, void *Pb) {
    k_to_bf16<<<(NP + 255) / 256, 256, 0, st>>>(P, (__nv_bfloat16 *)Pb, NP);
    return (int)cudaGetLastError();
}

int td_mlp_predict(cudaStream_t st, const void *Pb, const float *x, int64_t n, int *bins, float *logits,
                   int num_sms) {
    if (n <= 0) return 0;
    const int grid = (int)std::min<int64_t>((n + 127) / 128, (int64_t)num_sms * 8);
    k_mlp_predict<<<grid, 128, 0, st>>>((const __nv_bfloat16 *)Pb, x, n, bins, logits);
    return (int)cudaGetLastError();
}

int td_mlp_presize(cudaStream_t st, const void *Pb, const float *bfeat, const float *ffeat, int nfar, int Nu,
                   const int *far, const int *len, int kcap, int *kpred, int *ks, float *cost, int num_sms) {
    if (nfar <= 0) return 0;
    const int64_t n = (int64_t)nfar * Nu;
    const int grid = (int)std::min<int64_t>((n + 127) / 128, (int64_t)num_sms * 8);
    k_mlp_presize<<<grid, 128, 0, st>>>((const __nv_bfloat16 *)Pb, bfeat, ffeat, nfar, Nu, far, len, kcap, kpred, ks,
                                        cost);
    return (int)cudaGetLastError();
}

int td_mlp_grad(cudaStream_t st, const float *P, const float *x, const int *label, int64_t n, float *grad,
                float *loss, int num_sms) {
    cudaMemsetAsync(grad, 0, sizeof(float) * NP, st);
    cudaMemsetAsync(loss, 0, sizeof(float), st);
    if (n <= 0) return (int)cudaGetLastError();
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem));
    if (e != cudaSuccess) return (int)e;
    const int64_t tiles = std::min<int64_t>((n + 31) / 32, (int64_t)num_sms * 2);
    const int grid = (int)((tiles + kGC - 1) / kGC * kGC);  // (whole clusters; CTAs without a tile add zeros)
    k_mlp_grad<<<grid, kGT, sizeof(GradSmem), st>>>(P, x, label, n, grad, loss);
    return (int)cudaGetLastError();
}

int td_mlp_adam(cudaStream_t st, float *P, const float *G, float *m, float *v, float lr, float b1, float b2,
                float eps, int t) {
    const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
    k_adam<<<(NP + 255) / 256, 256, 0, st>>>(P, G, m, v, NP, lr, b1, b2, eps, c1, c2);
    return (int)cudaGetLastError();
}
