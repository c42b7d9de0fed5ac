// FP32 entries of the near field: regular pairs at several frequencies with the
// point geometry shared, and one entry of a near-field block at one frequency
// (regular pairs and touching pairs from the table).
#pragma once
#include "pair.cuh"

// Regular pair at FC frequencies with the geometry computed once per point
// pair (test triangle in registers, trial points streamed from the tables).
template <int OP, int FC>
TD_D void pair_multi(const TestF &X, const MeshDev &m, int tj, const float *sg, int nfc, c32 *acc, int loc) {
    // signed kernel normal: -n_y (DLP) or +n_x (ADLP), multiplied by d = y - x
    float nx = 0.f, ny = 0.f, nz = 0.f;
    if (OP == TD_DLP) {
        nx = -m.n32[tj];
        ny = -m.n32[m.nt + tj];
        nz = -m.n32[2 * m.nt + tj];
    } else if (OP == TD_ADLP) {
        nx = X.nx;
        ny = X.ny;
        nz = X.nz;
    }
#pragma unroll 1
    for (int b = 0; b < 7; ++b) {
        const int ob = b * m.nt + tj;
        const float yxh = m.qxh[ob], yyh = m.qyh[ob], yzh = m.qzh[ob];
        const float yxl = m.qxl[ob], yyl = m.qyl[ob], yzl = m.qzl[ob];
        const float wyb = m.qw32[ob] * (OP == TD_DLP ? bary7f(b, loc) : 1.0f);
#pragma unroll
        for (int a = 0; a < 7; ++a) {
            const float dx = (yxh - X.xh[a]) + (yxl - X.xl[a]);
            const float dy = (yyh - X.yh[a]) + (yyl - X.yl[a]);
            const float dz = (yzh - X.zh[a]) + (yzl - X.zl[a]);
            const float r2 = dx * dx + dy * dy + dz * dz;
            const float rinv = rsqrtf(r2);
            const float r = r2 * rinv;
            float w = X.w[a] * wyb * rinv;
            if (OP != TD_SLP) w *= (dx * nx + dy * ny + dz * nz) * rinv * rinv;
#pragma unroll
            for (int j = 0; j < FC; ++j) {
                if (j < nfc) {
                    const float sr = sg[2 * j], si = sg[2 * j + 1];
                    const c32 e = expm_sr(sr, si, r);
                    if (OP == TD_SLP) {
                        acc[j].x = fmaf(w, e.x, acc[j].x);
                        acc[j].y = fmaf(w, e.y, acc[j].y);
                    } else {
                        const float pr = fmaf(sr, r, 1.0f), pi = si * r;
                        acc[j].x = fmaf(w, pr * e.x - pi * e.y, acc[j].x);
                        acc[j].y = fmaf(w, pr * e.y + pi * e.x, acc[j].y);
                    }
                }
            }
        }
    }
}

// One entry A[row, col](s_k) of the mixed form (1/(4 pi) applied), summed as
// k_near_entries sums it: the regular pairs of the column's supports in FP32, the
// touching ones from the FP64 table [slot][nf][1 or 3].
template <int OP>
TD_D c32 near_entry(const MeshDev &m, int row, int col, float sr, float si, const c64 *table, int nf, int k) {
    constexpr int NV = TD_P1_TRIAL(OP) ? 3 : 1;
    const int p0 = TD_P1_TRIAL(OP) ? m.v2t_ptr[col] : 0, p1 = TD_P1_TRIAL(OP) ? m.v2t_ptr[col + 1] : 1;
    TestF X;
    load_test(m, row, X);
    const float sg[2] = {sr, si};
    c32 acc[1] = {{0.f, 0.f}};
    c64 sing = {0.0, 0.0};
    for (int p = p0; p < p1; ++p) {
        const int e = TD_P1_TRIAL(OP) ? m.v2t[p] : col, l = TD_P1_TRIAL(OP) ? m.v2t_loc[p] : 0;
        const int slot = touching_slot(m, row, e);
        if (slot >= 0) sing = sing + table[((int64_t)slot * nf + k) * NV + l];
        else pair_multi<OP, 1>(X, m, e, sg, 1, acc, l);
    }
    const float inv4pi = (float)(1.0 / TD_FOUR_PI);
    return c32{acc[0].x * inv4pi + (float)sing.x, acc[0].y * inv4pi + (float)sing.y};
}
