// Galerkin pair integrals of the Laplace-domain layer operators on flat
// triangles (Sec. 2 eqs. slp/dlp, Sec. 3 "Spatial discretisation").
//
//   SLP:  int_x int_y exp(-s r/c) / (4 pi r)                      (P0 x P0)
//   DLP:  int_x int_y phi_m(y) exp(-s r/c)(1 + s r/c)(x-y).n_y / (4 pi r^3)
//         for the three P1 hats phi_m of the trial triangle         (P0 x P1)
//   ADLP: int_x int_y exp(-s r/c)(1 + s r/c)(y-x).n_x / (4 pi r^3)
//         (K', eq. adlp: the conormal derivative at x)              (P0 x P0)
//
// Regular pairs: 7-point degree-5 rule in x and in y.  FP32 form: the
// quadrature-point coordinates are split into hi + lo floats so that the
// difference y - x keeps FP32 relative accuracy for close pairs.
// Touching pairs (identical, common edge, common vertex): Sauter-Schwab
// regularising transforms in FP64 with ng Gauss-Legendre points per variable:
//   identical: z = yh - xh in six sectors, z = xi (e_a + eta (e_b - e_a)),
//              weight xi (1 - xi)^2 / 2 (P0 x P0: kernel depends on z only);
//   edge:      (u, p, q) = (yh1 - xh1, xh2, yh2) on six cone triangles,
//              weight xi^2 e1 |det| (1 - xi), trial point at mid t-range;
//   vertex:    larger of xh1, yh1 is xi, weight xi^3 e1, two regions.
// The parametrisation of a triangle (P0, P1, P2) is
// chi(xh) = P0 + xh1 (P1 - P0) + xh2 (P2 - P1) on {0 <= xh2 <= xh1 <= 1}.
#pragma once
#include "common.cuh"

#define TD_FOUR_PI 12.566370614359172953850573533118
#define TD_INV_FOUR_PI_F 0.079577471545947667884f

enum { TD_SLP = 0, TD_DLP = 1, TD_ADLP = 2 };
// The double layer's trial space is P1 (a column is a vertex and its
// triangles); the single layer and the adjoint double layer have P0 columns.
#define TD_P1_TRIAL(OP) ((OP) == TD_DLP)

struct MeshDev {
    int nt, nv;
    // FP32 7-point tables, layout [7][nt]: hi/lo coordinates, weight*area
    const float *qxh, *qyh, *qzh, *qxl, *qyl, *qzl, *qw32;
    const float *n32;  // [3][nt] unit normals
    // the same FP32 tables packed for 16-byte loads: qp[2 (p nt + e)] =
    // (x_hi, y_hi, z_hi, weight*area), qp[2 (p nt + e) + 1] = (x_lo, y_lo,
    // z_lo, 0); nrm4[e] = (n_x, n_y, n_z, 0)
    const float4 *qp, *nrm4;
    // FP64 7-point tables [7][nt] and normals [3][nt]
    const double *qx, *qy, *qz, *qw, *n64;
    const double *verts;  // [nv][3]
    const int *tris;      // [nt][3]
    const double *area;   // [nt]
    const int *v2t_ptr, *v2t;      // P1 supports: triangles around a vertex
    const signed char *v2t_loc;    // local index of the vertex in that triangle
    const int *tp_ptr, *tp_tri, *tp_slot;  // touching triangles per triangle (sorted)
    int ng;
    const double *gx, *gw;  // Gauss-Legendre on [0,1]
};

// Barycentric coordinates of the 7 rule points: the centroid, the orbit
// (a, a, 1-2a) and the orbit (b, b, 1-2b), a, b = (6 -/+ sqrt 15)/21, in the
// order (a,a,1-2a), (a,1-2a,a), (1-2a,a,a), then the same for b.
#define TD_R7A 0.10128650732345633880098736191512
#define TD_R7A1 0.79742698535308732239802527616975
#define TD_R7B 0.47014206410511508977044120951345
#define TD_R7B1 0.05971587178976982045911758097311
TD_HD double bary7d(int b, int k) {
    if (b == 0) return 1.0 / 3.0;
    const int odd = 2 - (b - 1) % 3;
    const bool orb_a = b <= 3;
    return k == odd ? (orb_a ? TD_R7A1 : TD_R7B1) : (orb_a ? TD_R7A : TD_R7B);
}
TD_HD float bary7f(int b, int k) {
    if (b == 0) return 1.0f / 3.0f;
    const int odd = 2 - (b - 1) % 3;
    const bool orb_a = b <= 3;
    return k == odd ? (orb_a ? (float)TD_R7A1 : (float)TD_R7B1) : (orb_a ? (float)TD_R7A : (float)TD_R7B);
}

// ---------------------------------------------------------------------------
// Regular pairs.  The test triangle's 7 points are held in registers (the
// loop over them is fully unrolled); the trial triangle's points are read
// one at a time from the [7][nt] tables (coalesced when threads take
// different trial triangles, broadcast when they share one).
// ---------------------------------------------------------------------------
struct TestF {
    float xh[7], yh[7], zh[7], xl[7], yl[7], zl[7], w[7];
    float nx, ny, nz;  // unit normal of the test triangle (adjoint double layer)
};

TD_D void load_test(const MeshDev &m, int t, TestF &T) {
#pragma unroll
    for (int q = 0; q < 7; ++q) {
        const int o = q * m.nt + t;
        T.xh[q] = m.qxh[o];
        T.yh[q] = m.qyh[o];
        T.zh[q] = m.qzh[o];
        T.xl[q] = m.qxl[o];
        T.yl[q] = m.qyl[o];
        T.zl[q] = m.qzl[o];
        T.w[q] = m.qw32[o];
    }
    T.nx = m.n32[t];
    T.ny = m.n32[m.nt + t];
    T.nz = m.n32[2 * m.nt + t];
}

// e^{-sigma r} = e^{-sr r} (cos(si r) - i sin(si r)) for sigma = (sr, si), FP32
// on the special-function unit:
//   exponent: e^{-x} = 2^{t}, t = -x log2(e) formed as a rounded product plus
//     its FMA-recovered rounding error and the low part of log2(e), then
//     2^{t_hi} (1 + t_lo ln 2);
//   phase: Cody-Waite additive reduction y - k 2pi with k the nearest integer
//     to y / 2pi (formed by adding and subtracting 1.5 * 2^23, which rounds
//     to an integer in round-to-nearest for |y / 2pi| < 2^22, on the FMA pipe
//     instead of a separate rounding instruction) and 2pi split into a float
//     head and tail (two FMAs), then the SFU sin/cos, whose absolute error is
//     below 4e-7 on [-pi, pi].
// The power of two is the SFU's ex2 with subnormal results flushed to zero
// (values below 1.2e-38, far below the entries' resolution).
#define TD_L2E_HI 1.44269502162933349609375f
#define TD_L2E_LO 1.92596298909109e-08f
#define TD_LN2_F 0.693147180559945309417f
#define TD_2PI_HI 6.28318548202514648438f
#define TD_2PI_LO (-1.7484556025237907e-07f)
#define TD_INV_2PI_F 0.159154943091895335769f
TD_D float ex2_ftz(float t) {
    float v;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(v) : "f"(t));
    return v;
}
TD_D c32 expm_sr(float sr, float si, float r) {
    const float x = sr * r;
    const float th = -x * TD_L2E_HI;
    const float tl = fmaf(-x, TD_L2E_HI, -th) - x * TD_L2E_LO;
    const float ea = ex2_ftz(th) * fmaf(tl, TD_LN2_F, 1.0f);
    const float y = si * r;
    const float k = __fsub_rn(__fadd_rn(y * TD_INV_2PI_F, 12582912.0f), 12582912.0f);
    float yr = fmaf(-k, TD_2PI_HI, y);
    yr = fmaf(-k, TD_2PI_LO, yr);
    float sn, cs;
    __sincosf(yr, &sn, &cs);
    return {ea * cs, -ea * sn};
}

struct TestD {
    double x[7], y[7], z[7], w[7];
    double nx, ny, nz;  // unit normal of the test triangle (adjoint double layer)
};

TD_D void load_test(const MeshDev &m, int t, TestD &T) {
#pragma unroll
    for (int q = 0; q < 7; ++q) {
        const int o = q * m.nt + t;
        T.x[q] = m.qx[o];
        T.y[q] = m.qy[o];
        T.z[q] = m.qz[o];
        T.w[q] = m.qw[o];
    }
    T.nx = m.n64[t];
    T.ny = m.n64[m.nt + t];
    T.nz = m.n64[2 * m.nt + t];
}

// Tables of expm_sr (FP64): 2^{j/64} rounded to nearest with its relative rounding
// error, and cos, sin of 2 pi j / 64 with their rounding errors (from 300-bit
// values).
static __device__ const double2 c_exp2_64[64] = {
    {1.0, 0.0},
    {1.0108892860517005, -1.507066976926039e-17},
    {1.0218971486541166, 4.9997448722726326e-17},
    {1.0330248790212284, 7.357846871247418e-18},
    {1.0442737824274138, 8.189317638195514e-17},
    {1.0556451783605572, 1.6665881442326747e-18},
    {1.0671404006768237, -7.402825309426177e-17},
    {1.0787607977571199, -6.170654745608695e-17},
    {1.0905077326652577, -2.7939114859515733e-17},
    {1.102382583307841, 4.776959425256223e-17},
    {1.1143867425958924, 9.341710609905044e-17},
    {1.1265216186082418, 4.5856703266623505e-17},
    {1.1387886347566916, 7.826573258636075e-17},
    {1.1511892299529827, 2.823784425951061e-17},
    {1.1637248587775775, 3.2904726646008416e-17},
    {1.1763969916502812, 4.7213681211701275e-17},
    {1.189207115002721, 3.3484623336251524e-17},
    {1.202156731452703, 5.527550048505249e-17},
    {1.215247359980469, -6.346552106729484e-17},
    {1.22848053610687, -1.5456342819397733e-17},
    {1.241857812073484, 3.7508542013031266e-17},
    {1.255380757024691, -5.346099009198751e-18},
    {1.2690509571917332, 2.1023049675215714e-18},
    {1.2828700160787783, 1.3357510088834541e-17},
    {1.2968395546510096, 1.9572585293112036e-17},
    {1.3109612115247644, -5.4780691239267786e-17},
    {1.3252366431597413, -2.1571477251208756e-17},
    {1.339667524053303, 6.663804589232194e-17},
    {1.3542555469368927, 5.68648095791174e-17},
    {1.3690024229745905, 7.007875046906994e-17},
    {1.383909881963832, -4.8923067513522756e-17},
    {1.3989796725383112, -6.872303720902018e-17},
    {1.4142135623730951, -6.835808657661923e-17},
    {1.42961333839197, -8.416011634717156e-18},
    {1.4451808069770467, -2.092304381843353e-17},
    {1.460917794180647, -3.833464968654295e-17},
    {1.4768261459394993, -2.3591094770850053e-17},
    {1.4929077282912648, 9.50689710108796e-18},
    {1.5091644275934228, -6.735219232374683e-17},
    {1.5255981507445384, -7.226635472101257e-17},
    {1.5422108254079407, 5.1548301170786783e-17},
    {1.559004400237837, 2.4253985766689806e-17},
    {1.5759808451078865, -6.432131775424189e-18},
    {1.593142151342267, -6.336161863401293e-17},
    {1.6104903319492543, 1.5341410053603723e-17},
    {1.6280274218573478, -4.123367330661149e-17},
    {1.645755478153965, -6.152602891550265e-17},
    {1.6636765803267364, 3.540948262646183e-17},
    {1.681792830507429, 4.875160526227061e-17},
    {1.7001063537185235, -4.719539664590972e-18},
    {1.718619298122478, -1.0772487078934056e-17},
    {1.7373338352737062, 1.821405440362259e-17},
    {1.7562521603732995, 1.685487290628973e-17},
    {1.7753764925265212, 3.621615935336894e-17},
    {1.7947090750031072, 1.01562190116415e-17},
    {1.8142521755003989, -5.495118966122005e-17},
    {1.8340080864093424, 1.790126907604513e-17},
    {1.8539791250833855, 5.265370768556274e-17},
    {1.8741676341103, -3.266924100901318e-17},
    {1.8945759815869656, 1.7963932659833022e-17},
    {1.9152065613971474, -5.5450656186394274e-17},
    {1.9360617934922943, 5.336805878514151e-17},
    {1.9571441241754002, 4.578491527706009e-17},
    {1.978456026387951, 2.04142788975783e-17},
};
struct alignas(16) Cis64 { double x, y, z, w; };
static __device__ const Cis64 c_cis_64[64] = {  // cos, sin, errors
    {1.0, 0.0, 0.0, 0.0},
    {0.9951847266721969, 0.0980171403295606, -4.248691367830441e-17, -1.634582362244256e-18},
    {0.9807852804032304, 0.19509032201612828, 1.8546939997825006e-17, -7.991079068461731e-18},
    {0.9569403357322088, 0.2902846772544624, 4.05538698618757e-17, -1.892797870777425e-17},
    {0.9238795325112867, 0.3826834323650898, 1.7645047084336677e-17, -1.0050772696461588e-17},
    {0.881921264348355, 0.47139673682599764, -1.9843248405890562e-17, 6.516678136069013e-18},
    {0.8314696123025452, 0.5555702330196022, 1.4073856984728024e-18, 4.709410940561677e-17},
    {0.773010453362737, 0.6343932841636455, -3.256590703364977e-17, 1.0420901929280035e-17},
    {0.7071067811865476, 0.7071067811865476, -4.833646656726457e-17, -4.833646656726457e-17},
    {0.6343932841636455, 0.773010453362737, 1.0420901929280035e-17, -3.256590703364977e-17},
    {0.5555702330196022, 0.8314696123025452, 4.709410940561677e-17, 1.4073856984728024e-18},
    {0.47139673682599764, 0.881921264348355, 6.516678136069013e-18, -1.9843248405890562e-17},
    {0.3826834323650898, 0.9238795325112867, -1.0050772696461588e-17, 1.7645047084336677e-17},
    {0.2902846772544624, 0.9569403357322088, -1.892797870777425e-17, 4.05538698618757e-17},
    {0.19509032201612828, 0.9807852804032304, -7.991079068461731e-18, 1.8546939997825006e-17},
    {0.0980171403295606, 0.9951847266721969, -1.634582362244256e-18, -4.248691367830441e-17},
    {0.0, 1.0, 0.0, 0.0},
    {-0.0980171403295606, 0.9951847266721969, 1.634582362244256e-18, -4.248691367830441e-17},
    {-0.19509032201612828, 0.9807852804032304, 7.991079068461731e-18, 1.8546939997825006e-17},
    {-0.2902846772544624, 0.9569403357322088, 1.892797870777425e-17, 4.05538698618757e-17},
    {-0.3826834323650898, 0.9238795325112867, 1.0050772696461588e-17, 1.7645047084336677e-17},
    {-0.47139673682599764, 0.881921264348355, -6.516678136069013e-18, -1.9843248405890562e-17},
    {-0.5555702330196022, 0.8314696123025452, -4.709410940561677e-17, 1.4073856984728024e-18},
    {-0.6343932841636455, 0.773010453362737, -1.0420901929280035e-17, -3.256590703364977e-17},
    {-0.7071067811865476, 0.7071067811865476, 4.833646656726457e-17, -4.833646656726457e-17},
    {-0.773010453362737, 0.6343932841636455, 3.256590703364977e-17, 1.0420901929280035e-17},
    {-0.8314696123025452, 0.5555702330196022, -1.4073856984728024e-18, 4.709410940561677e-17},
    {-0.881921264348355, 0.47139673682599764, 1.9843248405890562e-17, 6.516678136069013e-18},
    {-0.9238795325112867, 0.3826834323650898, -1.7645047084336677e-17, -1.0050772696461588e-17},
    {-0.9569403357322088, 0.2902846772544624, -4.05538698618757e-17, -1.892797870777425e-17},
    {-0.9807852804032304, 0.19509032201612828, -1.8546939997825006e-17, -7.991079068461731e-18},
    {-0.9951847266721969, 0.0980171403295606, 4.248691367830441e-17, -1.634582362244256e-18},
    {-1.0, 0.0, 0.0, 0.0},
    {-0.9951847266721969, -0.0980171403295606, 4.248691367830441e-17, 1.634582362244256e-18},
    {-0.9807852804032304, -0.19509032201612828, -1.8546939997825006e-17, 7.991079068461731e-18},
    {-0.9569403357322088, -0.2902846772544624, -4.05538698618757e-17, 1.892797870777425e-17},
    {-0.9238795325112867, -0.3826834323650898, -1.7645047084336677e-17, 1.0050772696461588e-17},
    {-0.881921264348355, -0.47139673682599764, 1.9843248405890562e-17, -6.516678136069013e-18},
    {-0.8314696123025452, -0.5555702330196022, -1.4073856984728024e-18, -4.709410940561677e-17},
    {-0.773010453362737, -0.6343932841636455, 3.256590703364977e-17, -1.0420901929280035e-17},
    {-0.7071067811865476, -0.7071067811865476, 4.833646656726457e-17, 4.833646656726457e-17},
    {-0.6343932841636455, -0.773010453362737, -1.0420901929280035e-17, 3.256590703364977e-17},
    {-0.5555702330196022, -0.8314696123025452, -4.709410940561677e-17, -1.4073856984728024e-18},
    {-0.47139673682599764, -0.881921264348355, -6.516678136069013e-18, 1.9843248405890562e-17},
    {-0.3826834323650898, -0.9238795325112867, 1.0050772696461588e-17, -1.7645047084336677e-17},
    {-0.2902846772544624, -0.9569403357322088, 1.892797870777425e-17, -4.05538698618757e-17},
    {-0.19509032201612828, -0.9807852804032304, 7.991079068461731e-18, -1.8546939997825006e-17},
    {-0.0980171403295606, -0.9951847266721969, 1.634582362244256e-18, 4.248691367830441e-17},
    {0.0, -1.0, 0.0, 0.0},
    {0.0980171403295606, -0.9951847266721969, -1.634582362244256e-18, 4.248691367830441e-17},
    {0.19509032201612828, -0.9807852804032304, -7.991079068461731e-18, -1.8546939997825006e-17},
    {0.2902846772544624, -0.9569403357322088, -1.892797870777425e-17, -4.05538698618757e-17},
    {0.3826834323650898, -0.9238795325112867, -1.0050772696461588e-17, -1.7645047084336677e-17},
    {0.47139673682599764, -0.881921264348355, 6.516678136069013e-18, 1.9843248405890562e-17},
    {0.5555702330196022, -0.8314696123025452, 4.709410940561677e-17, -1.4073856984728024e-18},
    {0.6343932841636455, -0.773010453362737, 1.0420901929280035e-17, 3.256590703364977e-17},
    {0.7071067811865476, -0.7071067811865476, -4.833646656726457e-17, 4.833646656726457e-17},
    {0.773010453362737, -0.6343932841636455, -3.256590703364977e-17, -1.0420901929280035e-17},
    {0.8314696123025452, -0.5555702330196022, 1.4073856984728024e-18, -4.709410940561677e-17},
    {0.881921264348355, -0.47139673682599764, -1.9843248405890562e-17, -6.516678136069013e-18},
    {0.9238795325112867, -0.3826834323650898, 1.7645047084336677e-17, 1.0050772696461588e-17},
    {0.9569403357322088, -0.2902846772544624, 4.05538698618757e-17, 1.892797870777425e-17},
    {0.9807852804032304, -0.19509032201612828, 1.8546939997825006e-17, 7.991079068461731e-18},
    {0.9951847266721969, -0.0980171403295606, -4.248691367830441e-17, 1.634582362244256e-18},
};
// e^{-(x + i y)} = ea (c - i s) in FP64 by table lookup (P. T. P. Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point arithmetic",
// 1989, and the same idea for sine and cosine):
//   e^{-x} = 2^{k/64} e^{t}, |t| <= ln 2 / 128, k split into 2^{k >> 6} and a table value;
//   cos y, sin y from the nearest of 64 angles and |t| <= pi / 64;
// reductions by Cody-Waite splits whose products with k are exact, Taylor
// polynomials to below 2^-57.  The FP64 pipe (1/74 of the FP32 rate) bounds every
// FP64 kernel: 36 of its operations here, fewer than exp and sincos need for their
// whole ranges.  Error of the complex value 2.5e-16 max, 7.7e-17 rms (exp and sincos:
// 2.8e-16, 8.1e-17), over x < 690, |y| < 60000.  With sqrt_inv below: FP64
// compression of the 1280-triangle sphere 172 -> 152 ms, 320 x 320 x 16 FP64 entries
// 11.9 -> 10.5 ms.  Outside |x| < 704, |y| < 65536 (and for NaN) the library functions
// answer.
struct ExpParts {
    double ea, c, s;
};
static __device__ __noinline__ ExpParts exp_parts_any(double x, double y) {
    ExpParts e;
    e.ea = exp(-x);
    sincos(y, &e.s, &e.c);
    return e;
}
TD_D ExpParts exp_parts(double x, double y) {
    // range checks on the high words: integer instructions (0x40860000: 704, 0x40f00000: 65536)
    if ((__double2hiint(x) & 0x7fffffff) >= 0x40860000 || (__double2hiint(y) & 0x7fffffff) >= 0x40f00000)
        return exp_parts_any(x, y);
    const double magic = 6755399441055744.0;  // 1.5 * 2^52: adding it rounds to an integer
    // exponential of -x
    const double kx = fma(-x, 92.33248261689366, magic);
    const int ix = __double2loint(kx);
    const double fx = kx - magic;
    double t = fma(-fx, 0.010830424695996044, -x);
    t = fma(-fx, 2.5310172166650877e-13, t);
    double p = fma(t, 1.0 / 720.0, 1.0 / 120.0);
    p = fma(t, p, 1.0 / 24.0);
    p = fma(t, p, 1.0 / 6.0);
    p = fma(t, p, 0.5);
    const double2 te = c_exp2_64[ix & 63];
    p = fma(t * t, p, t) + te.y;  // e^t - 1, and the table value's rounding
    const double eb = __hiloint2double(__double2hiint(te.x) + ((ix >> 6) << 20), __double2loint(te.x));
    // angle y
    const double ky = fma(y, 10.185916357881302, magic);
    const int iy = __double2loint(ky);
    const double fy = ky - magic;
    double u = fma(-fy, 0.09817477042088285, y);
    u = fma(-fy, 3.798187816439979e-12, u);
    u = fma(-fy, 1.2639164054974691e-22, u);
    const double v = u * u;
    double s = fma(v, -1.0 / 5040.0, 1.0 / 120.0);
    s = fma(v, s, -1.0 / 6.0);
    s = fma(u * v, s, u);  // sin u
    double c = fma(v, 1.0 / 40320.0, -1.0 / 720.0);
    c = fma(v, c, 1.0 / 24.0);
    c = fma(v, c, -0.5) * v;  // cos u - 1
    const Cis64 w = c_cis_64[iy & 63];
    return {fma(eb, p, eb), w.x + fma(w.x, c, fma(-w.y, s, w.z)), w.y + fma(w.y, c, fma(w.x, s, w.w))};
}
TD_D c64 expm_sr(double sr, double si, double r) {
    const ExpParts e = exp_parts(sr * r, si * r);
    return {e.ea * e.c, -e.ea * e.s};
}
// sqrt(r2) and its reciprocal from one reciprocal square root, each corrected to
// the error of sqrt and 1 / sqrt (1.1e-16 and 1.7e-16 max, measured), without the
// FP64 operations of a second iterative function.
static __device__ __noinline__ double2 sqrt_inv_any(double r2) {
    const double r = sqrt(r2);
    return {r, 1.0 / r};
}
TD_D double sqrt_inv(double r2, double &ri) {
    if ((unsigned)(__double2hiint(r2) - 0x00100000) >= 0x7fe00000u) {  // 0, subnormal, infinite, NaN
        const double2 v = sqrt_inv_any(r2);
        ri = v.y;
        return v.x;
    }
    const double s = rsqrt(r2), g = r2 * s;
    const double r = fma(fma(-g, g, r2), 0.5 * s, g);
    ri = fma(fma(-r, s, 1.0), s, s);
    return r;
}

// Test triangle in registers, by precision.
template <class T> struct Reg;
template <> struct Reg<float> { using Test = TestF; };
template <> struct Reg<double> { using Test = TestD; };

// ---------------------------------------------------------------------------
// Touching pairs: classification and Sauter-Schwab quadrature points (FP64)
// ---------------------------------------------------------------------------
struct SingGeom {
    int cls;           // 3 identical, 2 edge, 1 vertex, 0 none
    double P[3][3];    // test parametrisation vertices
    double Q[3][3];    // trial parametrisation vertices
    int loc[3];        // mesh-local index of trial parametrisation vertex k
    double g;          // Jacobian factor (2|ti|)(2|tj|)
    double ny[3];      // trial unit normal
    double nx[3];      // test unit normal
};

// Shared vertices of ti and tj decide the class; the parametrisations follow
// the order described at the top of this file:
//   identical: both in mesh order; edge: shared vertices in increasing local
//   index of ti, then the remaining vertex; vertex: the shared vertex then the
//   next two in each triangle's own cyclic order.
TD_D int classify_pair(const MeshDev &m, int ti, int tj, SingGeom &G) {
    const int *A = m.tris + 3 * ti, *B = m.tris + 3 * tj;
    int a[3] = {A[0], A[1], A[2]}, b[3] = {B[0], B[1], B[2]};
    int ia[3], ib[3], ns = 0;
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int y = 0; y < 3; ++y)
            if (a[x] == b[y]) {
                ia[ns] = x;
                ib[ns] = y;
                ns++;
            }
    G.cls = ns;
    if (ns == 0) return 0;
    int la[3], lb[3];
    if (ns == 3) {
        for (int k = 0; k < 3; ++k) la[k] = lb[k] = k;
    } else if (ns == 2) {
        la[0] = ia[0];
        la[1] = ia[1];
        la[2] = 3 - ia[0] - ia[1];
        lb[0] = ib[0];
        lb[1] = ib[1];
        lb[2] = 3 - ib[0] - ib[1];
    } else {
        for (int k = 0; k < 3; ++k) {
            la[k] = (ia[0] + k) % 3;
            lb[k] = (ib[0] + k) % 3;
        }
    }
    for (int k = 0; k < 3; ++k) {
        G.loc[k] = lb[k];
        for (int c = 0; c < 3; ++c) {
            G.P[k][c] = m.verts[3 * a[la[k]] + c];
            G.Q[k][c] = m.verts[3 * b[lb[k]] + c];
        }
    }
    G.g = 4.0 * m.area[ti] * m.area[tj];
    G.ny[0] = m.n64[tj];
    G.ny[1] = m.n64[m.nt + tj];
    G.ny[2] = m.n64[2 * m.nt + tj];
    G.nx[0] = m.n64[ti];
    G.nx[1] = m.n64[m.nt + ti];
    G.nx[2] = m.n64[2 * m.nt + ti];
    return ns;
}

TD_HD int ss_npoints(int cls, int ng) {
    int n2 = ng * ng;
    return cls == 3 ? 6 * n2 : cls == 2 ? 6 * n2 * ng : cls == 1 ? 2 * n2 * n2 : 0;
}

// Identical pairs: rays of the six sectors of the z-plane (|det| = 1); common
// edge: cone triangles (u, p, q) with vertices on l(u,p,q) = 1.
static __constant__ float c_ss_rays[7][2] = {{1, 0}, {1, 1}, {0, 1}, {-1, 0}, {-1, -1}, {0, -1}, {1, 0}};
static __constant__ float c_ss_cones[6][3][3] = {
    {{0, 1, 0}, {1, 0, 0}, {1, 0, 1}},  {{0, 1, 0}, {1, 0, 1}, {0, 1, 1}},
    {{0, 0, 1}, {1, 0, 1}, {0, 1, 1}},  {{0, 1, 0}, {0, 1, 1}, {-1, 1, 0}},
    {{-1, 0, 0}, {0, 0, 1}, {0, 1, 1}}, {{-1, 0, 0}, {0, 1, 1}, {-1, 1, 0}}};

// Reference point q of a class's transformed integral: up to four coordinates
// a (identical: z1, z2, xi; edge: u, p, q; vertex: x1, x2, y1, y2), the weight
// without the Jacobian factor g, and the trial barycentric weights lam
// (parametrisation order; use G.loc to map to mesh-local vertices).
TD_D void ss_ref(int cls, int q, int ng, const double *gx, const double *gw, double a[4], double &wgt, double lam[3]) {
    a[3] = 0.0;
    if (cls == 3) {
        int sct = q / (ng * ng), i = (q / ng) % ng, b = q % ng;
        double xi = gx[i], eta = gx[b];
        const float *A = c_ss_rays[sct], *B = c_ss_rays[sct + 1];
        a[0] = A[0] + eta * (B[0] - A[0]);
        a[1] = A[1] + eta * (B[1] - A[1]);
        a[2] = xi;
        wgt = gw[i] * gw[b] * xi * (1.0 - xi) * (1.0 - xi) * 0.5;
        lam[0] = lam[1] = lam[2] = 0.0;  // identical pairs only occur for P0 x P0
    } else if (cls == 2) {
        int n3 = ng * ng * ng;
        int tr = q / n3, r = q % n3, i = r / (ng * ng), b = (r / ng) % ng, c = r % ng;
        double xi = gx[i], e1 = gx[b], e2 = gx[c];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double v0 = c_ss_cones[tr][0][k], v1 = c_ss_cones[tr][1][k], v2 = c_ss_cones[tr][2][k];
            a[k] = xi * (v0 + e1 * (v1 - v0) + e1 * e2 * (v2 - v1));
        }
        double u = a[0], p = a[1], qq = a[2];
        // |det| is 1 for all six cone triangles
        wgt = gw[i] * gw[b] * gw[c] * xi * xi * e1 * (1.0 - xi);
        double tlo = p > qq - u ? p : qq - u;
        double thi = u > 0.0 ? 1.0 - u : 1.0;
        double tm = 0.5 * (tlo + thi);
        double y1 = tm + u, y2 = qq;
        lam[0] = 1.0 - y1;
        lam[1] = y1 - y2;
        lam[2] = y2;
    } else {
        int n4 = ng * ng * ng * ng;
        int reg = q / n4, r = q % n4;
        int i = r / (ng * ng * ng), b = (r / (ng * ng)) % ng, c = (r / ng) % ng, e = r % ng;
        double xi = gx[i], w = gx[b], e1 = gx[c], e2 = gx[e];
        // region 0: the test triangle reaches out to xi, region 1: the trial triangle
        const double big0 = xi, big1 = xi * w, small0 = xi * e1, small1 = xi * e1 * e2;
        a[0] = reg == 0 ? big0 : small0;
        a[1] = reg == 0 ? big1 : small1;
        a[2] = reg == 0 ? small0 : big0;
        a[3] = reg == 0 ? small1 : big1;
        wgt = gw[i] * gw[b] * gw[c] * gw[e] * xi * xi * xi * e1;
        lam[0] = 1.0 - a[2];
        lam[1] = a[2] - a[3];
        lam[2] = a[3];
    }
}

// The reference points of the three classes in one array: per class eight rows
// (a0..a3, weight, lam0..lam2) of ss_npoints values, classes 1, 2, 3 in turn.
TD_HD int64_t ss_rule_off(int cls, int ng) {
    return (int64_t)8 * ((cls > 1 ? ss_npoints(1, ng) : 0) + (cls > 2 ? ss_npoints(2, ng) : 0));
}

// Edge vectors P1 - P0, P2 - P1, Q1 - Q0, Q2 - Q1 of a pair and the difference
// d = y - x of a reference point.
struct SsEdges {
    double p0[3], p1[3], q0[3], q1[3];
};
TD_D void ss_edges(const SingGeom &G, SsEdges &E) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        E.p0[k] = G.P[1][k] - G.P[0][k];
        E.p1[k] = G.P[2][k] - G.P[1][k];
        E.q0[k] = G.Q[1][k] - G.Q[0][k];
        E.q1[k] = G.Q[2][k] - G.Q[1][k];
    }
}
TD_D void ss_diff(int cls, const double a[4], const SsEdges &E, double d[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (cls == 3)
            d[k] = a[2] * (a[0] * E.p0[k] + a[1] * E.p1[k]);
        else if (cls == 2)
            d[k] = a[0] * E.p0[k] + a[2] * E.q1[k] - a[1] * E.p1[k];
        else
            d[k] = a[2] * E.q0[k] + a[3] * E.q1[k] - a[0] * E.p0[k] - a[1] * E.p1[k];
    }
}

// Quadrature point q of the transformed integral: difference vector d = y - x,
// weight (including the Jacobian factor g) and trial barycentric weights lam.
TD_D void ss_point(const SingGeom &G, int q, int ng, const double *gx, const double *gw,
                   double d[3], double &wgt, double lam[3]) {
    double a[4];
    SsEdges E;
    ss_ref(G.cls, q, ng, gx, gw, a, wgt, lam);
    ss_edges(G, E);
    ss_diff(G.cls, a, E, d);
    wgt *= G.g;
}

// Signed normal factor of the double-layer kernels at difference d = y - x:
// (x - y).n_y (DLP) or (y - x).n_x (ADLP).
template <int OP>
TD_HD double ss_dn(const SingGeom &G, const double d[3]) {
    return OP == TD_DLP ? -(d[0] * G.ny[0] + d[1] * G.ny[1] + d[2] * G.ny[2])
                        : d[0] * G.nx[0] + d[1] * G.nx[1] + d[2] * G.nx[2];
}

// Index of tj in ti's touching list, or -1.
TD_D int touching_slot(const MeshDev &m, int ti, int tj) {
    for (int p = m.tp_ptr[ti]; p < m.tp_ptr[ti + 1]; ++p)
        if (m.tp_tri[p] == tj) return m.tp_slot[p];
    return -1;
}
