// Per-source exact Hessians (Section IV-D: Newton steps need the exact 44 x 44
// Hessian of each source's block).
//
//   k_hess           per part of a work item: value, gradient and Hessian of the pixel
//                    terms wrt ten intermediate variables z of the (source, patch);
//                    the mixture terms are recomputed here, nothing is stored.  Its first
//                    CTAs take the sources' KL terms and parameter-only derivatives.
//   k_finalize_hess  one CTA per source: chain rule z -> theta over the source's patches,
//                    added to the KL Hessian; the full symmetric 44 x 44 matrix, the
//                    gradient and the local objective.
//
// The pixel terms depend on theta through ten variables z of the (source, patch).  With
// E_s = k_0 g_0 + k_1 g_1,  E2_s = q_0 g_0^2 + q_1 g_1^2,  Var_s = E2_s - E_s^2,
// k_i = a_i iota E[l_i] and q_i = a_i iota^2 E[l_i^2] (i = star, galaxy), the first four are A_i and
// Q_i with k_i = K_i A_i, q_i = L_i (A_i + Q_i), K_i = iota E[l_i] and L_i = iota^2 E[l_i^2] held at theta,
// where A_i = a_i and Q_i = 0.  (d/dA_i is d/da_i, whose parts K_i d/dk_i and L_i d/dq_i cancel
// in part: they are added at the pixel, before the sums are rounded.)
// z = (A_0, A_1, Q_0, Q_1, the mean, e_dev, G).  (The twelve y of the gradient passes hold
// a_i, E[l_i] and E[l_i^2] apart: their rows of the Hessian are multiples of each other.)
// With e = dE_s/dz, v = dVar_s/dz = dE2_s/dz - 2 E_s e and the second derivatives
// DE = d2E_s/dz2, DE2 = d2E2_s/dz2:
//   d2 ll/dz2 = (h_EE - 2 c_V) e e' + h_EV (e v' + v e') + (c_E - 2 c_V E_s) DE + c_V DE2
//   h_EE = -x (1/E^2 + 3 Var/E^4),  h_EV = x / E^3,  h_VV = 0.
// Per Gaussian component N (log-density derivatives, q = P d, C = Sigma_psf + nu G):
//   dlogN/dmu = q,  d2logN/dmu2 = -P,
//   dlogN/dC[E] = (q'Eq - tr PE)/2,   d2logN/dmu dC[F] = -P F q,
//   d2logN/dC[E]dC[F] = -q'E P F q + tr(P E P F)/2,   d2N = N (dlogN dlogN' + d2logN).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "fp64_profile.cuh"
#include "internal.cuh"
#include "async_copy.cuh"
#include "source_math.cuh"
#include "whiten.cuh"

namespace cel {

namespace {

// 2^x on the SFU (results below 2^-126 become 0)
__device__ __forceinline__ float ex2h(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lgh(float x) { return logf(x); }
__device__ __forceinline__ double lgh(double x) { return log(x); }

// packed index of a symmetric N x N (upper triangle by rows; a <= b not required)
template <int N>
__host__ __device__ __forceinline__ constexpr int sym(int a, int b) {
    return a <= b ? a * N - a * (a - 1) / 2 + b - a : b * N - b * (b - 1) / 2 + a - b;
}

}  // namespace

// Sums v[0 .. 64) over the warp's 32 lanes: lane l is left with the sums of entries 2 l,
// 2 l + 1 in v[0], v[1].  Five halving steps: at the step on lane bit m the two lanes that
// differ in m hold the same index range; the one with m set keeps the upper half and adds
// its partner's upper half, the other keeps and adds the lower half.  62 shuffles instead
// of 5 per entry.  v[64], v[65] are summed onto every lane.
static_assert(HV == 66, "64 scattered sums and two");
template <class R>
__device__ __forceinline__ void warp_reduce_scatter(R (&v)[HV], int lane) {
#pragma unroll
    for (int m = 16, n = 64; m > 0; m >>= 1, n >>= 1) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const R send = up ? v[i] : v[i + n / 2];
            const R keep = up ? v[i + n / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
#pragma unroll
        for (int i = 64; i < HV; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], m);
    }
}

// the sums of lower degree: A (3), B (2), L (2), N from the base sums
template <class R>
__host__ __device__ __forceinline__ void derived_sums(const R (&b)[NBS], R g1, R g2, R (&A)[3], R (&B)[2], R (&L)[2],
                                                      R& N) {
    A[0] = b[BS_C] + g1 * b[BS_D3];
    A[1] = b[BS_C + 1] + g1 * b[BS_D3 + 1];
    A[2] = b[BS_C + 3] + g2 * b[BS_D3 + 3];
    B[0] = A[0] + g1 * b[BS_D2];
    B[1] = A[2] + g2 * b[BS_D2 + 2];
    L[0] = b[BS_LL] + g1 * A[0];
    L[1] = b[BS_LL + 2] + g2 * A[2];
    N = L[0] + g1 * B[0];
}

// the 35 sums from the base sums over the exp components and over the dev components (each
// at unit e_dev weight): N's at weights 1 - e_dev and e_dev, the e_dev sums their difference
template <class R>
__host__ __device__ __forceinline__ void combine_groups(const R (&be)[NBS], const R (&bd)[NBS], R g1, R g2, R edev,
                                                        R (&s)[NWS]) {
    R c[NBS], A[3], B[2], L[2], N;
    const R fe = (R)1 - edev;
#pragma unroll
    for (int i = 0; i < NBS; ++i) c[i] = fe * be[i] + edev * bd[i];
    derived_sums(c, g1, g2, A, B, L, N);
    s[WS_N] = N;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        s[WS_L + i] = L[i];
        s[WS_B + i] = B[i];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        s[WS_A + i] = A[i];
        s[WS_LL + i] = c[BS_LL + i];
        s[WS_D2 + i] = c[BS_D2 + i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        s[WS_C + i] = c[BS_C + i];
        s[WS_D3 + i] = c[BS_D3 + i];
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) s[WS_D4 + i] = c[BS_D4 + i];
#pragma unroll
    for (int i = 0; i < NBS; ++i) c[i] = bd[i] - be[i];   // those that the e_dev sums need
    derived_sums(c, g1, g2, A, B, L, N);
    s[WS_NE] = N;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        s[WS_LE + i] = L[i];
        s[WS_BE + i] = B[i];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) s[WS_AE + i] = A[i];
}

// adds PSF component k's galaxy terms at one pixel, from its 35 sums, to the pixel-frame
// value, gradient (mx, my, Gxx, Gxy, Gyy), e_dev derivatives and packed 5 x 5 Hessian.
// (The Kronecker deltas are branches on constants: a product with a constant 0 would be
// computed.)
template <class R>
__host__ __device__ __forceinline__ void whitened_add(const R (&s)[NWS], R z1, R z2, const R* fr, R& g1, R (&d1)[5],
                                                      R& de, R (&h1)[15], R (&he)[5]) {
    const R z[2] = {z1, z2};
    const R Z2[3] = {z1 * z1, z1 * z2, z2 * z2};
    const R Z3[4] = {z1 * Z2[0], z1 * Z2[1], z1 * Z2[2], z2 * Z2[2]};
    const R Z4[5] = {Z2[0] * Z2[0], Z2[0] * Z2[1], Z2[0] * Z2[2], Z2[1] * Z2[2], Z2[2] * Z2[2]};
    R T[2][2], K[3][3];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        T[a][0] = fr[2 * a];
        T[a][1] = fr[2 * a + 1];
    }
#pragma unroll
    for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int p = 0; p < 3; ++p) K[e][p] = fr[WF_K + 3 * e + p];
    g1 += s[WS_N];
    de += s[WS_NE];
    // d/dmu = T' r-sums; d/dG[E] = K (W11, 2 W12, W22), W_ab = (z_a z_b A_ab - delta_ab B_a) / 2
    const R gm[2] = {z1 * s[WS_L], z2 * s[WS_L + 1]};
    const R ge[2] = {z1 * s[WS_LE], z2 * s[WS_LE + 1]};
    R Wv[3], Wev[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int a = wpa(p), b = wpb(p);
        R v = Z2[a + b] * s[WS_A + a + b], u = Z2[a + b] * s[WS_AE + a + b];
        if (a == b) {
            v = (R)0.5 * (v - s[WS_B + a]);
            u = (R)0.5 * (u - s[WS_BE + a]);
        }
        Wv[p] = v;
        Wev[p] = u;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        d1[i] += T[0][i] * gm[0] + T[1][i] * gm[1];
        he[i] += T[0][i] * ge[0] + T[1][i] * ge[1];
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        d1[2 + e] += K[e][0] * Wv[0] + K[e][1] * Wv[1] + K[e][2] * Wv[2];
        he[2 + e] += K[e][0] * Wev[0] + K[e][1] * Wev[1] + K[e][2] * Wev[2];
    }
    // (mu, mu) = T' X T, X_ab = z_a z_b LL_ab - delta_ab L_a: the pixel-frame entries are K X
    {
        const R X[3] = {Z2[0] * s[WS_LL] - s[WS_L], Z2[1] * s[WS_LL + 1], Z2[2] * s[WS_LL + 2] - s[WS_L + 1]};
        h1[0] += K[0][0] * X[0] + (R)2 * K[0][1] * X[1] + K[0][2] * X[2];
        h1[1] += (R)0.5 * (K[1][0] * X[0] + K[1][2] * X[2]) + K[1][1] * X[1];
        h1[5] += K[2][0] * X[0] + (R)2 * K[2][1] * X[1] + K[2][2] * X[2];
    }
    // (mu, G): T' (Yv K'), Y_{a,bc} = (z_a z_b z_c C_abc - delta_bc z_a A_ab - delta_ab z_c A_ac
    //                                  - delta_ac z_b A_ab) / 2
    R YK[2][3];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        R Yv[3];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const int b = wpa(p), c = wpb(p);
            R v = Z3[a + b + c] * s[WS_C + a + b + c];
            if (b == c && a == b) v -= (R)3 * z[a] * s[WS_A + 2 * a];
            else if (b == c) v -= z[a] * s[WS_A + 1];
            else v -= z[1 - a] * s[WS_A + 1];   // p = (1, 2): a is one of the two
            Yv[p] = b == c ? (R)0.5 * v : v;
        }
#pragma unroll
        for (int e = 0; e < 3; ++e) YK[a][e] = K[e][0] * Yv[0] + K[e][1] * Yv[1] + K[e][2] * Yv[2];
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        h1[2 + e] += T[0][0] * YK[0][e] + T[1][0] * YK[1][e];
        h1[6 + e] += T[0][1] * YK[0][e] + T[1][1] * YK[1][e];
    }
    // (G, G) = K Vm K', Vm_pq = m_p m_q V_{ab,cd} / 4 (pairs p = ab, q = cd; symmetric):
    //   V = z_a z_b z_c z_d D4 - delta_cd z_a z_b D3_abc - delta_ab z_c z_d D3_acd + delta_ab delta_cd D2_ac
    //       - (delta_bc z_a z_d + delta_bd z_a z_c) D3 - (delta_ac z_b z_d + delta_ad z_b z_c) D3
    //       + (delta_bc delta_ad + delta_ac delta_bd) D2_ab
    R Vm[3][3];
    {
        const R* D2 = s + WS_D2;
        const R* D3 = s + WS_D3;
        const R* D4 = s + WS_D4;
        Vm[0][0] = (R)0.25 * (Z4[0] * D4[0] + (R)3 * D2[0]) - (R)1.5 * Z2[0] * D3[0];
        Vm[2][2] = (R)0.25 * (Z4[4] * D4[4] + (R)3 * D2[2]) - (R)1.5 * Z2[2] * D3[3];
        Vm[0][2] = (R)0.25 * (Z4[2] * D4[2] - Z2[0] * D3[1] - Z2[2] * D3[2] + D2[1]);
        Vm[0][1] = (R)0.5 * Z4[1] * D4[1] - (R)1.5 * Z2[1] * D3[1];
        Vm[1][2] = (R)0.5 * Z4[3] * D4[3] - (R)1.5 * Z2[1] * D3[2];
        Vm[1][1] = Z4[2] * D4[2] - Z2[0] * D3[1] - Z2[2] * D3[2] + D2[1];
        Vm[1][0] = Vm[0][1];
        Vm[2][0] = Vm[0][2];
        Vm[2][1] = Vm[1][2];
    }
    R KV[3][3];
#pragma unroll
    for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int q = 0; q < 3; ++q) KV[e][q] = K[e][0] * Vm[0][q] + K[e][1] * Vm[1][q] + K[e][2] * Vm[2][q];
    int c = 9;
#pragma unroll
    for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int f = e; f < 3; ++f, ++c) h1[c] += KV[e][0] * K[f][0] + KV[e][1] * K[f][1] + KV[e][2] * K[f][2];
}

// The pixel-frame ellipse is G = A W A' with W = ah I + bh (cos 2phi, sin 2phi; sin 2phi,
// -cos 2phi), ah = sigma^2 (1 + rho^2) / 2, bh = sigma^2 (1 - rho^2) / 2.  Its first and
// second derivatives over s = (e_axis, e_angle, e_scale) are A (dW) A' and A (d2W) A':
// dW and d2W depend on theta alone (computed once per source, by one thread), and each
// patch maps them through its own A (one output per thread).  Host-callable for tests.
__host__ __device__ void shape_w_derivs(const double* th, double dW[3][3], double d2W[3][3][3]) {
    const double rho = th[P_AXIS], phi = th[P_ANGLE], sg = th[P_SCALE];
    const double bh = 0.5 * sg * sg * (1.0 - rho * rho);
    double s2, c2;
    sincos(2.0 * phi, &s2, &c2);
    // first derivatives (index order rho = 0, phi = 1, sigma = 2; W as xx, xy, yy)
    {
        const double da = sg * sg * rho, db = -sg * sg * rho;
        dW[0][0] = da + db * c2; dW[0][1] = db * s2; dW[0][2] = da - db * c2;
    }
    dW[1][0] = -2.0 * bh * s2; dW[1][1] = 2.0 * bh * c2; dW[1][2] = 2.0 * bh * s2;
    {
        const double da = sg * (1.0 + rho * rho), db = sg * (1.0 - rho * rho);
        dW[2][0] = da + db * c2; dW[2][1] = db * s2; dW[2][2] = da - db * c2;
    }
    // second derivatives of ah, bh over (rho, sigma)
    const double bh_r = -sg * sg * rho, bh_s = sg * (1.0 - rho * rho);
    const double ah_rr = sg * sg, ah_ss = 1.0 + rho * rho, ah_rs = 2.0 * sg * rho;
    const double bh_rr = -sg * sg, bh_ss = 1.0 - rho * rho, bh_rs = -2.0 * sg * rho;
    auto set = [&](int a, int b, double xx, double xy, double yy) {
        d2W[a][b][0] = d2W[b][a][0] = xx;
        d2W[a][b][1] = d2W[b][a][1] = xy;
        d2W[a][b][2] = d2W[b][a][2] = yy;
    };
    set(0, 0, ah_rr + bh_rr * c2, bh_rr * s2, ah_rr - bh_rr * c2);
    set(2, 2, ah_ss + bh_ss * c2, bh_ss * s2, ah_ss - bh_ss * c2);
    set(0, 2, ah_rs + bh_rs * c2, bh_rs * s2, ah_rs - bh_rs * c2);
    set(0, 1, -2.0 * bh_r * s2, 2.0 * bh_r * c2, 2.0 * bh_r * s2);
    set(2, 1, -2.0 * bh_s * s2, 2.0 * bh_s * c2, 2.0 * bh_s * s2);
    set(1, 1, -4.0 * bh * c2, -4.0 * bh * s2, 4.0 * bh * c2);
}

// component c (xx, xy, yy) of A w A' for a symmetric w = (wxx, wxy, wyy)
__host__ __device__ __forceinline__ double a_transform(const double* A, const double* w, int c) {
    const double wxx = w[0], wxy = w[1], wyy = w[2];
    if (c == 0) return A[0] * A[0] * wxx + 2.0 * A[0] * A[1] * wxy + A[1] * A[1] * wyy;
    if (c == 1) return A[0] * A[2] * wxx + (A[0] * A[3] + A[1] * A[2]) * wxy + A[1] * A[3] * wyy;
    return A[2] * A[2] * wxx + 2.0 * A[2] * A[3] * wxy + A[3] * A[3] * wyy;
}

// ---- The terms of a source that depend on its parameters alone, two tasks ahead of the pixel
// work in k_hess's queue (their FP64 latencies then pass behind it): the KL value, gradient and
// Hessian, the brightness moments of the five bands and the world-frame shape derivatives.
// hess_out receives -KL'' and zeros; the rest goes to the source's record.
constexpr int HR_KL = 0, HR_KLG = 1, HR_MOM = HR_KLG + NP, HR_DW = HR_MOM + 20, HR_D2W = HR_DW + 9,
              HR_A = HR_D2W + 27;
static_assert(HR_A + 2 <= HREC && HREC % 2 == 0, "the source's record");

struct SourceTerms {
    int n_src;
    const double* theta;
    const ModelDev* md;
    double* hsrc;        // [n_src][HREC]
    double* kl;
    double* hess;        // [n_src][NP][NP]
    int32_t* status;     // nullable: no domain check
};

// KL value, gradient and Hessian of one source by one warp (the closed forms of
// kl_value_grad and their derivatives).  One logarithm and one reciprocal per lane (lanes
// 8 i + d: k_id; 16 + 4 i + j: c2; 24 + i: a_i; 26 + i: r2_i), the 4 x 4 algebra of
// colour-prior component (i, d) on lane 8 i + d, the sums over components by shuffles, and
// then every entry written by one lane.
__device__ __forceinline__ void kl_terms_warp(const ModelDev& md, const double* th, double* rec, double* kl_out,
                                              double* H) {
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int i = (lane >> 3) & 1, d = lane & 7;
    auto put = [&](int p, int q, double v) {
        H[p * NP + q] = -v;
        if (p != q) H[q * NP + p] = -v;
    };
    double x = 1.0;
    if (lane < 16) x = th[P_K + lane];
    else if (lane < 24) x = th[P_C2 + lane - 16];
    else if (lane < 26) x = th[P_A + lane - 24];
    else if (lane < 28) x = th[P_R2 + lane - 26];
    double lv = log(x);
    const double rv = 1.0 / x;
    if (lane < 16) lv -= md.prior_logw[i][d];
    else if (lane >= 24 && lane < 26) lv -= md.prior_logphi[lane - 24];
    else if (lane >= 26 && lane < 28) lv = md.prior_logpv[lane - 26] - lv;
    double slog = 0.0, ic2[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        slog += __shfl_sync(full, lv, 16 + 4 * i + j);
        ic2[j] = __shfl_sync(full, rv, 16 + 4 * i + j);
    }
    const double a = th[P_A + i];
    // sums over the components of: k (log k / w + KL_d), k, k P diff, k diag P, k P (upper)
    double sum[20];
#pragma unroll
    for (int u = 0; u < 20; ++u) sum[u] = 0.0;
    if (lane < 16) {
        const double k = th[P_K + lane];
        const double* Pm = md.prior_P[i][d];
        const double* mu = md.prior_mu[i][d];
        double diff[4], quad = 0.0, tr = 0.0;
#pragma unroll
        for (int j = 0; j < 4; ++j) diff[j] = th[P_C1 + 4 * i + j] - mu[j];
        const int ik = P_K + lane;
        int c = 10;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            double pd = 0.0;
#pragma unroll
            for (int l = 0; l < 4; ++l) pd += Pm[4 * j + l] * diff[l];
            quad += diff[j] * pd;
            tr += Pm[5 * j] * th[P_C2 + 4 * i + j];
            sum[2 + j] = k * pd;
            sum[6 + j] = k * Pm[5 * j];
            put(ik, P_C1 + 4 * i + j, a * pd);
            put(ik, P_C2 + 4 * i + j, 0.5 * a * (Pm[5 * j] - ic2[j]));
#pragma unroll
            for (int l = j; l < 4; ++l, ++c) sum[c] = k * Pm[4 * j + l];
        }
        const double klc = 0.5 * (tr + quad - 4.0 + md.prior_logdet[i][d] - slog);
        sum[0] = k * (lv + klc);
        sum[1] = k;
        const double dk = lv + 1.0 + klc;
        rec[HR_KLG + ik] = a * dk;
        put(P_A + i, ik, dk);
        put(ik, ik, a * rv);
    }
#pragma unroll
    for (int u = 0; u < 20; ++u)
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) sum[u] += __shfl_xor_sync(full, sum[u], o);
    const double la = __shfl_sync(full, lv, 24 + i), ia = __shfl_sync(full, rv, 24 + i);
    const double lpr = __shfl_sync(full, lv, 26 + i), ir2 = __shfl_sync(full, rv, 26 + i);
    double klv = 0.0;
    if (lane < 16) {
        const int iA = P_A + i;
        if (d < 4) {
            // colour j = d; the row's upper entries of sum_d k_d P_d
            double kp = sum[2], kd = sum[6], ic = ic2[0], row[4] = {sum[10], sum[11], sum[12], sum[13]};
            if (d == 1) { kp = sum[3]; kd = sum[7]; ic = ic2[1]; row[1] = sum[14]; row[2] = sum[15]; row[3] = sum[16]; }
            if (d == 2) { kp = sum[4]; kd = sum[8]; ic = ic2[2]; row[2] = sum[17]; row[3] = sum[18]; }
            if (d == 3) { kp = sum[5]; kd = sum[9]; ic = ic2[3]; row[3] = sum[19]; }
            const int c1 = P_C1 + 4 * i + d, c2 = P_C2 + 4 * i + d;
            const double sc2 = 0.5 * (kd - sum[1] * ic);
            rec[HR_KLG + c1] = a * kp;
            rec[HR_KLG + c2] = a * sc2;
            put(iA, c1, kp);
            put(iA, c2, sc2);
            put(c2, c2, 0.5 * a * sum[1] * ic * ic);
#pragma unroll
            for (int l = 0; l < 4; ++l)
                if (l >= d) put(c1, P_C1 + 4 * i + l, a * row[l]);
        } else {
            const double r1 = th[P_R1 + i], r2 = th[P_R2 + i];
            const double dr = r1 - md.prior_r[i][0], ipv = md.prior_inv_pv[i];
            if (d == 4) {
                const double K = 0.5 * (lpr + (r2 + dr * dr) * ipv - 1.0) + sum[0];
                klv = a * (la + K);
                rec[HR_KLG + iA] = la + 1.0 + K;
                put(iA, iA, ia);
            } else if (d == 5) {
                rec[HR_KLG + P_R1 + i] = a * dr * ipv;
                put(iA, P_R1 + i, dr * ipv);
                put(P_R1 + i, P_R1 + i, a * ipv);
            } else if (d == 6) {
                const double v = 0.5 * (ipv - ir2);
                rec[HR_KLG + P_R2 + i] = a * v;
                put(iA, P_R2 + i, v);
                put(P_R2 + i, P_R2 + i, 0.5 * a * ir2 * ir2);
            }
        }
    }
    if (lane < 6) rec[HR_KLG + lane] = 0.0;   // position and shape carry no prior
    klv += __shfl_xor_sync(full, klv, 8);
    klv = __shfl_sync(full, klv, 4);
    if (lane == 0) {
        rec[HR_KL] = klv;
        *kl_out = klv;
    }
}

// task 0 or 1 of source s by one warp; sm: NP doubles of the warp's shared memory
__device__ __forceinline__ void source_terms(const SourceTerms& a, int s, int task, double* sm) {
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < NP; i += 32) {
        sm[i] = a.theta[(size_t)NP * s + i];
        if (a.status && task == 0) theta_domain_check(i, sm[i], a.status);
    }
    __syncwarp();
    double* rec = a.hsrc + (size_t)HREC * s;
    if (task == 0) {
        double* H = a.hess + (size_t)NP * NP * s;   // the caller's: 8-byte aligned
        for (int i = lane; i < NP * NP; i += 32) H[i] = 0.0;
        __syncwarp();
        kl_terms_warp(*a.md, sm, rec, a.kl + s, H);
    } else {
        if (lane < 10) band_moments(sm, lane >> 1, lane & 1, rec[HR_MOM + 2 * lane], rec[HR_MOM + 2 * lane + 1]);
        if (lane >= 30) rec[HR_A + lane - 30] = sm[P_A + lane - 30];
        if (lane == 10) {
            double dW[3][3], d2W[3][3][3];
            shape_w_derivs(sm, dW, d2W);
            for (int i = 0; i < 9; ++i) rec[HR_DW + i] = dW[i / 3][i % 3];
            for (int i = 0; i < 27; ++i) rec[HR_D2W + i] = d2W[i / 9][i / 3 % 3][i % 3];
        }
    }
    __syncwarp();
}

// Shared memory of k_hess: in FP64 the CTA's table of 2^x; then per warp two stages, each a
// part's record, its patch's table and (FP32) frames, the part's frames (FP64) and rows, and the
// part's sums.  In bytes, for tables of n_comp components.
constexpr int HESS_WARPS = 4;
template <class R>
struct HessLay {
    static constexpr bool DBL = sizeof(R) == 8;
    static constexpr int tab_bytes = DBL ? EX_N * 8 : 0;
    static constexpr int tbl = (int)sizeof(HItem);   // in the stage
    int sfr, stage, fr, rows, sums, warp;
    __host__ __device__ explicit HessLay(int n_comp) {
        sfr = tbl + (T_GAL + n_comp * GAL_STRIDE) * (int)sizeof(R);
        stage = sfr + (DBL ? 0 : MAXPSF * WFR * 4);
        fr = 2 * stage;
        rows = fr + (DBL ? MAXPSF * WFR * 8 : 0);
        sums = rows + n_comp * BROW * (int)sizeof(R);
        warp = sums + HV * 8;
    }
    __host__ __device__ int bytes() const { return tab_bytes + HESS_WARPS * warp; }
};
static_assert(sizeof(HItem) % 16 == 0 && GAL_STRIDE % 4 == 0 && BROW % 4 == 0 && HV % 2 == 0,
              "every piece starts on a 16-byte boundary");

// 16 bytes from global to shared memory, asynchronously
__device__ __forceinline__ void copy16_async(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Per part of a work item: the sums over its pixels of ll, d ll / dz and d2 ll / dz2.  The
// mixture in the whitened frame; FP64 as in fp64_profile.cuh.  E and Var of a singly covered
// pixel (single) are formed here, those of the others come from the maps.
// Persistent warps take tasks from a queue, warp w's first two being tasks w and w + W (W warps):
// the sources' parameter-only terms, then the parts.  While a part is computed the next one's
// record and table are on their way to the warp's other stage.  A warp goes through its part 32
// pixels at a time and shares nothing with the others, so it waits neither for memory nor at a
// barrier; one CTA per part had its warps waiting for loads and barriers 40 % of the time.
// 500 sources, FP32: 125 -> 112 us back to back (117 alone with cold caches: issue slots 62 % used,
// FMA pipe 48 %; 56 us at that pipe's peak); 64 crowded sources, FP64: 608 -> 587 us (FP64 pipe 88 %).
// Bound by the FP32 or the FP64 pipe: 12 (packed) / 25 of its instructions per component, where
// the 35 sums accumulated one by one took 38 and the pixel-frame formulas about 140.
template <class R>
struct HessArgs {
    const HItem* parts;
    int n_part;
    const ImgMeta* img;
    const PatchGeo* geo;
    int n_comp, nprof, n_exp;   // components of the largest table; profile components
    const float* pixels;
    const float* sky_map;
    const R* tbl;
    const float* hframe;
    const uint8_t* single;
    const R* emap;
    const R* vmap;
    double* part;
    const int32_t* src_active;
    int32_t* queue;
    SourceTerms src;
};

// NE, ND: the exp and dev components of the model where they are known (the paper's model and
// the synthetic workloads: 6 and 8), else 0.
template <class R, int NE, int ND>
__global__ void __launch_bounds__(32 * HESS_WARPS, sizeof(R) == 8 ? 2 : 4) k_hess(const HessArgs<R> a) {
    constexpr bool DBL = std::is_same<R, double>::value;
    extern __shared__ __align__(16) unsigned char smem[];
    const HessLay<R> L(a.n_comp);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* tab = reinterpret_cast<double*>(smem);
    unsigned char* sm = smem + HessLay<R>::tab_bytes + warp * L.warp;   // this warp's
    R* rows = reinterpret_cast<R*>(sm + L.rows);
    double* sums = reinterpret_cast<double*>(sm + L.sums);
    const int nprof = a.nprof, n_exp = a.n_exp;
    if constexpr (DBL) {
        load_exp2_table(tab);
        __syncthreads();
    }
    // tasks [0, n_term): the sources' terms; then the parts
    const int W = (int)gridDim.x * HESS_WARPS, n_term = 2 * a.src.n_src, n_task = n_term + a.n_part;
    auto patch_of = [&](int task) {   // -1: not a part
        return task >= n_term && task < n_task ? a.parts[task - n_term].patch : -1;
    };
    // the copies of one part: its record, its patch's table and (FP32) frames
    auto fetch = [&](int task, int patch, int b) {
        unsigned char* st = sm + b * L.stage;
        auto copy = [&](int to, const void* from, int n) {
            for (int i = lane; i < n; i += 32)
                copy16_async(st + to + 16 * i, reinterpret_cast<const unsigned char*>(from) + 16 * i);
        };
        if (patch >= 0) {
            copy(0, a.parts + (task - n_term), (int)sizeof(HItem) / 16);
            copy(HessLay<R>::tbl, a.tbl + (size_t)patch * TBL_STRIDE, (L.sfr - HessLay<R>::tbl) / 16);
            if (!DBL) copy(L.sfr, a.hframe + (size_t)patch * HF_STRIDE, MAXPSF * WFR / 4);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int task = warp * (int)gridDim.x + (int)blockIdx.x, next = task + W;
    fetch(task, patch_of(task), 0);
    int next_patch = patch_of(next);
    for (int b = 0; task < n_task; b ^= 1) {
        const int cur = task;
        fetch(next, next_patch, b ^ 1);   // the stage was last read in the previous task
        int claim = 0;
        if (lane == 0) claim = 2 * W + atomicAdd(a.queue, 1);
        task = next;
        if (cur < n_term) {
            const int s = cur >> 1;
            if (!a.src_active || a.src_active[s]) source_terms(a.src, s, cur & 1, sums);
            next = __shfl_sync(0xffffffffu, claim, 0);
            next_patch = patch_of(next);
            continue;
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const HItem& it = *reinterpret_cast<const HItem*>(sm + b * L.stage);
        if (a.src_active && !a.src_active[it.src]) {
            __syncwarp();
            next = __shfl_sync(0xffffffffu, claim, 0);
            next_patch = patch_of(next);
            continue;
        }
        const R* sT = reinterpret_cast<const R*>(sm + b * L.stage + HessLay<R>::tbl);
        R* frames = reinterpret_cast<R*>(DBL ? sm + L.fr : sm + b * L.stage + L.sfr);
        const int npsf = it.npsf;
        if (DBL && lane < npsf) {
            const R* F = sT + T_STAR + lane * STAR_STRIDE;
            R* fr = frames + lane * WFR;
            for (int i = 0; i < 4; ++i) fr[i] = F[i];
            fr[WF_G] = F[4];
            fr[WF_G + 1] = F[5];
            whiten_shape_map(fr);
            fr[15] = F[6];
        }
        for (int i = lane; i < npsf * nprof; i += 32) {
            // the exponent's coefficients and the 19 weights at unit e_dev weight
            const R* Gr = sT + T_GAL + i * GAL_STRIDE;
            R* row = rows + i * BROW;
            if constexpr (DBL) {
                row[0] = Gr[0];
                row[1] = Gr[1];
                row[2] = Gr[2];
                base_row(Gr[3], Gr[9], Gr[0] * EX_IHALF, Gr[1] * EX_IHALF, row + 3);
                row[3 + NBS] = 0;
            } else {
                const float* fr = frames + (i / nprof) * WFR;
                const float nu = Gr[9], l1 = 1.f / (1.f + nu * fr[WF_G]), l2 = 1.f / (1.f + nu * fr[WF_G + 1]);
                row[0] = (float)(-0.5 * LOG2E_W) * l1;
                row[1] = (float)(-0.5 * LOG2E_W) * l2;
                row[2] = Gr[3];
                base_row(i % nprof >= n_exp ? Gr[8] : -Gr[8], nu, l1, l2, row + 4);   // on a 16-byte boundary
                row[4 + NBS] = 0;
            }
        }
        for (int i = lane; i < HV; i += 32) sums[i] = 0.0;
        __syncwarp();
        // a_i, K_i, L_i, a_i K_i, a_i L_i: once per part in FP64 (for all of its pixels' FP64 instructions),
        // per pixel in FP32, where the registers are short
        struct Light {
            R a0, a1, K0, K1, L0, L1, k0, k1, l0, l1;
        };
        auto light = [&]() {
            const R iota = sT[H_IOTA];
            Light p;
            p.a0 = sT[H_A0];
            p.a1 = sT[H_A1];
            p.K0 = iota * sT[H_EL0];
            p.K1 = iota * sT[H_EL1];
            p.L0 = iota * iota * sT[H_EL20];
            p.L1 = iota * iota * sT[H_EL21];
            p.k0 = p.a0 * p.K0;
            p.k1 = p.a1 * p.K1;
            p.l0 = p.a0 * p.L0;
            p.l1 = p.a1 * p.L1;
            return p;
        };
        Light part_light;
        if constexpr (DBL) part_light = light();
        for (int c0 = 0; c0 < it.n; c0 += 32) {
            // the pixel's data, asked for before the mixture
            const bool ok = c0 + lane < it.n;
            const int q = it.q0 + (ok ? c0 + lane : 0);
            const int yy = q / it.w, xx = q - yy * it.w;
            const int64_t m = it.m0 + (int64_t)yy * it.W + xx;
            const R x = (R)a.pixels[m];
            const bool alone = a.single && a.single[it.sp0 + q];
            R E, V = 0;
            if (alone) {
                const ImgMeta& im = a.img[a.geo[it.patch].img];
                E = im.has_sky_map ? (R)a.sky_map[m] : (R)im.sky;
            } else {
                E = a.emap[m];
                V = a.vmap[m];
            }
            R out[HV];
#pragma unroll
            for (int i = 0; i < HV; ++i) out[i] = 0;
            if (ok) {
                // star: value, gradient (mx, my), Hessian (xx, xy, yy)
                R g0 = 0, d0[2] = {0, 0}, h0[3] = {0, 0, 0};
                // galaxy: value; gradient over z5 = (mx, my, Gxx, Gxy, Gyy); e_dev derivative;
                // Hessian over z5 (packed 15); e_dev x z5
                R g1 = 0, d1[5] = {0, 0, 0, 0, 0}, de = 0, h1[15], he[5] = {0, 0, 0, 0, 0};
#pragma unroll
                for (int i = 0; i < 15; ++i) h1[i] = 0;
                const R edev = sT[H_EDEV];
                for (int k = 0; k < npsf; ++k) {
                    const R dx = (R)xx - sT[T_MEAN + 2 * k], dy = (R)yy - sT[T_MEAN + 2 * k + 1];
                    const R* fr = frames + k * WFR;
                    const R z1 = fr[0] * dx + fr[1] * dy, z2 = fr[2] * dx + fr[3] * dy;
                    const R z1s = z1 * z1, z2s = z2 * z2;
                    float f1 = 0.f, f2 = 0.f;
                    if constexpr (DBL) {
                        f1 = (float)z1s;
                        f2 = (float)z2s;
                    }
                    auto star = [&]() {
                        R n, qx, qy, pxx, pxy, pyy;
                        if constexpr (DBL) {
                            // P d = T' z and P = T' T
                            n = fr[15] *
                                ex2_quad(EX_HALF, z1s, EX_HALF, z2s, (float)EX_HALF, f1, (float)EX_HALF, f2, tab);
                            qx = fr[0] * z1 + fr[2] * z2;
                            qy = fr[1] * z1 + fr[3] * z2;
                            pxx = fr[WF_K] + fr[WF_K + 2];
                            pxy = (R)0.5 * (fr[WF_K + 3] + fr[WF_K + 5]);
                            pyy = fr[WF_K + 6] + fr[WF_K + 8];
                        } else {
                            // in the pixel frame: with z in FP32 a source's gradient and Hessian were off
                            // by a quarter more (500 sources, the medians of their errors against 64
                            // bits: 2.5e-7 and 1.7e-7, here 1.9e-7 and 1.3e-7)
                            const R* S = sT + T_STAR + k * STAR_STRIDE;
                            pxx = S[4];
                            pxy = S[5];
                            pyy = S[6];
                            qx = pxx * dx + pxy * dy;
                            qy = pxy * dx + pyy * dy;
                            n = S[7] * ex2h(fmaf((float)(-0.5 * LOG2E_W), fmaf(dx, qx, dy * qy), S[3]));
                        }
                        g0 += n;
                        d0[0] += n * qx;
                        d0[1] += n * qy;
                        h0[0] += n * (qx * qx - pxx);
                        h0[1] += n * (qx * qy - pxy);
                        h0[2] += n * (qy * qy - pyy);
                    };
                    if (DBL) star();   // (behind the galaxy's terms in FP32: fewer registers spill)
                    const R* row = rows + k * nprof * BROW;
                    // the base sums over one group's components (N of them where N > 0, else n)
                    auto group = [&](auto N, int n, R (&b)[NBS]) {
                        if constexpr (DBL) {
#pragma unroll
                            for (int m = 0; m < NBS; ++m) b[m] = 0;
                            for (int j = 0; j < n; ++j, row += BROW) {
                                double cw[BROW];
#pragma unroll
                                for (int u = 0; u < (3 + NBS + 1) / 2; ++u) {
                                    const double2 v = reinterpret_cast<const double2*>(row)[u];
                                    cw[2 * u] = v.x;
                                    cw[2 * u + 1] = v.y;
                                }
                                const float2 ab = as_float2(cw[2]);
                                const double e = ex2_quad(cw[0], z1s, cw[1], z2s, ab.x, f1, ab.y, f2, tab);
#pragma unroll
                                for (int m = 0; m < NBS; ++m) b[m] += e * cw[3 + m];
                            }
                        } else {
                            // packed FP32x2: the 19 weights as ten pairs (half the issue slots)
                            constexpr int NPR = (NBS + 1) / 2;
                            float2 bb[NPR];
#pragma unroll
                            for (int m = 0; m < NPR; ++m) bb[m] = make_float2(0.f, 0.f);
                            auto value = [&](const R* r) {
                                const float4 c = *reinterpret_cast<const float4*>(r);
                                return ex2h(fmaf(c.x, z1s, fmaf(c.y, z2s, c.z)));
                            };
                            auto add = [&](const R* r, float e) {
                                const float2 ee = make_float2(e, e);
#pragma unroll
                                for (int u = 0; u < NPR / 2; ++u) {
                                    const float4 w = reinterpret_cast<const float4*>(r)[1 + u];
                                    bb[2 * u] = __ffma2_rn(ee, make_float2(w.x, w.y), bb[2 * u]);
                                    bb[2 * u + 1] = __ffma2_rn(ee, make_float2(w.z, w.w), bb[2 * u + 1]);
                                }
                            };
                            if constexpr (decltype(N)::value > 0) {
                                // a known count: the values first, so that their latency overlaps, then the sums
                                constexpr int n_c = decltype(N)::value;
                                float ev[n_c];
#pragma unroll
                                for (int j = 0; j < n_c; ++j) ev[j] = value(row + j * BROW);
#pragma unroll
                                for (int j = 0; j < n_c; ++j) add(row + j * BROW, ev[j]);
                                row += n_c * BROW;
                            } else {
                                for (int j = 0; j < n; ++j, row += BROW) add(row, value(row));
                            }
#pragma unroll
                            for (int m = 0; m < NBS; ++m) b[m] = m & 1 ? bb[m / 2].y : bb[m / 2].x;
                        }
                    };
                    R be[NBS], bd[NBS], s[NWS];
                    group(std::integral_constant<int, NE>{}, n_exp, be);
                    group(std::integral_constant<int, ND>{}, nprof - n_exp, bd);
                    combine_groups(be, bd, fr[WF_G], fr[WF_G + 1], edev, s);
                    whitened_add(s, z1, z2, fr, g1, d1, de, h1, he);
                    if (!DBL) star();
                }
                // ---- E, Var and the pixel's weights
                const Light p = DBL ? part_light : light();
                const R a0 = p.a0, a1 = p.a1, K0 = p.K0, K1 = p.K1, L0 = p.L0, L1 = p.L1, k0 = p.k0, k1 = p.k1;
                const R Es = k0 * g0 + k1 * g1;
                if (alone) {
                    if constexpr (DBL) {
                        double em0, em1, es;
                        moment_ratios64(sT, em0, em1);
                        source_ev64(sT, em0, em1, g0, g1, es, V);
                        E += es;
                    } else {
                        // Var_s in the form that does not cancel (k_contrib's)
                        const float f0 = K0 * g0, f1 = K1 * g1;
                        const float em0 = sT[H_EL20] / (sT[H_EL0] * sT[H_EL0]) - 1.f;
                        const float em1 = sT[H_EL21] / (sT[H_EL1] * sT[H_EL1]) - 1.f;
                        V = a0 * f0 * f0 * (em0 + (1.f - a0)) + a1 * f1 * f1 * (em1 + (1.f - a1)) -
                            2.f * a0 * a1 * f0 * f1;
                        E += Es;
                    }
                }
                const R iE = (R)1 / E, iE2 = iE * iE;
                const R cE = x * (iE + V * iE2 * iE) - (R)1;
                const R cV = (R)-0.5 * x * iE2;
                const R hEV = x * iE2 * iE;
                out[0] = x * (lgh(E) - (R)0.5 * V * iE2) - E;
                // ---- assemble the pixel's z-derivatives (entries known to be zero are left out: a
                // product with a constant 0 would be computed)
                const R w1 = cE - (R)2 * cV * Es, w2 = cV;
                // gradient of g_1 over (mx, my, e_dev, Gxx, Gxy, Gyy); g_0's is (d0[0], d0[1], 0, 0, 0, 0)
                const R dg1[6] = {d1[0], d1[1], de, d1[2], d1[3], d1[4]};
                // e = dE_s/dz (0 for Q_i), v2 = dE2_s/dz
                R e[NZ], v2[NZ];
                e[Z_A0] = K0 * g0;
                e[Z_A1] = K1 * g1;
                v2[Z_A0] = v2[Z_Q0] = L0 * g0 * g0;
                v2[Z_A1] = v2[Z_Q1] = L1 * g1 * g1;
                // L_i g_i twice, and with a_i
                const R m0 = (R)2 * L0 * g0, m1 = (R)2 * L1 * g1, n0 = a0 * m0, n1 = a1 * m1;
#pragma unroll
                for (int z = 0; z < 6; ++z) {
                    e[Z_MX + z] = k1 * dg1[z];
                    v2[Z_MX + z] = n1 * dg1[z];
                    if (z < 2) {
                        e[Z_MX + z] += k0 * d0[z];
                        v2[Z_MX + z] += n0 * d0[z];
                    }
                }
                auto has_e = [](int z) { return z != Z_Q0 && z != Z_Q1; };
                // gradient, and the outer-product part of the Hessian: with v = v2 - 2 E_s e,
                //   (h_EE - 2 c_V) e e' + h_EV (e v' + v e') = e p' + p e',
                //   p = (h_EE / 2 - c_V - 2 h_EV E_s) e + h_EV v2,  h_EE / 2 - c_V = -3 h_EV Var / (2 E)
                const R c1 = -hEV * ((R)1.5 * V * iE + (R)2 * Es);
                R pv[NZ];
#pragma unroll
                for (int z = 0; z < NZ; ++z) {
                    if (!has_e(z)) {
                        out[1 + z] = w2 * v2[z];
                        pv[z] = hEV * v2[z];
                    } else {
                        out[1 + z] = w1 * e[z] + w2 * v2[z];
                        pv[z] = c1 * e[z] + hEV * v2[z];
                    }
                }
                R* H = out + 1 + NZ;
#pragma unroll
                for (int a = 0; a < NZ; ++a)
#pragma unroll
                    for (int b = a; b < NZ; ++b) {
                        R h = 0;
                        if (has_e(a) && has_e(b)) h = e[a] * pv[b] + pv[a] * e[b];
                        else if (has_e(a)) h = e[a] * pv[b];
                        else if (has_e(b)) h = pv[a] * e[b];
                        H[sym<NZ>(a, b)] = h;
                    }
                // second-derivative part  w1 DE + w2 DE2
                const R r0 = w2 * m0, r1 = w2 * m1, s0 = w1 * K0 + r0, s1 = w1 * K1 + r1;
                const R u0 = a0 * s0, u1 = a1 * s1;
                const R b0 = (R)2 * w2 * p.l0, b1 = (R)2 * w2 * p.l1;
                R bd1[6];
#pragma unroll
                for (int z = 0; z < 6; ++z) {
                    H[sym<NZ>(Z_A1, Z_MX + z)] += s1 * dg1[z];
                    H[sym<NZ>(Z_Q1, Z_MX + z)] += r1 * dg1[z];
                    if (z < 2) {
                        H[sym<NZ>(Z_A0, Z_MX + z)] += s0 * d0[z];
                        H[sym<NZ>(Z_Q0, Z_MX + z)] += r0 * d0[z];
                    }
                    bd1[z] = b1 * dg1[z];
                }
                // mean / shape block: u0 d2g0 + b0 dg0 dg0' + u1 d2g1 + b1 dg1 dg1', d2g1 over
                // (mx, my, e_dev, Gxx, Gxy, Gyy) from h1 (packed without e_dev) and he (the e_dev row;
                // its diagonal is zero)
                const int zmap[5] = {0, 1, 3, 4, 5};   // position without e_dev -> position among the six
                {
                    int c = 0;
#pragma unroll
                    for (int a = 0; a < 5; ++a) {
                        H[sym<NZ>(Z_ED, Z_MX + zmap[a])] += u1 * he[a];
#pragma unroll
                        for (int b = a; b < 5; ++b, ++c) H[sym<NZ>(Z_MX + zmap[a], Z_MX + zmap[b])] += u1 * h1[c];
                    }
                }
#pragma unroll
                for (int a = 0; a < 6; ++a)
#pragma unroll
                    for (int b = a; b < 6; ++b) {
                        R v = bd1[a] * dg1[b];
                        if (a < 2 && b < 2) v += b0 * d0[a] * d0[b] + u0 * h0[a + b];
                        H[sym<NZ>(Z_MX + a, Z_MX + b)] += v;
                    }
            }
            // ---- the 32 pixels' sums in R (a reduce-scatter), added to the part's in FP64
            warp_reduce_scatter(out, lane);
            sums[2 * lane] += (double)out[0];
            sums[2 * lane + 1] += (double)out[1];
            if (lane < HV - 64) sums[64 + lane] += (double)(lane == 0 ? out[64] : out[65]);
        }
        __syncwarp();
        double* rec = a.part + (size_t)(cur - n_term) * HV;
        for (int i = lane; i < HV; i += 32) rec[i] = sums[i];
        next = __shfl_sync(0xffffffffu, claim, 0);
        next_patch = patch_of(next);
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // the last CTA resets the queue for the next launch
        __threadfence();
        if (atomicAdd(a.queue + 1, 1) == (int)gridDim.x - 1) {
            a.queue[0] = 0;
            a.queue[1] = 0;
            __threadfence();
        }
    }
}

// ---------------------------------------------------------------------------------
// per-source chain rule

// The chain rule goes from z to twelve variables w per (source, patch) that stand in the
// places of y: a_0, a_1, then per type i the mean m_i and variance v_i of the log brightness
// in the patch's band (places Y_EL0, Y_EL20, Y_EL1, Y_EL21), u_0, u_1, e_dev, and e_axis,
// e_angle, e_scale.  A parameter theta_j < P_K enters exactly one of them, with a factor of
// the band alone that is -1, 0 or 1, so the w-Hessians of a band's patches are added first
// and spread over the 28 x 28 block once per source by additions.
__device__ __forceinline__ int w_of_param(int j) {
    if (j < 2) return Y_MX + j;
    if (j == P_EDEV) return Y_EDEV;
    if (j <= P_SCALE) return Y_GXX + j - P_AXIS;
    if (j >= P_A) return j == P_A ? Y_A0 : Y_A1;
    const bool var = (j >= P_R2 && j < P_C1) || j >= P_C2;
    const int i = j < P_R2 ? j - P_R1 : j < P_C1 ? j - P_R2 : j < P_C2 ? (j - P_C1) >> 2 : (j - P_C2) >> 2;
    return (i == 0 ? Y_EL0 : Y_EL1) + (var ? 1 : 0);
}
__device__ __forceinline__ int w_factor(int band, int j) {
    if (j < P_C1 || j >= P_A) return 1;
    const int c = (j - P_C1) & 3, ref = 2;   // color_beta as an integer
    const int beta = band < ref ? (c >= band && c < ref ? -1 : 0) : band > ref ? (c >= ref && c < band ? 1 : 0) : 0;
    return j < P_C2 ? beta : beta * beta;
}

// One CTA per source, two warps per band, which add the parts of a patch half and half and take
// turns to map the 66 sums to w (X = H_z J, then J' X, J at most three entries per column) and
// to add the result to the warp's shared accumulator; then the block is spread and added to the
// -KL terms that source_terms left in hess_out.
// Latency-bound, so the patches of a source run side by side and a patch costs about 50 FP64
// instructions; per-patch loops over the 44 x 44 entries with the KL and its Hessian in the
// same CTA took 119 us for 500 sources and 49 us for 64, this 36 and 26 (alone, cold caches).
// barrier of a band's two warps
__device__ __forceinline__ void pair_barrier(int band) { asm volatile("bar.sync %0, 64;" ::"r"(band + 1) : "memory"); }

constexpr int FH_SPLIT = 2, FH_WARPS = 5 * FH_SPLIT, FH_THREADS = 32 * FH_WARPS;
constexpr int NPIX = P_K;                         // parameters that the pixels depend on
constexpr int NPIXH = NPIX * (NPIX + 1) / 2;
__device__ const PackedTriangle<NPIX> g_pix = packed_triangle<NPIX>();
__device__ const PackedTriangle<NY> g_ypk = packed_triangle<NY>();

__global__ void __launch_bounds__(FH_THREADS, 4)
k_finalize_hess(int n_src, int hchunk, const PatchGeo* __restrict__ geo, const int32_t* __restrict__ patch_off,
                const ImgMeta* __restrict__ img, const float* __restrict__ tbl32, const double* __restrict__ part,
                const double* __restrict__ hsrc, double* __restrict__ local_out, double* __restrict__ grad_out,
                double* __restrict__ hess_out, const int32_t* __restrict__ src_active) {
    const int s = blockIdx.x;
    if (s >= n_src || (src_active && !src_active[s])) return;
    constexpr int NACC = 1 + NY + NYH;
    __shared__ double acc[FH_WARPS][NACC];   // ll, d/dw, d2/dw2 (packed) of the warp's patches
    __shared__ double rec[HREC];
    __shared__ double sy[FH_WARPS][HV];      // the patch's sums over z
    __shared__ double sx[FH_WARPS][NZ][NY];  // H_z J
    __shared__ double sj[FH_WARPS][NY][3];   // J: column w's entries ...
    __shared__ uint8_t si[FH_WARPS][NY][3];  // ... and their z
    __shared__ double sg[FH_WARPS][36];      // dG, d2G of the patch
    __shared__ double sr[FH_WARPS][4];       // r_K, r_L of each type (below)
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int band = warp % 5, half = warp / 5;
    for (int i = t; i < HREC; i += FH_THREADS) rec[i] = hsrc[(size_t)HREC * s + i];
    for (int i = lane; i < NACC; i += 32) acc[warp][i] = 0.0;
    __syncthreads();
    const int p0 = patch_off[s], p1 = patch_off[s + 1];
    int seen = 0;   // patches of this band so far
    for (int pb = p0; pb < p1; pb += 32) {
        const int pl = pb + lane;
        unsigned mine = __ballot_sync(0xffffffffu, pl < p1 && img[geo[pl < p1 ? pl : p0].img].band == band);
        for (; mine; mine &= mine - 1) {
            const int p = pb + __ffs(mine) - 1;
            const PatchGeo g = geo[p];
            const double* A = img[g.img].A;
            float el = 0.f, el_iota = 0.f;   // FP32: the moments that the pass had (lanes 0 .. 3)
            if (tbl32 && lane < 4) {
                el = tbl32[(size_t)p * TBL_STRIDE + H_EL0 + lane];
                el_iota = tbl32[(size_t)p * TBL_STRIDE + H_IOTA];
            }
            // the patch's parts, each warp of the band half of them in order, loaded four at a
            // time before any is added; the two sums meet in the warp whose turn the patch is
            double v[3] = {0.0, 0.0, 0.0};
            const int np = (g.w * g.h + hchunk - 1) / hchunk, mid = g.hpart0 + (np + 1) / 2;
            const int i1 = half ? g.hpart0 + np : mid;
            for (int i0 = half ? mid : g.hpart0; i0 < i1; i0 += 4) {
                double x[4][3];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        x[u][c] = i0 + u < i1 && lane + 32 * c < HV
                                      ? part[(size_t)(i0 + u) * HV + lane + 32 * c] : 0.0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i0 + u < i1)
#pragma unroll
                        for (int c = 0; c < 3; ++c) v[c] += x[u][c];
            }
            const bool turn = (seen++ & 1) == half;
            if (!turn)
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    if (lane + 32 * c < HV) sy[warp][lane + 32 * c] = v[c];
            pair_barrier(band);
            if (turn)
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    if (lane + 32 * c < HV) v[c] += sy[band + 5 * (1 - half)][lane + 32 * c];
            pair_barrier(band);   // the other warp may write its sums of the next patch
            if (!turn) continue;
            // the shape derivatives through the patch's map
            for (int i = lane; i < 36; i += 32)
                sg[warp][i] = a_transform(A, rec + HR_DW + 3 * (i / 3), i % 3);
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (lane + 32 * c < HV) sy[warp][lane + 32 * c] = v[c];
            __syncwarp();
            // K_0, L_0, K_1, L_1 over the ones that the FP32 pass had, for the rows of the log brightness.
            // (Not for those of a_i: the pass's rounding is in its E_s and Var_s too, and with
            // the FP64 moments against these the a_i's gradient and Hessian entries were off by
            // 1.3 to 2.3 times as much against 64 bits.)
            if (lane < 4) {
                double r = 1.0;
                if (tbl32) {
                    const double iota = img[g.img].iota;
                    const double k = (lane & 1 ? iota * iota : iota) * rec[HR_MOM + 4 * band + lane];
                    const float pass = (lane & 1 ? el_iota * el_iota : el_iota) * el;
                    const float off = (float)(k - (double)pass) / pass;
                    if (fabsf(off) < 1e-3f) r += (double)off;   // (rounding, not a denormal or an overflow)
                }
                sr[warp][lane] = r;
            }
            __syncwarp();
            const double* Gz = sy[warp] + 1;
            const double* Hz = sy[warp] + 1 + NZ;
            if (lane < NY) {
                const int w = lane;
                int z0 = Z_ED, z1 = 0, z2 = 0;
                double c0 = 1.0, c1 = 0.0, c2 = 0.0;
                if (w <= Y_EL21) {
                    // A_i and Q_i over a_i, m_i, v_i: A = a r_K e^{dm + dv/2}, A + Q = a r_L e^{2 dm + 2 dv}
                    const int i = w == Y_A1 || w >= Y_EL1;
                    z0 = Z_A0 + i;
                    z1 = Z_Q0 + i;
                    if (w >= Y_EL0) {
                        const double f = (w - Y_EL0) & 1 ? 0.5 : 1.0;
                        c0 = f * sr[warp][2 * i] * rec[HR_A + i];
                        c1 = 2.0 * sr[warp][2 * i + 1] * rec[HR_A + i] - c0;
                    }
                } else if (w == Y_MX || w == Y_MY) {
                    z0 = Z_MX;
                    z1 = Z_MY;
                    c0 = A[w - Y_MX];
                    c1 = A[2 + w - Y_MX];
                } else if (w >= Y_GXX) {
                    const double* d = sg[warp] + 3 * (w - Y_GXX);
                    z0 = Z_GXX; z1 = Z_GXX + 1; z2 = Z_GXX + 2;
                    c0 = d[0]; c1 = d[1]; c2 = d[2];
                }
                sj[warp][w][0] = c0; sj[warp][w][1] = c1; sj[warp][w][2] = c2;
                si[warp][w][0] = (uint8_t)z0; si[warp][w][1] = (uint8_t)z1; si[warp][w][2] = (uint8_t)z2;
                acc[warp][1 + w] += c0 * Gz[z0] + c1 * Gz[z1] + c2 * Gz[z2];
            }
            if (lane == 0) acc[warp][0] += sy[warp][0];
            __syncwarp();
            for (int i = lane; i < NZ * NY; i += 32) {
                const int z = i / NY, w = i % NY;
                double x = 0.0;
#pragma unroll
                for (int e = 0; e < 3; ++e) x += Hz[sym<NZ>(z, si[warp][w][e])] * sj[warp][w][e];
                sx[warp][z][w] = x;
            }
            __syncwarp();
            for (int i = lane; i < NYH; i += 32) {
                const int b = g_ypk.v[i] >> 8, a = g_ypk.v[i] & 255;   // a <= b
                double h = 0.0;
#pragma unroll
                for (int e = 0; e < 3; ++e) h += sj[warp][a][e] * sx[warp][si[warp][a][e]][b];
                // second derivatives of z over w: A = a r_K e^{dm + dv/2}, A + Q = a r_L e^{2 dm + 2 dv}, and G
                const int ia = a == Y_A1 || a >= Y_EL1, ib = b == Y_A1 || b >= Y_EL1;
                if (b <= Y_EL21 && b >= Y_EL0 && ia == ib) {
                    // K d/dk and L d/dq
                    const double Gk = (Gz[Z_A0 + ia] - Gz[Z_Q0 + ia]) * sr[warp][2 * ia];
                    const double Gq = Gz[Z_Q0 + ia] * sr[warp][2 * ia + 1];
                    const double fb = (b - Y_EL0) & 1 ? 0.5 : 1.0;
                    if (a >= Y_EL0) {
                        const double fa = (a - Y_EL0) & 1 ? 0.5 : 1.0;
                        h += rec[HR_A + ia] * (fa * fb * Gk + 4.0 * Gq);
                    } else {
                        h += fb * Gk + 2.0 * Gq;
                    }
                } else if (a >= Y_GXX) {
                    const double* d = sg[warp] + 9 + 9 * (a - Y_GXX) + 3 * (b - Y_GXX);
                    h += Gz[Z_GXX] * d[0] + Gz[Z_GXX + 1] * d[1] + Gz[Z_GXX + 2] * d[2];
                }
                acc[warp][1 + NY + yh_index(a, b)] += h;
            }
            __syncwarp();
        }
    }
    __syncthreads();
    // the band's warps together, in order
    for (int i = t; i < 5 * NACC; i += FH_THREADS)
#pragma unroll
        for (int h = 1; h < FH_SPLIT; ++h) acc[i / NACC][i % NACC] += acc[i / NACC + 5 * h][i % NACC];
    __syncthreads();
    auto band_sum = [&](int col, int i, int j) {
        double h = 0.0;
#pragma unroll
        for (int b = 0; b < 5; ++b) {
            const int f = w_factor(b, i) * w_factor(b, j);
            if (f != 0) h += f > 0 ? acc[b][col] : -acc[b][col];
        }
        return h;
    };
    double* Ho = hess_out + (size_t)NP * NP * s;
    for (int q = t; q < NPIXH; q += FH_THREADS) {
        const int i = g_pix.v[q] >> 8, j = g_pix.v[q] & 255;   // j <= i
        const int wi = w_of_param(i), wj = w_of_param(j);
        const double h = Ho[i * NP + j] + band_sum(1 + NY + sym<NY>(wi, wj), i, j);
        Ho[i * NP + j] = h;
        if (i != j) Ho[j * NP + i] = h;
    }
    if (t < NP && grad_out)
        grad_out[(size_t)NP * s + t] =
            (t < NPIX ? band_sum(1 + w_of_param(t), t, P_U) : 0.0) - rec[HR_KLG + t];
    if (t == 0 && local_out) {
        double l = 0.0;
        for (int b = 0; b < 5; ++b) l += acc[b][0];
        local_out[s] = l - rec[HR_KL];
    }
}

template <class R>
static cudaError_t hess_pixels(const DevProblem& P, const R* tbl, const double* d_theta, double* d_hess,
                               cudaStream_t st) {
    HessArgs<R> a{};
    a.parts = P.hitems;
    a.n_part = P.n_hitem;
    a.img = P.img;
    a.geo = P.geo;
    a.n_comp = P.npsf_max * P.nprof;
    a.nprof = P.nprof;
    a.n_exp = P.model_ne;
    a.pixels = P.pixels;
    a.sky_map = P.sky_map;
    a.tbl = tbl;
    a.hframe = (const float*)P.tbl64;
    a.single = P.single;
    a.emap = (const R*)P.emap;
    a.vmap = (const R*)P.vmap;
    a.part = P.hpart;
    a.src_active = P.src_active;
    a.queue = P.hqueue;
    a.src = SourceTerms{P.n_src, d_theta, P.model, P.hsrc, P.kl, d_hess, P.status};
    // resident CTAs per SM: the registers allow 4 (FP32) or 2, the shared memory (228 KB, 1 KB of
    // it the system's per CTA) perhaps fewer
    const int bytes = HessLay<R>(a.n_comp).bytes();
    const int per_sm = std::max(1, std::min(sizeof(R) == 8 ? 2 : 4, 228 * 1024 / (bytes + 1024)));
    const int64_t tasks = 2LL * P.n_src + P.n_hitem;
    const int grid = (int)std::min<int64_t>((tasks + HESS_WARPS - 1) / HESS_WARPS, (int64_t)per_sm * sm_count());
    if (grid == 0) return cudaSuccess;
    auto* fn = k_hess<R, 0, 0>;
    if constexpr (sizeof(R) == 4)
        if (P.model_ne == 6 && P.model_nd == 8) fn = k_hess<R, 6, 8>;
    fn<<<grid, 32 * HESS_WARPS, bytes, st>>>(a);
    return cudaGetLastError();
}

// shared-memory limits of the Hessian kernels on the current device, set at problem
// creation (outside any stream capture)
cudaError_t prime_hess_kernels() {
    constexpr int most = MAXPSF * MAXPROF;
    cudaError_t e = cudaSuccess;
    for (auto* fn : {k_hess<float, 0, 0>, k_hess<float, 6, 8>})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, HessLay<float>(most).bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_hess<double, 0, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 HessLay<double>(most).bytes());
    return e;
}

cudaError_t launch_hess_pixels(const DevProblem& P, int precision, const double* d_theta, double* d_hess,
                               cudaStream_t st) {
    return precision == CELESTE_FP64 ? hess_pixels<double>(P, P.tbl64, d_theta, d_hess, st)
                                     : hess_pixels<float>(P, P.tbl32, d_theta, d_hess, st);
}

cudaError_t launch_finalize_hess(const DevProblem& P, int precision, double* d_local, double* d_grad, double* d_hess,
                                 cudaStream_t st) {
    if (P.n_src == 0) return cudaSuccess;
    const float* tbl32 = precision == CELESTE_FP64 ? nullptr : P.tbl32;
    k_finalize_hess<<<P.n_src, FH_THREADS, 0, st>>>(P.n_src, P.hchunk, P.geo, P.patch_off, P.img, tbl32, P.hpart, P.hsrc,
                                                    d_local, d_grad, d_hess, P.src_active);
    return cudaGetLastError();
}

}  // namespace cel
