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
// The pixel terms depend on theta through ten variables z of the (source, patch): with
// k_i = a_i iota E[l_i] and q_i = a_i iota^2 E[l_i^2] (i = star, galaxy),
//   E_s = k_0 g_0 + k_1 g_1,  E2_s = q_0 g_0^2 + q_1 g_1^2,  Var_s = E2_s - E_s^2,
// z = (k_0, k_1, q_0, q_1, the mean, e_dev, G).  (The twelve y of the gradient passes hold
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

#include <type_traits>

#include "fp64_profile.cuh"
#include "internal.cuh"
#include "source_math.cuh"

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

constexpr double LOG2E_H = 1.4426950408889634;   // log2(e)

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

// ---- The galaxy components in the frame that whitens PSF component k.
// T_k maps a pixel offset d to z = T_k d with T_k Sigma_k T_k' = I and T_k G T_k' =
// diag(g1, g2), so component j's precision is T_k' diag(lam1, lam2) T_k with
// lam_a = 1 / (1 + nu_j g_a).  With r = lam z and E~ = T_k E T_k', every derivative of
// N_kj over (mu, G) is N_kj times T_k' (a polynomial in z) T_k:
//   d/dmu: r;   d/dG[E]: (nu/2)(r' E~ r - tr(lam E~));   d2/dmu2: r r' - lam;
//   d2/dmu dG[E]: r d/dG[E] - nu lam E~ r;
//   d2/dG[E] dG[F]: d/dG[E] d/dG[F] - nu^2 r' E~ lam F~ r + (nu^2/2) tr(lam E~ lam F~).
// A pixel therefore needs, per k, 35 sums over j of N_kj (or of its e_dev derivative)
// times a monomial in (nu, lam1, lam2); the z-polynomials and the maps back to the
// pixel frame are applied once per (pixel, k) instead of once per component.
// Sums (monomial lam1^(deg - i) lam2^i at offset i):
constexpr int WS_N = 0,    // N
              WS_L = 1,    // N lam            (deg 1)
              WS_LL = 3,   // N lam lam        (deg 2)
              WS_B = 6,    // N nu lam         (deg 1)
              WS_A = 8,    // N nu lam lam     (deg 2)
              WS_C = 11,   // N nu lam^3       (deg 3)
              WS_D2 = 15,  // N nu^2 lam^2
              WS_D3 = 18,  // N nu^2 lam^3
              WS_D4 = 22,  // N nu^2 lam^4
              WS_NE = 27,  // dN/de_dev
              WS_LE = 28,  // dN/de_dev lam
              WS_BE = 30,  // dN/de_dev nu lam
              WS_AE = 32,  // dN/de_dev nu lam lam
              NWS = 35;
// Of these, with lam_a (1 + nu g_a) = 1, the ones of lower degree follow from 19 (all terms
// positive, so nothing cancels):  A_0 = C_0 + g1 D3_0, A_1 = C_1 + g1 D3_1, A_2 = C_3 + g2 D3_3,
// B = A + g D2, L = LL + g A, N = L_0 + g1 B_0; and the e_dev sums are the difference of the
// dev and the exp components' sums at unit weight.  So the kernel accumulates 19 sums over
// the exp components, then over the dev components, and forms the 35 once per (pixel, k).
constexpr int BS_LL = 0, BS_C = 3, BS_D2 = 7, BS_D3 = 10, BS_D4 = 14, NBS = 19;
constexpr int WROW = 40;   // a full row: exponent coefficients of z1^2, z2^2, constant; 35 weights; pad
constexpr int BROW = 24;   // a kernel row: the exponent's three coefficients, (FP32: a pad,) 19 weights, pad
constexpr int WFR = 16;    // entries per k: T (row-major), K (3 x 3), g1, g2, pad
// K[e][p] = (T E_e T')_p for the pixel-frame shape directions E_e = (xx, xy + yx, yy)
// and the whitened pairs p = (11, 12, 22)
constexpr int WF_K = 4, WF_G = 13;
static_assert(3 + NWS <= WROW && 4 + NBS < BROW && BROW % 4 == 0 && WFR % 4 == 0 && WF_G + 2 <= WFR,
              "whitened rows are read as 16-byte vectors from a 16-byte aligned array");

__host__ __device__ __forceinline__ int wpa(int p) { return p == 2 ? 1 : 0; }
__host__ __device__ __forceinline__ int wpb(int p) { return p == 0 ? 0 : 1; }

// K of a frame whose T is in place
template <class R>
__host__ __device__ __forceinline__ void whiten_shape_map(R* fr) {
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const R* Ta = fr + 2 * wpa(p);
        const R* Tb = fr + 2 * wpb(p);
        fr[WF_K + 0 * 3 + p] = Ta[0] * Tb[0];
        fr[WF_K + 1 * 3 + p] = Ta[0] * Tb[1] + Ta[1] * Tb[0];
        fr[WF_K + 2 * 3 + p] = Ta[1] * Tb[1];
    }
    fr[15] = 0;
}

// T_k from the Cholesky factor of the component's precision and one Jacobi rotation, in
// FP32 (a few threads per work item, before its pixels: FP64 square roots and divisions
// there would hold every warp of the item at the barrier; host-callable for tests)
__host__ __device__ void whiten_frame(const float* sT, int k, float* fr) {
    const float* S = sT + T_STAR + k * STAR_STRIDE;
    const float pxx = S[4], pxy = S[5], pyy = S[6];
    const float gxx = sT[T_G], gxy = sT[T_G + 1], gyy = sT[T_G + 2];
    // T0 = [[r11, r21], [0, r22]] with T0 Sigma T0' = I (r the lower factor of Sigma^-1)
    const float r11 = sqrtf(pxx), r21 = pxy / r11, r22 = sqrtf(fmaxf(pyy - r21 * r21, 0.f));
    const float u0 = r11 * gxx + r21 * gxy, u1 = r11 * gxy + r21 * gyy;
    const float b11 = u0 * r11 + u1 * r21, b12 = u1 * r22, b22 = r22 * gyy * r22;
    // Q = [[c, s], [-s, c]] with Q B Q' diagonal, B = T0 G T0' (the smaller rotation; an
    // infinite tau gives t = 0)
    float c = 1.f, s = 0.f;
    if (b12 != 0.f) {
        const float tau = (b22 - b11) / (2.f * b12);
        const float t = tau == 0.f ? 1.f : -copysignf(1.f, tau) / (fabsf(tau) + sqrtf(1.f + tau * tau));
        c = 1.f / sqrtf(1.f + t * t);
        s = t * c;
    }
    const float T[2][2] = {{c * r11, c * r21 + s * r22}, {-s * r11, -s * r21 + c * r22}};
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        fr[2 * a] = T[a][0];
        fr[2 * a + 1] = T[a][1];
        const float v0 = T[a][0] * gxx + T[a][1] * gxy, v1 = T[a][0] * gxy + T[a][1] * gyy;
        fr[WF_G + a] = fmaxf(v0 * T[a][0] + v1 * T[a][1], 0.f);
    }
    whiten_shape_map(fr);
}

// lam1^(deg - i) lam2^i, i = 0 .. deg, times w
template <class R>
__host__ __device__ __forceinline__ void monomials(R w, R l1, R l2, int deg, R* c) {
#pragma unroll
    for (int i = 0; i <= deg; ++i) {
        R v = w;
#pragma unroll
        for (int u = 0; u < deg; ++u) v *= u < i ? l2 : l1;
        c[i] = v;
    }
}

// the row of galaxy component (k, j): exponent in z and the 35 monomial weights
__host__ __device__ void whiten_row(const float* G, const float* fr, float* row) {
    const float nu = G[9], w = G[7], dw = G[8];
    const float l1 = 1.f / (1.f + nu * fr[WF_G]), l2 = 1.f / (1.f + nu * fr[WF_G + 1]);
    row[0] = -0.5f * (float)LOG2E_H * l1;
    row[1] = -0.5f * (float)LOG2E_H * l2;
    row[2] = G[3];
    float* c = row + 3;
    c[WS_N] = w;
    c[WS_NE] = dw;
    monomials(w, l1, l2, 1, c + WS_L);
    monomials(w, l1, l2, 2, c + WS_LL);
    monomials(w * nu, l1, l2, 1, c + WS_B);
    monomials(w * nu, l1, l2, 2, c + WS_A);
    monomials(w * nu, l1, l2, 3, c + WS_C);
    monomials(w * nu * nu, l1, l2, 2, c + WS_D2);
    monomials(w * nu * nu, l1, l2, 3, c + WS_D3);
    monomials(w * nu * nu, l1, l2, 4, c + WS_D4);
    monomials(dw, l1, l2, 1, c + WS_LE);
    monomials(dw * nu, l1, l2, 1, c + WS_BE);
    monomials(dw * nu, l1, l2, 2, c + WS_AE);
    row[3 + NWS] = 0.f;
    row[4 + NWS] = 0.f;
}

// the kernel's row: three exponent coefficients (given) and the 19 weights at weight w
template <class R>
__host__ __device__ __forceinline__ void base_row(R w, R nu, R l1, R l2, R* c) {
    monomials(w, l1, l2, 2, c + BS_LL);
    monomials(w * nu, l1, l2, 3, c + BS_C);
    monomials(w * nu * nu, l1, l2, 2, c + BS_D2);
    monomials(w * nu * nu, l1, l2, 3, c + BS_D3);
    monomials(w * nu * nu, l1, l2, 4, c + BS_D4);
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

// ---- The terms of a source that depend on its parameters alone, by the first CTAs of
// k_hess (their FP64 latencies then pass behind the pixel work): the KL value, gradient and
// Hessian, the brightness moments of the five bands and the world-frame shape derivatives.
// hess_out receives -KL'' and zeros; the rest goes to the source's record.
constexpr int HR_KL = 0, HR_KLG = 1, HR_MOM = HR_KLG + NP, HR_DW = HR_MOM + 20, HR_D2W = HR_DW + 9,
              HR_A = HR_D2W + 27;
static_assert(HR_A + 2 <= HREC && HREC % 2 == 0, "the source's record");
constexpr int TERM_SRC = HCHUNK / 64;   // sources per CTA: two warps each

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

// the terms of sources s0 .. s0 + TERM_SRC, one CTA of k_hess; sm: TERM_SRC NP doubles
__device__ __forceinline__ void source_terms(const SourceTerms& a, int s0, const int32_t* __restrict__ src_active,
                                             double* sm) {
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int n = min(TERM_SRC, a.n_src - s0);
    for (int u = 0; u < n; ++u) {
        if (src_active && !src_active[s0 + u]) continue;
        double* H = a.hess + (size_t)NP * NP * (s0 + u);   // the caller's: 8-byte aligned
        for (int i = t; i < NP * NP; i += HCHUNK) H[i] = 0.0;
    }
    for (int i = t; i < n * NP; i += HCHUNK) {
        sm[i] = a.theta[(size_t)NP * s0 + i];
        if (a.status) theta_domain_check(i % NP, sm[i], a.status);
    }
    __syncthreads();
    const int u = warp % TERM_SRC, s = s0 + u;
    if (u >= n || (src_active && !src_active[s])) return;
    const double* th = sm + u * NP;
    double* rec = a.hsrc + (size_t)HREC * s;
    if (warp < TERM_SRC) {
        kl_terms_warp(*a.md, th, rec, a.kl + s, a.hess + (size_t)NP * NP * s);
        return;
    }
    if (lane < 10) band_moments(th, lane >> 1, lane & 1, rec[HR_MOM + 2 * lane], rec[HR_MOM + 2 * lane + 1]);
    if (lane >= 30) rec[HR_A + lane - 30] = th[P_A + lane - 30];
    if (lane == 10) {
        double dW[3][3], d2W[3][3][3];
        shape_w_derivs(th, dW, d2W);
        for (int i = 0; i < 9; ++i) rec[HR_DW + i] = dW[i / 3][i % 3];
        for (int i = 0; i < 27; ++i) rec[HR_D2W + i] = d2W[i / 9][i / 3 % 3][i % 3];
    }
}

// Shared memory of k_hess (bytes): the patch's table (R), per PSF component its frame, the
// component rows and, FP64, the table of 2^x; the warps' sums take the rows' place at the end.
template <class R>
struct HessLay {
    static constexpr int tbl = 0;
    static constexpr int fr = tbl + TBL_STRIDE * (int)sizeof(R);
    static constexpr int rows = fr + MAXPSF * WFR * (int)sizeof(R);
    static constexpr int rows_bytes = MAXPSF * MAXPROF * BROW * (int)sizeof(R);
    static constexpr int red_bytes = (HCHUNK / 32) * HV * 8;
    static constexpr int tab = rows + (rows_bytes > red_bytes ? rows_bytes : red_bytes);
    static constexpr int bytes = tab + (sizeof(R) == 8 ? EX_N * 8 : 0);
    static_assert(fr % 16 == 0 && rows % 16 == 0 && tab % 16 == 0, "16-byte alignment");
};

// Per part of a work item: the sums over its pixels of ll, d ll / d y and d2 ll / dy2.  The mixture in
// the whitened frame (above); FP64 as in fp64_profile.cuh, E and Var of a singly covered
// pixel (single, FP64 only) formed here, those of the others from the maps.
// Bound by the FP32 or the FP64 pipe: 22 / 25 of its instructions per component, where the
// 35 sums accumulated one by one took 38 (FP32: 500 sources, 909,100 source-pixels, 180 ->
// 140 us) and the pixel-frame formulas about 140 (FP64: fp64_profile.cuh has the figures).
template <class R>
__global__ void __launch_bounds__(HCHUNK, sizeof(R) == 8 ? 2 : 4) k_hess(const WorkItem* __restrict__ items,
                                                const PatchGeo* __restrict__ geo,
                                                const ImgMeta* __restrict__ img, int nprof, int n_exp,
                                                const float* __restrict__ pixels,
                                                const float* __restrict__ sky_map,
                                                const R* __restrict__ tbl,
                                                const uint8_t* __restrict__ single,
                                                const R* __restrict__ emap,
                                                const R* __restrict__ vmap,
                                                double* __restrict__ part,
                                                const int32_t* __restrict__ src_active, SourceTerms src) {
    constexpr bool DBL = std::is_same<R, double>::value;
    using Lay = HessLay<R>;
    extern __shared__ __align__(16) unsigned char smem[];
    R* sT = reinterpret_cast<R*>(smem + Lay::tbl);
    R* frames = reinterpret_cast<R*>(smem + Lay::fr);
    R* rows = reinterpret_cast<R*>(smem + Lay::rows);
    double* tab = reinterpret_cast<double*>(smem + Lay::tab);
    // the first CTAs take the sources' terms that do not depend on the pixels
    const int n_term_cta = (src.n_src + TERM_SRC - 1) / TERM_SRC;
    if ((int)blockIdx.x < n_term_cta) {
        source_terms(src, (int)blockIdx.x * TERM_SRC, src_active, reinterpret_cast<double*>(smem));
        return;
    }
    // one HCHUNK-pixel part of an item
    const int rec = (int)blockIdx.x - n_term_cta, sub = rec % HSPLIT * HCHUNK;
    const WorkItem it = items[rec / HSPLIT];
    const int n_px = it.n - sub;
    if (n_px <= 0) return;
    const PatchGeo g = geo[it.patch];
    if (src_active && !src_active[g.src]) return;
    const ImgMeta& im = img[g.img];
    const int npsf = im.npsf;
    const int t = threadIdx.x;
    {
        const R* gT = tbl + (size_t)it.patch * TBL_STRIDE;
        const int n = T_GAL + npsf * nprof * GAL_STRIDE;
        for (int i = t; i < n; i += blockDim.x) sT[i] = gT[i];
        if constexpr (DBL) load_exp2_table(tab);
        __syncthreads();
    }
    if (t < npsf) {
        if constexpr (DBL) {
            const R* F = sT + T_STAR + t * STAR_STRIDE;
            R* fr = frames + t * WFR;
            for (int i = 0; i < 4; ++i) fr[i] = F[i];
            fr[WF_G] = F[4];
            fr[WF_G + 1] = F[5];
            whiten_shape_map(fr);
        } else {
            whiten_frame(sT, t, frames + t * WFR);
        }
    }
    __syncthreads();
    for (int i = t; i < npsf * nprof; i += blockDim.x) {
        // the exponent's coefficients and the 19 weights at unit e_dev weight
        const R* G = sT + T_GAL + i * GAL_STRIDE;
        const R* fr = frames + (i / nprof) * WFR;
        R* row = rows + i * BROW;
        R l1, l2, w;
        const R nu = G[9];
        if constexpr (DBL) {
            l1 = G[0] * EX_IHALF;
            l2 = G[1] * EX_IHALF;
            w = G[3];
        } else {
            l1 = 1.f / (1.f + nu * fr[WF_G]);
            l2 = 1.f / (1.f + nu * fr[WF_G + 1]);
            w = i % nprof >= n_exp ? G[8] : -G[8];
        }
        row[0] = DBL ? G[0] : (R)(-0.5 * LOG2E_H) * l1;
        row[1] = DBL ? G[1] : (R)(-0.5 * LOG2E_H) * l2;
        row[2] = DBL ? G[2] : G[3];
        constexpr int W0 = DBL ? 3 : 4;   // FP32: the weights on a 16-byte boundary
        base_row(w, nu, l1, l2, row + W0);
        row[W0 + NBS] = 0;
    }
    __syncthreads();
    R out[HV];
#pragma unroll
    for (int i = 0; i < HV; ++i) out[i] = 0;
    if (t < n_px) {
        const int q = it.q0 + sub + t;
        const int yy = q / g.w, xx = q - yy * g.w;
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
            {
                // P d = T' z and P = T' T
                const R* S = sT + T_STAR + k * STAR_STRIDE;
                R n, qx, qy, pxx, pxy, pyy;
                if constexpr (DBL) {
                    n = S[6] * ex2_quad(EX_HALF, z1s, EX_HALF, z2s, (float)EX_HALF, f1, (float)EX_HALF, f2, tab);
                    qx = fr[0] * z1 + fr[2] * z2;
                    qy = fr[1] * z1 + fr[3] * z2;
                    pxx = fr[WF_K] + fr[WF_K + 2];
                    pxy = (R)0.5 * (fr[WF_K + 3] + fr[WF_K + 5]);
                    pyy = fr[WF_K + 6] + fr[WF_K + 8];
                } else {
                    n = S[7] * ex2h(S[0] * (dx * dx) + S[1] * (dx * dy) + S[2] * (dy * dy) + S[3]);
                    qx = S[4] * dx + S[5] * dy;
                    qy = S[5] * dx + S[6] * dy;
                    pxx = S[4];
                    pxy = S[5];
                    pyy = S[6];
                }
                g0 += n;
                d0[0] += n * qx;
                d0[1] += n * qy;
                h0[0] += n * (qx * qx - pxx);
                h0[1] += n * (qx * qy - pxy);
                h0[2] += n * (qy * qy - pyy);
            }
            const R* row = rows + k * nprof * BROW;
            auto group = [&](int n, R (&b)[NBS]) {
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
                    for (int j = 0; j < n; ++j, row += BROW) {
                        float4 cw[BROW / 4];
#pragma unroll
                        for (int u = 0; u < BROW / 4; ++u) cw[u] = reinterpret_cast<const float4*>(row)[u];
                        const float e = ex2h(fmaf(cw[0].x, z1s, fmaf(cw[0].y, z2s, cw[0].z)));
                        const float2 ee = make_float2(e, e);
#pragma unroll
                        for (int m = 0; m < NPR; ++m) {
                            const float4 w = cw[1 + m / 2];
                            bb[m] = __ffma2_rn(ee, m & 1 ? make_float2(w.z, w.w) : make_float2(w.x, w.y), bb[m]);
                        }
                    }
#pragma unroll
                    for (int m = 0; m < NBS; ++m) b[m] = m & 1 ? bb[m / 2].y : bb[m / 2].x;
                }
            };
            R be[NBS], bd[NBS], s[NWS];
            group(n_exp, be);
            group(nprof - n_exp, bd);
            combine_groups(be, bd, fr[WF_G], fr[WF_G + 1], edev, s);
            whitened_add(s, z1, z2, fr, g1, d1, de, h1, he);
        }
        // ---- E, Var and the pixel's weights
        const R iota = sT[H_IOTA], a0 = sT[H_A0], a1 = sT[H_A1];
        const R k0 = a0 * iota * sT[H_EL0], k1 = a1 * iota * sT[H_EL1];
        const R q0 = a0 * iota * iota * sT[H_EL20], q1 = a1 * iota * iota * sT[H_EL21];
        const R Es = k0 * g0 + k1 * g1;
        const int64_t m = im.px_off + (int64_t)(g.y0 + yy) * im.W + (g.x0 + xx);
        const R x = (R)pixels[m];
        R E, V;
        if (DBL && single && single[g.sp_off + q]) {
            if constexpr (DBL) {
                double em0, em1, es;
                moment_ratios64(sT, em0, em1);
                source_ev64(sT, em0, em1, g0, g1, es, V);
                E = (im.has_sky_map ? (double)sky_map[m] : im.sky) + es;
            }
        } else {
            E = emap[m];
            V = vmap[m];
        }
        const R iE = (R)1 / E, iE2 = iE * iE;
        const R cE = x * (iE + V * iE2 * iE) - (R)1;
        const R cV = (R)-0.5 * x * iE2;
        const R hEE = -x * iE2 * ((R)1 + (R)3 * V * iE2);
        const R hEV = x * iE2 * iE;
        out[0] = x * (lgh(E) - (R)0.5 * V * iE2) - E;
        // ---- assemble the pixel's z-derivatives (entries known to be zero are left out: a
        // product with a constant 0 would be computed)
        const R w1 = cE - (R)2 * cV * Es, w2 = cV;
        // gradient of g_1 over (mx, my, e_dev, Gxx, Gxy, Gyy); g_0's is (d0[0], d0[1], 0, 0, 0, 0)
        const R dg1[6] = {d1[0], d1[1], de, d1[2], d1[3], d1[4]};
        // e = dE_s/dz (0 for q), v2 = dE2_s/dz (0 for k)
        R e[NZ], v2[NZ];
        e[Z_K0] = g0;
        e[Z_K1] = g1;
        v2[Z_Q0] = g0 * g0;
        v2[Z_Q1] = g1 * g1;
        const R m0 = (R)2 * q0, m1 = (R)2 * q1, n0 = m0 * g0, n1 = m1 * g1;
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
        auto has_v2 = [](int z) { return z != Z_K0 && z != Z_K1; };
        // gradient, and the outer-product part of the Hessian: with v = v2 - 2 E_s e,
        //   (h_EE - 2 c_V) e e' + h_EV (e v' + v e') = e p' + p e',
        //   p = (h_EE / 2 - c_V - 2 h_EV E_s) e + h_EV v2
        const R c1 = (R)0.5 * hEE - cV - (R)2 * hEV * Es;
        R pv[NZ];
#pragma unroll
        for (int z = 0; z < NZ; ++z) {
            if (!has_e(z)) {
                out[1 + z] = w2 * v2[z];
                pv[z] = hEV * v2[z];
            } else if (!has_v2(z)) {
                out[1 + z] = w1 * e[z];
                pv[z] = c1 * e[z];
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
        const R b0 = w2 * m0, b1 = w2 * m1;
        const R u0 = w1 * k0 + b0 * g0, u1 = w1 * k1 + b1 * g1;
        const R r0 = (R)2 * w2 * g0, r1 = (R)2 * w2 * g1;
        R bd1[6];
#pragma unroll
        for (int z = 0; z < 6; ++z) {
            H[sym<NZ>(Z_K1, Z_MX + z)] += w1 * dg1[z];
            H[sym<NZ>(Z_Q1, Z_MX + z)] += r1 * dg1[z];
            if (z < 2) {
                H[sym<NZ>(Z_K0, Z_MX + z)] += w1 * d0[z];
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
    // ---- CTA reduction: in R within a warp (a reduce-scatter), FP64 across warps
    const int lane = t & 31, warp = t >> 5;
    double(*red)[HV] = reinterpret_cast<double(*)[HV]>(smem + Lay::rows);
    warp_reduce_scatter(out, lane);
    __syncthreads();   // every warp is past its reads of the rows
    red[warp][2 * lane] = (double)out[0];
    red[warp][2 * lane + 1] = (double)out[1];
    if (lane < HV - 64) red[warp][64 + lane] = (double)(lane == 0 ? out[64] : out[65]);
    __syncthreads();
    for (int i = t; i < HV; i += blockDim.x) {
        double s = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w][i];
        part[(size_t)rec * HV + i] = s;
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

// One CTA per source, two warps per band: a warp takes every second patch of its band, adds
// the 66 sums of the patch's records (in order), maps them to w (X = H_z J, then J' X, J at
// most three entries per column) and adds the result to the warp's shared accumulator; then
// the block is spread and added to the -KL terms that source_terms left in hess_out.
// Latency-bound, so the patches of a source run side by side and a patch costs about 50 FP64
// instructions; per-patch loops over the 44 x 44 entries with the KL and its Hessian in the
// same CTA took 119 us for 500 sources and 49 us for 64.
constexpr int FH_SPLIT = 2, FH_WARPS = 5 * FH_SPLIT, FH_THREADS = 32 * FH_WARPS;
constexpr int NPIX = P_K;                         // parameters that the pixels depend on
constexpr int NPIXH = NPIX * (NPIX + 1) / 2;
__device__ const PackedTriangle<NPIX> g_pix = packed_triangle<NPIX>();
__device__ const PackedTriangle<NY> g_ypk = packed_triangle<NY>();

__global__ void __launch_bounds__(FH_THREADS)
k_finalize_hess(int n_src, const PatchGeo* __restrict__ geo, const int32_t* __restrict__ patch_off,
                const ImgMeta* __restrict__ img, const double* __restrict__ part, const double* __restrict__ hsrc,
                double* __restrict__ local_out, double* __restrict__ grad_out, double* __restrict__ hess_out,
                const int32_t* __restrict__ src_active) {
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
            if ((seen++ & (FH_SPLIT - 1)) != half) continue;
            const int p = pb + __ffs(mine) - 1;
            const PatchGeo g = geo[p];
            const double* A = img[g.img].A;
            // the patch's records in order (items cut into HCHUNK-pixel parts, so one per HCHUNK
            // pixels), loaded four at a time before any is added
            double v[3] = {0.0, 0.0, 0.0};
            const int r0 = g.item0 * HSPLIT, i1 = r0 + (g.w * g.h + HCHUNK - 1) / HCHUNK;
            for (int i0 = r0; i0 < i1; i0 += 4) {
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
            // the shape derivatives through the patch's map
            for (int i = lane; i < 36; i += 32)
                sg[warp][i] = a_transform(A, rec + HR_DW + 3 * (i / 3), i % 3);
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (lane + 32 * c < HV) sy[warp][lane + 32 * c] = v[c];
            __syncwarp();
            // iota E[l_i] and iota^2 E[l_i^2] of type i
            const double iota = img[g.img].iota;
            const double* mom = rec + HR_MOM + 4 * band;
            const double m[4] = {iota * mom[0], iota * iota * mom[1], iota * mom[2], iota * iota * mom[3]};
            const double* Gz = sy[warp] + 1;
            const double* Hz = sy[warp] + 1 + NZ;
            if (lane < NY) {
                const int w = lane;
                int z0 = Z_ED, z1 = 0, z2 = 0;
                double c0 = 1.0, c1 = 0.0, c2 = 0.0;
                if (w <= Y_EL21) {
                    // k_i = a_i iota E[l_i], q_i = a_i iota^2 E[l_i^2] over a_i, m_i, v_i
                    const int i = w == Y_A1 || w >= Y_EL1;
                    z0 = Z_K0 + i;
                    z1 = Z_Q0 + i;
                    c0 = i ? m[2] : m[0];
                    c1 = i ? m[3] : m[1];
                    if (w >= Y_EL0) {
                        c0 *= rec[HR_A + i] * ((w - Y_EL0) & 1 ? 0.5 : 1.0);
                        c1 *= 2.0 * rec[HR_A + i];
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
                // second derivatives of z over w: k = a iota e^{m + v/2}, q = a iota^2 e^{2m + 2v}, and G
                const int ia = a == Y_A1 || a >= Y_EL1, ib = b == Y_A1 || b >= Y_EL1;
                if (b <= Y_EL21 && b >= Y_EL0 && ia == ib) {
                    const double Gk = Gz[Z_K0 + ia] * (ia ? m[2] : m[0]), Gq = Gz[Z_Q0 + ia] * (ia ? m[3] : m[1]);
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
    const SourceTerms src{P.n_src, d_theta, P.model, P.hsrc, P.kl, d_hess, P.status};
    const int grid = P.n_item * HSPLIT + (P.n_src + TERM_SRC - 1) / TERM_SRC;
    if (grid == 0) return cudaSuccess;
    k_hess<R><<<grid, HCHUNK, HessLay<R>::bytes, st>>>(P.items, P.geo, P.img, P.nprof, P.model_ne, P.pixels, P.sky_map,
                                                      tbl, P.single, (const R*)P.emap, (const R*)P.vmap, P.item_part,
                                                      P.src_active, src);
    return cudaGetLastError();
}

// shared-memory limits of the Hessian kernels on the current device, set at problem
// creation (outside any stream capture)
cudaError_t prime_hess_kernels() {
    cudaError_t e = cudaFuncSetAttribute(k_hess<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         HessLay<float>::bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_hess<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, HessLay<double>::bytes);
    return e;
}

cudaError_t launch_hess_pixels(const DevProblem& P, int precision, const double* d_theta, double* d_hess,
                               cudaStream_t st) {
    return precision == CELESTE_FP64 ? hess_pixels<double>(P, P.tbl64, d_theta, d_hess, st)
                                     : hess_pixels<float>(P, P.tbl32, d_theta, d_hess, st);
}

cudaError_t launch_finalize_hess(const DevProblem& P, double* d_local, double* d_grad, double* d_hess,
                                 cudaStream_t st) {
    if (P.n_src == 0) return cudaSuccess;
    k_finalize_hess<<<P.n_src, FH_THREADS, 0, st>>>(P.n_src, P.geo, P.patch_off, P.img, P.item_part, P.hsrc, d_local,
                                                    d_grad, d_hess, P.src_active);
    return cudaGetLastError();
}

}  // namespace cel
