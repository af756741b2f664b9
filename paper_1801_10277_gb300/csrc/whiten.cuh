// The galaxy components of a PSF component in the frame that whitens it: the frames, the
// coefficient rows and the sums they serve.  Host-callable for tests.
#pragma once

#include <math.h>

#include "internal.cuh"

namespace cel {

constexpr double LOG2E_W = 1.4426950408889634;   // log2(e)

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
constexpr int WROW = 40;   // a full row (whiten_row): exponent coefficients of z1^2, z2^2, constant; 35 weights; pad
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
__host__ __device__ inline void whiten_frame(const float* sT, int k, float* fr) {
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

// The 35 sums' weights one by one, the plain form that the host test of the frame sums (no kernel
// does: they take the 19 of base_row): lam1^(deg - i) lam2^i, i = 0 .. deg, times w
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

// ... and the row of galaxy component (k, j): exponent in z and the 35 monomial weights
__host__ __device__ inline void whiten_row(const float* G, const float* fr, float* row) {
    const float nu = G[9], w = G[7], dw = G[8];
    const float l1 = 1.f / (1.f + nu * fr[WF_G]), l2 = 1.f / (1.f + nu * fr[WF_G + 1]);
    row[0] = -0.5f * (float)LOG2E_W * l1;
    row[1] = -0.5f * (float)LOG2E_W * l2;
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

// the kernel's row: three exponent coefficients (given) and the 19 weights at weight w, each
// degree from the one below
template <class R>
__host__ __device__ __forceinline__ void base_row(R w, R nu, R l1, R l2, R* c) {
    const R w1 = w * l1, w2 = w * l2;
    c[BS_LL] = w1 * l1;
    c[BS_LL + 1] = w1 * l2;
    c[BS_LL + 2] = w2 * l2;
    R n[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        n[i] = nu * c[BS_LL + i];
        c[BS_C + i] = n[i] * l1;
        c[BS_D2 + i] = nu * n[i];
    }
    c[BS_C + 3] = n[2] * l2;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        c[BS_D3 + i] = nu * c[BS_C + i];
        c[BS_D4 + i] = c[BS_D3 + i] * l1;
    }
    c[BS_D4 + 4] = c[BS_D3 + 3] * l2;
}

// The FP32 Hessian pass's frames of a patch (MAXPSF of them) take the place of the FP64 tables,
// which an FP32 evaluation does not use.
constexpr int HF_STRIDE = MAXPSF * WFR;   // floats per patch
static_assert(HF_STRIDE * sizeof(float) <= TBL_STRIDE * sizeof(double), "in the place of a table");

}  // namespace cel
