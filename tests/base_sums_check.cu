// Host check of the Hessian kernels' galaxy terms as they are computed now: 19 sums over the
// exponential components and 19 over the de Vaucouleurs ones (base_row), the other sums from
// these through lam (1 + nu g) = 1, the groups combined with e_dev (combine_groups), the maps
// back to the pixel frame (whiten_shape_map, whitened_add).  FP32 with the kernel's own frame
// (whiten_frame), FP64 with a frame formed here, both against the pixel-frame formulas of the
// mixture's derivatives over the mean and the shape in long double, and beside the same
// formulas in the type itself.  Random PSF and galaxy covariances (round ones, G = 0, a tiny
// G), numbers of components and e_dev (0 and 1 among them), offsets to three standard deviations.
// Output: "type quantity worst worst_of_the_pixel_frame_formulas".
#include "hess_kernels.cu"

#include <cmath>
#include <cstdio>
#include <random>

using namespace cel;

// value, mean/shape gradient, e_dev derivative, packed 5 x 5 Hessian, e_dev x gradient of
// sum_j w_j N(d; 0, Sigma + nu_j G) (dw_j in the e_dev terms): 27 numbers
template <class F>
static void pixel_frame(F dx, F dy, const double* Sg, const double* Gm, int n, const double* nu, const double* w,
                        const double* dw, long double* out) {
    F o[27] = {};
    for (int j = 0; j < n; ++j) {
        const F v = (F)nu[j], cxx = (F)Sg[0] + v * (F)Gm[0], cxy = (F)Sg[1] + v * (F)Gm[1], cyy = (F)Sg[2] + v * (F)Gm[2];
        const F det = cxx * cyy - cxy * cxy, pxx = cyy / det, pxy = -cxy / det, pyy = cxx / det;
        const F e = std::exp(-(F)0.5 * (pxx * dx * dx + 2 * pxy * dx * dy + pyy * dy * dy)) /
                    ((F)6.283185307179586476925L * std::sqrt(det));
        const F N = (F)w[j] * e, D = (F)dw[j] * e;
        // P and the shape directions E as matrices: xx, xy + yx, yy
        const F P[2][2] = {{pxx, pxy}, {pxy, pyy}}, q[2] = {pxx * dx + pxy * dy, pxy * dx + pyy * dy};
        const F E[3][2][2] = {{{1, 0}, {0, 0}}, {{0, 1}, {1, 0}}, {{0, 0}, {0, 1}}};
        F l[5], L[5][5];   // log-density derivatives
        F PE[3][2][2], Eq[3][2], PEq[3][2];
        for (int a = 0; a < 3; ++a)
            for (int i = 0; i < 2; ++i) {
                Eq[a][i] = E[a][i][0] * q[0] + E[a][i][1] * q[1];
                for (int k = 0; k < 2; ++k) PE[a][i][k] = P[i][0] * E[a][0][k] + P[i][1] * E[a][1][k];
            }
        for (int a = 0; a < 3; ++a)
            for (int i = 0; i < 2; ++i) PEq[a][i] = P[i][0] * Eq[a][0] + P[i][1] * Eq[a][1];
        for (int i = 0; i < 2; ++i) {
            l[i] = q[i];
            for (int k = 0; k < 2; ++k) L[i][k] = -P[i][k];
        }
        for (int a = 0; a < 3; ++a) {
            l[2 + a] = v * (F)0.5 * (q[0] * Eq[a][0] + q[1] * Eq[a][1] - PE[a][0][0] - PE[a][1][1]);
            for (int i = 0; i < 2; ++i) L[i][2 + a] = L[2 + a][i] = -v * PEq[a][i];
            for (int b = 0; b < 3; ++b) {
                F tr = 0, qq = 0;
                for (int i = 0; i < 2; ++i) {
                    qq += Eq[a][i] * PEq[b][i];
                    for (int k = 0; k < 2; ++k) tr += PE[a][i][k] * PE[b][k][i];
                }
                L[2 + a][2 + b] = v * v * ((F)0.5 * tr - qq);
            }
        }
        o[0] += N;
        o[6] += D;
        int c = 7;
        for (int a = 0; a < 5; ++a) {
            o[1 + a] += N * l[a];
            o[22 + a] += D * l[a];
            for (int b = a; b < 5; ++b, ++c) o[c] += N * (l[a] * l[b] + L[a][b]);
        }
    }
    for (int i = 0; i < 27; ++i) out[i] = o[i];
}

// the frame T, g1, g2 of (Sigma, G) in FP64: T = Q' L^-1, one Jacobi rotation
static void frame(const double* S, const double* G, double* fr) {
    const double l11 = sqrt(S[0]), l21 = S[1] / l11, l22 = sqrt(S[2] - l21 * l21);
    const double a = 1 / l11, b = -l21 / (l11 * l22), c = 1 / l22;
    const double bx = b * G[0] + c * G[1], by = b * G[1] + c * G[2];
    const double m11 = a * a * G[0], m12 = a * bx, m22 = bx * b + by * c;
    double cs = 1, sn = 0;
    if (m12 != 0) {
        const double tau = (m22 - m11) / (2 * m12), t = copysign(1.0, tau) / (fabs(tau) + sqrt(1 + tau * tau));
        cs = 1 / sqrt(1 + t * t);
        sn = t * cs;
    }
    const double T[4] = {cs * a - sn * b, -sn * c, sn * a + cs * b, cs * c};
    for (int i = 0; i < 4; ++i) fr[i] = T[i];
    for (int i = 0; i < 2; ++i)
        fr[WF_G + i] = fmax(0.0, T[2 * i] * (T[2 * i] * G[0] + T[2 * i + 1] * G[1]) + T[2 * i + 1] * (T[2 * i] * G[1] + T[2 * i + 1] * G[2]));
    whiten_shape_map(fr);
}

template <class R>
static void kernel_form(const double* Sg, const double* Gm, int n_exp, int n, const double* nu, const double* w, R edev, R dx,
                        R dy, long double* out) {
    const double det = Sg[0] * Sg[2] - Sg[1] * Sg[1];
    R fr[WFR], be[NBS] = {}, bd[NBS] = {}, s[NWS];
    if (sizeof(R) == 4) {
        float sT[TBL_STRIDE] = {}, f[WFR];
        sT[T_STAR + 4] = (float)(Sg[2] / det);
        sT[T_STAR + 5] = (float)(-Sg[1] / det);
        sT[T_STAR + 6] = (float)(Sg[0] / det);
        for (int c = 0; c < 3; ++c) sT[T_G + c] = (float)Gm[c];
        whiten_frame(sT, 0, f);
        for (int i = 0; i < WFR; ++i) fr[i] = (R)f[i];
    } else {
        double f[WFR];
        frame(Sg, Gm, f);
        for (int i = 0; i < WFR; ++i) fr[i] = (R)f[i];
    }
    const R z1 = fr[0] * dx + fr[1] * dy, z2 = fr[2] * dx + fr[3] * dy;
    for (int j = 0; j < n; ++j) {
        const R v = (R)nu[j], l1 = 1 / (1 + v * fr[WF_G]), l2 = 1 / (1 + v * fr[WF_G + 1]);
        // the density at unit e_dev weight, its normaliser from the FP64 covariance as in the tables
        const double cd = (Sg[0] + nu[j] * Gm[0]) * (Sg[2] + nu[j] * Gm[2]) - (Sg[1] + nu[j] * Gm[1]) * (Sg[1] + nu[j] * Gm[1]);
        const R e = std::exp((R)-0.5 * (l1 * z1 * z1 + l2 * z2 * z2)) * (R)(1 / (6.283185307179586 * sqrt(cd)));
        R row[BROW] = {};
        base_row((R)w[j], v, l1, l2, row);
        for (int m = 0; m < NBS; ++m) (j < n_exp ? be : bd)[m] += e * row[m];
    }
    combine_groups(be, bd, fr[WF_G], fr[WF_G + 1], edev, s);
    R g1 = 0, d1[5] = {}, de = 0, h1[15] = {}, he[5] = {};
    whitened_add(s, z1, z2, fr, g1, d1, de, h1, he);
    out[0] = g1;
    out[6] = de;
    for (int i = 0; i < 5; ++i) {
        out[1 + i] = d1[i];
        out[22 + i] = he[i];
    }
    for (int i = 0; i < 15; ++i) out[7 + i] = h1[i];
}

template <class R>
static void run(const char* type) {
    std::mt19937 rng(5);
    std::normal_distribution<double> N01;
    std::uniform_real_distribution<double> U01(0, 1);
    const char* name[5] = {"value", "gradient", "e_dev", "hessian", "e_dev_gradient"};
    const int lo[5] = {0, 1, 6, 7, 22}, hi[5] = {1, 6, 7, 22, 27};
    long double worst[5] = {}, formulas[5] = {};
    for (int trial = 0; trial < 6000; ++trial) {
        const double a0 = N01(rng), a1 = N01(rng), a2 = N01(rng), a3 = N01(rng), sc = 0.1 + 5 * U01(rng);
        double Sg[3] = {a0 * a0 + a1 * a1 + 0.5, a0 * a2 + a1 * a3, a2 * a2 + a3 * a3 + 0.5};
        const double b0 = N01(rng) * sc, b1 = N01(rng) * sc, b2 = N01(rng) * sc, b3 = N01(rng) * sc;
        double Gm[3] = {b0 * b0 + b1 * b1, b0 * b2 + b1 * b3, b2 * b2 + b3 * b3};
        if (trial % 5 == 0) {   // round galaxy, round PSF: no preferred axes
            Gm[0] = Gm[2] = 2.0;
            Sg[0] = Sg[2] = 1.3;
            Gm[1] = Sg[1] = 0.0;
        }
        if (trial % 5 == 1) Gm[0] = Gm[1] = Gm[2] = 0.0;   // a point source
        if (trial % 5 == 2)
            for (double& g : Gm) g *= 1e-6;
        const int n_exp = 1 + (int)(8 * U01(rng)), n = n_exp + 1 + (int)(8 * U01(rng));
        const double edev = trial % 7 == 0 ? 0.0 : trial % 7 == 1 ? 1.0 : (double)(float)U01(rng);
        double nu[16], u[16], w[16], dw[16], dwa[16];
        for (int j = 0; j < n; ++j) {
            nu[j] = 0.02 + 4 * U01(rng);
            u[j] = 0.05 + U01(rng);
            w[j] = u[j] * (j < n_exp ? 1 - edev : edev);
            dw[j] = j < n_exp ? -u[j] : u[j];
            dwa[j] = u[j];
        }
        const double r = 3.0 * U01(rng) * sqrt(Sg[0] + Sg[2] + 4 * (Gm[0] + Gm[2])), ang = 6.283185307179586 * U01(rng);
        const float dx = (float)(r * cos(ang)), dy = (float)(r * sin(ang));
        long double got[27], ref[27], scale_e[27], same[27];
        kernel_form<R>(Sg, Gm, n_exp, n, nu, u, (R)edev, (R)dx, (R)dy, got);
        pixel_frame<long double>(dx, dy, Sg, Gm, n, nu, w, dw, ref);
        pixel_frame<R>((R)dx, (R)dy, Sg, Gm, n, nu, w, dw, same);
        pixel_frame<long double>(dx, dy, Sg, Gm, n, nu, w, dwa, scale_e);   // the e_dev sums mix signs
        for (int g = 0; g < 5; ++g) {
            long double scale = 0, err = 0, err_f = 0;
            for (int i = lo[g]; i < hi[g]; ++i) {
                scale = std::fmax(scale, std::fabs(ref[i]));
                if (g == 2 || g == 4) scale = std::fmax(scale, std::fabs(scale_e[i]));
                err = std::fmax(err, std::fabs(got[i] - ref[i]));
                err_f = std::fmax(err_f, std::fabs(same[i] - ref[i]));
            }
            if (scale < 1e-30L) continue;   // FP32 subnormal range
            worst[g] = std::fmax(worst[g], err / scale);
            formulas[g] = std::fmax(formulas[g], err_f / scale);
        }
    }
    for (int g = 0; g < 5; ++g) printf("%s %s %.6Le %.6Le\n", type, name[g], worst[g], formulas[g]);
}

int main() {
    run<float>("float");
    run<double>("double");
    return 0;
}
