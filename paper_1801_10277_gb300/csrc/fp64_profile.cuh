// The FP64 pixel path's mixture evaluation: a source's star and galaxy profile sums at a
// pixel, with (gradient) their derivatives over the mean and the shape, from the patch's
// FP64 table in the frame that whitens each PSF component (Section III model).
//
// What bounds it is the FP64 pipe alone: a warp's FP64 instruction holds a sub-partition's
// pipe for 64 cycles, in which some 60 FP32 and integer instructions issue.  So FP64
// instructions are what is counted here, and whatever can be done on the other pipes is:
//   - the whitened frame (item_kernels.cu describes it): every profile component of PSF
//     component k shares T_k, its exponent is -(l1 z1^2 + l2 z2^2) / 2, and its derivatives
//     need only sums over the components of N times constants of the table;
//   - 2^x by table and a cubic (Tang, "Table-driven implementation of the exponential
//     function", ACM TOMS 15, 1989): x = n / 2048 + r with n found from an FP32 copy of x
//     (two FP32 operations; r need not be the smallest remainder, only exact, and the FMA
//     chain that forms x takes -n as its addend), 2^(n mod 2048 / 2048) from a table, the
//     power of two into the exponent field with integer operations.
// A component costs 7 FP64 instructions for the value (2 exponent, 4 for 2^x, 1 sum) and
// 14 with its derivatives, where the pixel-frame formulas and exp2() took 21 and 36.
// Measured (500 sources, 909,100 source-pixels): the adjoint 3.64 -> 1.51 ms, about 800 FP64
// instructions per warp, which is the pipe's rate; the map pass, now at the 59,000 multiply
// covered pixels alone, 2.13 -> 0.14 ms; the Hessian pass of 64 crowded sources (118,800
// source-pixels) 1.53 -> 0.58 ms.  Error of the gradient against 64-bit autograd unchanged.
#pragma once

#include "internal.cuh"

namespace cel {

namespace {

constexpr int EX_N = 2048;                        // table entries per octave
constexpr double EX_HALF = -1477.3197218702985;   // -(2048 log2 e) / 2: exponents in 1/2048 octaves
constexpr double EX_IHALF = 1.0 / EX_HALF;
// 2^(r / 2048) - 1 = r (c1 + r (c2 + r c3)) + O(r^4): c_k = (ln 2 / 2048)^k / k!; |r| <= 1/2
// (a little more where x is large) leaves 3.4e-17
constexpr double EX_C1 = 0x1.62e42fefa39efp-12, EX_C2 = 0x1.ebfbdff82c58fp-25, EX_C3 = 0x1.c6b08d704a0c0p-38;
// below 2^-1020 the value is taken as 0
constexpr float EX_MIN = -1020.f * EX_N;

struct alignas(16) Exp2Table {
    double v[EX_N];
};
struct DoubleDouble {
    double h, l;
};
// a b in double-double (Dekker's product; exact but for the products of low parts)
constexpr DoubleDouble dd_mul(DoubleDouble a, DoubleDouble b) {
    const double ca = 134217729.0 * a.h, cb = 134217729.0 * b.h;
    const double ah = ca - (ca - a.h), bh = cb - (cb - b.h), al = a.h - ah, bl = b.h - bh;
    const double p = a.h * b.h;
    const double e = (((ah * bh - p) + ah * bl + al * bh) + al * bl) + (a.h * b.l + a.l * b.h);
    const double h = p + e;
    return DoubleDouble{h, e - (h - p)};
}
// 2^(i / 2048), correctly rounded from products of the roots 2^(1/2), 2^(1/4), ...
constexpr Exp2Table exp2_table() {
    // 2^(2^b / 2048), b = 0 .. 10
    const DoubleDouble root[11] = {
        {0x1.00162f3904052p+0, -0x1.7b5d0d58ea8f4p-58}, {0x1.002c605e2e8cfp+0, -0x1.d7c96f201bb2fp-55},
        {0x1.0058c86da1c0ap+0, -0x1.5e00e62d6b30dp-56}, {0x1.00b1afa5abcbfp+0, -0x1.4f6b2a7609f71p-55},
        {0x1.0163da9fb3335p+0, 0x1.b61299ab8cdb7p-54},  {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56},
        {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55},  {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54},
        {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55},
        {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}};
    Exp2Table t{};
    for (int i = 0; i < EX_N; ++i) {
        DoubleDouble x{1.0, 0.0};
        for (int b = 0; b < 11; ++b)
            if (i >> b & 1) x = dd_mul(x, root[b]);
        t.v[i] = x.h;
    }
    return t;
}
__device__ const Exp2Table g_exp2 = exp2_table();

// the table into shared memory (16-byte aligned, EX_N doubles; the caller synchronises)
__device__ __forceinline__ void load_exp2_table(double* tab) {
    const double2* s = reinterpret_cast<const double2*>(g_exp2.v);
    for (int i = threadIdx.x; i < EX_N / 2; i += blockDim.x) reinterpret_cast<double2*>(tab)[i] = s[i];
}

// 2^((a q1 + b q2) / 2048) for a, b <= 0 <= q1, q2; (a32, b32, f1, f2): the same in FP32,
// accurate to FP32 rounding.  Below 2^22 units the rounding constant leaves rint(t) in s.
__device__ __forceinline__ double ex2_quad(double a, double q1, double b, double q2, float a32, float f1,
                                           float b32, float f2, const double* tab) {
    const float t = __fmaf_rn(a32, f1, __fmul_rn(b32, f2));
    const float s = __fadd_rn(t, 12582912.f);
    const int n = __float_as_int(s) - 0x4B400000;
    // -n as a double, from its FP32 bits (0 becomes 2^-127, which r does not see)
    const unsigned u = __float_as_uint(__fsub_rn(12582912.f, s));
    const double m = __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
    const double r = __fma_rn(a, q1, __fma_rn(b, q2, m));
    const double p = __dmul_rn(r, __fma_rn(r, __fma_rn(r, EX_C3, EX_C2), EX_C1));
    const double T = tab[n & (EX_N - 1)];
    const double e = __fma_rn(T, p, T);
    const int hi = __double2hiint(e) + ((n >> 11) << 20);
    return t < EX_MIN ? 0.0 : __hiloint2double(hi, __double2loint(e));
}

__device__ __forceinline__ float2 as_float2(double x) {
    return make_float2(__int_as_float(__double2loint(x)), __int_as_float(__double2hiint(x)));
}
__device__ __forceinline__ double pack_float2(float a, float b) {
    return __hiloint2double(__float_as_int(b), __float_as_int(a));
}

// profile sums of one source at one pixel: g0 the star's, ge / gd the galaxy's exp and dev
// parts, and the derivatives (g1 = (1 - e_dev) ge + e_dev gd)
struct Profile64 {
    double g0, gx0, gy0, ge, gd, gx1, gy1, sxx, sxy, syy;
};

// KG: 9 doubles per PSF component, the map of the whitened shape sums back through T
// (xx: T11^2, 2 T11 T21, T21^2; xy: T11 T12, T11 T22 + T21 T12, T21 T22; yy: T12^2,
// 2 T12 T22, T22^2).  The value (g0, ge, gd) is formed by the same operations with and
// without GRAD.
constexpr int KG_STRIDE = 10;
__device__ __forceinline__ void load_shape_maps(double* KG, const double* sT, int npsf) {
    for (int i = threadIdx.x; i < npsf * 9; i += blockDim.x) {
        const int k = i / 9, c = (i % 9) / 3, e = i % 3;
        const double* F = sT + T_STAR + k * STAR_STRIDE;   // T11 T12 T21 T22
        const int p = c == 2, q = c > 0, r = e == 2 ? 2 : 0, s = e > 0 ? 2 : 0;
        // T_rp T_sq, symmetrised over (r, s); the mixed sum enters xx and yy twice
        double v = F[r + p] * F[s + q];
        if (e == 1) v += F[s + p] * F[r + q];
        KG[k * KG_STRIDE + 3 * c + e] = v;
    }
}

template <bool GRAD>
__device__ __forceinline__ void profile64(const double* sT, const double* KG, const double* tab, int npsf, int nprof,
                                          int n_exp, double X, double Y, Profile64& o) {
    o.g0 = o.ge = o.gd = 0.0;
    if (GRAD) o.gx0 = o.gy0 = o.gx1 = o.gy1 = o.sxx = o.sxy = o.syy = 0.0;
    for (int k = 0; k < npsf; ++k) {
        const double2 mean = *reinterpret_cast<const double2*>(sT + T_MEAN + 2 * k);
        const double2* F = reinterpret_cast<const double2*>(sT + T_STAR + k * STAR_STRIDE);
        const double2 t0 = F[0], t1 = F[1];
        const double cs = F[3].x;
        const double dx = __dsub_rn(X, mean.x), dy = __dsub_rn(Y, mean.y);
        const double z1 = __fma_rn(t0.x, dx, __dmul_rn(t0.y, dy)), z2 = __fma_rn(t1.x, dx, __dmul_rn(t1.y, dy));
        const double q1 = __dmul_rn(z1, z1), q2 = __dmul_rn(z2, z2);
        const float f1 = (float)q1, f2 = (float)q2;
        const double es = __dmul_rn(
            cs, ex2_quad(EX_HALF, q1, EX_HALF, q2, (float)EX_HALF, f1, (float)EX_HALF, f2, tab));
        o.g0 = __dadd_rn(o.g0, es);
        if (GRAD) {
            const double su = es * z1, sv = es * z2;
            o.gx0 = fma(t0.x, su, fma(t1.x, sv, o.gx0));
            o.gy0 = fma(t0.y, su, fma(t1.y, sv, o.gy0));
        }
        double u1 = 0.0, u2 = 0.0, w11 = 0.0, w12 = 0.0, w22 = 0.0;
        const double2* row = reinterpret_cast<const double2*>(sT + T_GAL + k * nprof * GAL_STRIDE);
        auto component = [&](double& g) {
            const double2 ab = row[0], pu = row[1];
            const float2 ab32 = as_float2(pu.x);
            const double e = ex2_quad(ab.x, q1, ab.y, q2, ab32.x, f1, ab32.y, f2, tab);
            g = __fma_rn(pu.y, e, g);
            if (GRAD) {
                const double2 u = row[2], wa = row[3], wv = row[5];
                u1 = fma(u.x, e, u1);
                u2 = fma(u.y, e, u2);
                w11 = fma(fma(wa.x, q1, wa.y), e, w11);
                w12 = fma(row[4].x, e, w12);
                w22 = fma(fma(wv.x, q2, wv.y), e, w22);
            }
            row += GAL_STRIDE / 2;
        };
#pragma unroll 2
        for (int j = 0; j < n_exp; ++j) component(o.ge);
#pragma unroll 2
        for (int j = n_exp; j < nprof; ++j) component(o.gd);
        if (GRAD) {
            const double a = z1 * u1, b = z2 * u2;
            o.gx1 = fma(t0.x, a, fma(t1.x, b, o.gx1));
            o.gy1 = fma(t0.y, a, fma(t1.y, b, o.gy1));
            const double w = z1 * z2 * w12;
            const double* m = KG + k * KG_STRIDE;
            o.sxx = fma(m[0], w11, fma(m[1], w, fma(m[2], w22, o.sxx)));
            o.sxy = fma(m[3], w11, fma(m[4], w, fma(m[5], w22, o.sxy)));
            o.syy = fma(m[6], w11, fma(m[7], w, fma(m[8], w22, o.syy)));
        }
    }
}

// E_s = a0 f0 + a1 f1 and Var_s = a0 f0^2 em0 + a1 f1^2 em1 + a0 (1 - a0) f0^2 + a1 (1 - a1) f1^2
// - 2 a0 a1 f0 f1 (em_i = E[l_i^2] / E[l_i]^2 - 1) from the profile sums, f_i = iota E[l_i] g_i;
// every rounding written out (the map pass and the adjoint form the same bits)
__device__ __forceinline__ void source_ev64(const double* sT, double em0, double em1, double g0, double g1,
                                            double& es, double& vs) {
    const double a0 = sT[H_A0], a1 = sT[H_A1], iota = sT[H_IOTA];
    const double f0 = __dmul_rn(__dmul_rn(iota, sT[H_EL0]), g0), f1 = __dmul_rn(__dmul_rn(iota, sT[H_EL1]), g1);
    es = __fma_rn(a0, f0, __dmul_rn(a1, f1));
    const double f00 = __dmul_rn(f0, f0), f11 = __dmul_rn(f1, f1);
    const double k0 = __dmul_rn(a0, __dadd_rn(em0, __dsub_rn(1.0, a0)));
    const double k1 = __dmul_rn(a1, __dadd_rn(em1, __dsub_rn(1.0, a1)));
    vs = __fma_rn(k0, f00, __fma_rn(k1, f11, __dmul_rn(__dmul_rn(-2.0, __dmul_rn(a0, a1)), __dmul_rn(f0, f1))));
}
__device__ __forceinline__ double galaxy64(const double* sT, const Profile64& o) {
    const double ed = sT[H_EDEV];
    return __fma_rn(__dsub_rn(1.0, ed), o.ge, __dmul_rn(ed, o.gd));
}
// E[l^2] / E[l]^2 - 1 of each type
__device__ __forceinline__ void moment_ratios64(const double* sT, double& em0, double& em1) {
    const double el0 = sT[H_EL0], el1 = sT[H_EL1];
    em0 = __dsub_rn(__ddiv_rn(sT[H_EL20], __dmul_rn(el0, el0)), 1.0);
    em1 = __dsub_rn(__ddiv_rn(sT[H_EL21], __dmul_rn(el1, el1)), 1.0);
}
// x (log E - Var / (2 E^2)) - E, iE = 1 / E
__device__ __forceinline__ double pixel_ll64(double x, double E, double V, double iE) {
    return __dsub_rn(__dmul_rn(x, __dsub_rn(log(E), __dmul_rn(__dmul_rn(0.5, V), __dmul_rn(iE, iE)))), E);
}

}  // namespace

}  // namespace cel
