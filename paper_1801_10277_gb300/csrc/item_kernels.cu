// FP32 value / gradient pass of the ELBO over every source's active pixels, in the frame
// that whitens each PSF component (Section III model; Section VI-B: the cost is
// proportional to active pixel visits).
//
// Frame.  For PSF component k (covariance Sigma_k = L L^T) and the source's galaxy shape G
// in the patch's pixel frame, let L^-1 G L^-T = Q D Q^T (D = diag(D1, D2) >= 0) and
// T = Q^T L^-1.  Then T Sigma_k T^T = I and T G T^T = D, so every galaxy component j of
// PSF component k, covariance C_kj = Sigma_k + nu_j G, has precision T^T Lam_j T with
// Lam_j = diag(l1_j, l2_j), l_i = 1 / (1 + nu_j D_i), and det C_kj = det Sigma_k / (l1 l2).
// With z = T d (d = pixel - mean):
//   N_kj         = exp2(-log2(e)/2 (l1 z1^2 + l2 z2^2) + c_j)            (two FMAs)
//   dN/dmean     = N T^T (l1 z1, l2 z2)
//   dN/dG        = nu_j N T^T (Lam z z^T Lam - Lam) T / 2
// so per component only the sums over j of N times (1, l1, l2, nu (l1^2 z1^2 - l1),
// nu l1 l2, nu (l2^2 z2^2 - l2)) are accumulated (ten FMA-pipe operations), and T maps
// them back once per (pixel, k).  The star's component is the case nu = 0.  Packed FP32x2
// arithmetic pairs two mixture components per instruction (coefficients of adjacent
// components side by side in the table).
//
// Work.  Three launches.  k_tables builds every patch's table and chain-rule record (a
// warp per patch or per four, FP32 with the position in FP64), publishing each with a ready flag, and
// every source's KL terms (one warp per source).  k_items, its programmatic dependent,
// runs on persistent CTAs of four warps that take items from a queue (a global counter over
// the items in decreasing cost): up to ZIMAX pixels of one patch, the multiply covered ones
// first.  An item's patch table, its pixel records and the value records of up to ZSTAGE other
// patches covering its pixels are copied into a shared-memory stage with bulk asynchronous
// copies (two stages, completing on mbarriers; the warp that finishes an item last waits for
// the tables that the item after the next reads and starts its copies), while the warps take the
// chunks of 64 pixels of the item in the other stage in turn.  They evaluate the mixture and its
// derivatives at the chunk's pixels; where other patches cover a pixel, E = sky + sum_s
// E_s and Var = sum_s Var_s are summed over every covering source in ascending source
// order (every covering item forms the same sum, bit for bit).  FP32 sums per chunk, added
// in FP64 to the item's record (ll and d ll / d y).  k_finish, k_items' programmatic
// dependent, runs every source's epilogue once the items are done (FP64 sums of each patch's
// item records in a fixed order, the patch's chain rule dy/dtheta, minus the KL); the last
// CTA to finish adds the sources' shares of the total in source order.
// Every wait is bounded (~1 s), after which the kernel records CELESTE_ERR_TIMEOUT and
// ends.
#include <math.h>

#include "internal.cuh"
#include "source_math.cuh"
#include "epilogue.cuh"
#include "async_copy.cuh"

namespace cel {

namespace {

constexpr float HL = -0.72134752044448170368f;   // -log2(e) / 2


// Table layout (floats).  Value part (the prefix that another patch's items copy):
//   header [0..15]: a0 a1 el0 el20 el1 el21 iota e_dev em0 em1 (1 - e_dev) band A[4]
//   per PSF component k at VH + k VK:
//     [0..3] -mean_x -mean_y c_star sign   [4..7] T11 T12 T21 T22
//     profile component pair q at VKH + q VPAIR, the entries of components 2q and 2q + 1
//     side by side (so that one 8-byte half of a 16-byte load is a packed FP32x2 operand):
//       [A A B B] [C C U1 U1]
// Gradient part, per PSF component k at VFULL + k GK:
//     [0..8] finishing coefficients of T^T W T (xx: T11^2, 2 T11 T21, T21^2; xy: T11 T12,
//            T11 T22 + T21 T12, T21 T22; yy: T12^2, 2 T12 T22, T22^2), [9..11] unused
//     component pair q at GKH + q GPAIR: [U2 U2 Wa Wa] [Wb Wb W12 W12] [Va Va Vb Vb]
//   A, B = -log2(e)/2 (l1, l2); C = log2(|alpha_k| w_j) - log2(2 pi sqrt(det C_kj));
//   U1, U2 = s (l1, l2); Wa, Wb = s nu (l1^2, -l1); W12 = s nu l1 l2; Va, Vb = s nu (l2^2, -l2)
//   (s = sign(alpha_k) (1 - e_dev) for exp components, sign(alpha_k) e_dev for dev ones);
//   exp components fill pairs 0 .. npe-1, dev components pairs npe .. npe+npd-1, each
//   group padded to an even count with a component of weight zero (C = -1e30).
// Chain-rule record of a patch: per theta column j < ZCHAIN (the pixels do not depend on the
// others), (k0, k1, k2, y0 | y1 << 4 | y2 << 8):
// d y_{y_e} / d theta_j = k_e (unused pairs y = 0, k = 0).
constexpr int ZMAXPAIR = (MAXPROF + 2) / 2;
constexpr int VH = 16, VKH = 8, VPAIR = 8, VK = VKH + ZMAXPAIR * VPAIR, VFULL = VH + MAXPSF * VK;
constexpr int GKH = 12, GPAIR = 12, GK = GKH + ZMAXPAIR * GPAIR, GFULL = MAXPSF * GK;
constexpr int ZFULL = VFULL + GFULL;
static_assert(ZFULL == ZFULL_FLOATS, "table size");
static_assert(VFULL % 4 == 0 && ZFULL % 4 == 0, "tables are copied in 16-byte units");

// CTA shape: four warps
constexpr int NWC = 4;
constexpr int NTC = 32 * NWC;

// One shared-memory stage (bytes): the item's table, its pixel records, and its first
// ZSTAGE candidates' records and value tables.
constexpr int ST_TBL = 0;
constexpr int ST_PX = ST_TBL + ZFULL * 4;
constexpr int ST_ZC = ST_PX + ZIMAX * 16;
constexpr int ST_VREC = ST_ZC + ZSTAGE * (int)sizeof(ZCand);
constexpr int ST_BYTES = ST_VREC + ZSTAGE * VFULL * 4;
static_assert(ST_PX % 16 == 0 && ST_ZC % 16 == 0 && ST_VREC % 16 == 0 && ST_BYTES % 16 == 0,
              "bulk copies land on 16-byte boundaries");
static_assert(sizeof(ZCand) == 32 && sizeof(ZTask) == 64, "record sizes");

constexpr int PG_F = 10;                 // floats of a ProfileGrad
constexpr int SCR_W = 880;               // bytes per warp of the table kernel: KL arrays (2 x 44
                                         // doubles, 44 floats) or the table builder's 96 floats

// Pixels per thread; a chunk is the 32 PX pixels of one pass of a warp
constexpr int PX = 2;
static_assert(32 * PX == ZCHUNK, "chunk size");

// the rest of the item kernel's shared memory (bytes), after the two stages
struct Lay {
    static constexpr int pg = 2 * ST_BYTES;                        // stashed derivatives [PX PG_F][NTC]
    static constexpr int nch = ZIMAX / ZCHUNK;                     // most chunks of an item
    static constexpr int red = pg + PX * PG_F * NTC * 4;           // [2][nch][16] chunk sums
    static constexpr int bar = red + 2 * nch * 16 * 4;             // full[2], fetched[2]
    static constexpr int task = bar + 4 * 8;                       // [2] ZTask: the stages' items
    static constexpr int next = task + 2 * (int)sizeof(ZTask);     // [2] ZTask: records fetched ahead
    static constexpr int cnt = next + 2 * (int)sizeof(ZTask);      // [2] warps done with the stage's item,
                                                                   // [2] its chunks taken
    static constexpr int bytes = cnt + 16;
    static_assert(task % 16 == 0 && bar % 8 == 0, "alignment");
};

// Registers per thread with MINB CTAs of four warps per SM (one per sub-partition, whose 16K
// registers its MINB warps share), in multiples of 8.
constexpr int regs_for(int minb) {
    const int r = (16384 / (minb * 32)) & ~7;
    return r < 248 ? r : 248;
}

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 ex2x2(float2 a) { return make_float2(ex2f(a.x), ex2f(a.y)); }
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// ---------------------------------------------------------------------------------
// table construction: LP lanes per patch, written to the table in global memory

// A patch's table and chain-rule record, built by LP lanes (32 or 8: one or four patches per
// warp; every lane of the warp calls it, live: its patch is one to build).  Every lane first converts
// a share of theta to FP32 (FP64 -> FP32 conversions and FP64 arithmetic have ~70-cycle
// latencies on GB300's narrow FP64 pipe, so each is done once); lane 0 forms the position
// in FP64 (relative to the patch origin, so FP32 offsets stay exact).  Then every lane
// computes, and one lane each stores: PSF component k's frame (lanes k < npsf), the
// brightness moments of each type (lanes npsf, npsf + 1), the weights (lane npsf + 2)
// and the shape Jacobian (lane npsf + 3);
// finally one lane per (PSF component, component slot) the slot's coefficients and one
// lane per theta column its chain-rule pairs.  sm: 96 floats of this patch's shared memory.

template <int LP>
__device__ __forceinline__ void build_patch_table(const double* __restrict__ theta, const ZBuild& g, bool live,
                                                  const ImgMeta* __restrict__ img, const ModelDev& md,
                                                  float* __restrict__ ztbl, float4* __restrict__ zchain,
                                                  float* sm) {
    static_assert(LP >= MAXPSF + 4, "a lane per part of phase one");
    const int lane = threadIdx.x & (LP - 1);
    const int patch = g.patch;
    const ImgMeta& im = img[g.img];
    const double* th = theta + (size_t)NP * g.src;
    float* T = ztbl + (size_t)patch * ZFULL;
    float* thf = sm;        // [44] theta in FP32
    float* dscr = sm + 44;  // [8] D1, D2 per PSF component
    float* mu = sm + 52;    // [2] position relative to the patch origin
    float* elv = sm + 56;   // [4] el0, el1, el20, el21
    float* dgs = sm + 60;   // [9] dG
    float* Af = sm + 69;    // [4] A
    // every global value this lane reads below, loaded together (one memory round trip)
    const int npsf = im.npsf, band = im.band;
    const float a0 = im.A_f[0], a1 = im.A_f[1], a2 = im.A_f[2], a3 = im.A_f[3];
    const int kk = lane < npsf ? lane : 0;
    const float li0 = im.psf_li[kk][0], li1 = im.psf_li[kk][1], li2 = im.psf_li[kk][2], dmk = im.psf_dm[kk];
    const float ps1 = im.psf_f[kk][1], ps2 = im.psf_f[kk][2], csk = im.psf_cs[kk], sgk = im.psf_sg[kk];
    const float iota = im.iota_f;
    const int n_exp = md.n_exp, n_dev = md.n_dev;
#pragma unroll
    for (int i = 0; i < (NP + LP - 1) / LP; ++i)
        if (lane + LP * i < NP) thf[lane + LP * i] = (float)th[lane + LP * i];
    if (lane == 0) {
        const double u0 = th[0], u1 = th[1];
        mu[0] = (float)fma(im.A[0], u0, fma(im.A[1], u1, g.ox));
        mu[1] = (float)fma(im.A[2], u0, fma(im.A[3], u1, g.oy));
    }
    __syncwarp();
    const float rho = thf[P_AXIS], phi = thf[P_ANGLE], sg = thf[P_SCALE], ed = thf[P_EDEV];
    // Phase one, straight-line on every lane (the four parts are independent, so their
    // latencies overlap instead of adding up); each lane stores only its own part.
    float s2, c2;
    sincosf(2.f * phi, &s2, &c2);
    {
        // PSF component kk's frame: shape G = A W A^T in this patch's pixel frame,
        // W = sigma^2 R(phi) diag(1, rho^2), R(phi)^T = ah I + bh (cos 2phi, sin 2phi;
        // sin 2phi, -cos 2phi)
        const float ah = 0.5f * sg * sg * (1.f + rho * rho), bh = 0.5f * sg * sg * (1.f - rho * rho);
        const float wxx = ah + bh * c2, wxy = bh * s2, wyy = ah - bh * c2;
        const float gxx = a0 * a0 * wxx + 2.f * a0 * a1 * wxy + a1 * a1 * wyy;
        const float gxy = a0 * a2 * wxx + (a0 * a3 + a1 * a2) * wxy + a1 * a3 * wyy;
        const float gyy = a2 * a2 * wxx + 2.f * a2 * a3 * wxy + a3 * a3 * wyy;
        const float a = li0, b = li1, c = li2;
        // M = L^-1 G L^-T
        const float bxc = b * gxx + c * gxy, byc = b * gxy + c * gyy;
        const float m11 = a * a * gxx, m12 = a * bxc, m22 = bxc * b + byc * c;
        // Jacobi rotation diagonalising M (symmetric 2 x 2 Schur decomposition)
        float cs = 1.f, sn = 0.f, d1 = m11, d2 = m22;
        if (m12 != 0.f) {
            const float tau = __fdividef(m22 - m11, 2.f * m12);
            const float t = fabsf(tau) > 1e15f ? __fdividef(0.5f, tau)
                                               : copysignf(1.f, tau) * __frcp_rn(fabsf(tau) + sqrtf(1.f + tau * tau));
            cs = rsqrtf(1.f + t * t);
            sn = t * cs;
            d1 = m11 - t * m12;
            d2 = m22 + t * m12;
        }
        // the smaller eigenvalue from det M = psf_dm sigma^4 rho^2 (no cancellation)
        const float detm = dmk * (sg * sg * rho) * (sg * sg * rho);
        if (d1 >= d2 && d1 > 0.f) d2 = detm * __frcp_rn(d1);
        else if (d2 > d1 && d2 > 0.f) d1 = detm * __frcp_rn(d2);
        d1 = fmaxf(d1, 0.f);
        d2 = fmaxf(d2, 0.f);
        const float t11 = cs * a - sn * b, t12 = -sn * c, t21 = sn * a + cs * b, t22 = cs * c;
        if (live && lane < npsf) {
            const int k = lane;
            float4* K = reinterpret_cast<float4*>(T + VH + k * VK);
            K[0] = make_float4(-(mu[0] + ps1), -(mu[1] + ps2), csk, sgk);
            K[1] = make_float4(t11, t12, t21, t22);
            float4* KG = reinterpret_cast<float4*>(T + VFULL + k * GK);
            KG[0] = make_float4(t11 * t11, 2.f * t11 * t21, t21 * t21, t11 * t12);
            KG[1] = make_float4(t11 * t22 + t21 * t12, t21 * t22, t12 * t12, 2.f * t12 * t22);
            KG[2] = make_float4(t22 * t22, 0.f, 0.f, 0.f);
            dscr[2 * k] = d1;
            dscr[2 * k + 1] = d2;
        }
    }
    {
        // brightness of type i in this band: log l ~ N(m, v); E[l] = e^{m+v/2},
        // E[l^2] = e^{2m+2v}, E[l^2] / E[l]^2 - 1 = e^v - 1
        const int i = lane == npsf + 1 ? 1 : 0;
        float m = thf[P_R1 + i], v = thf[P_R2 + i];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float bb = band_beta<float>(band, j);
            m += bb * thf[P_C1 + 4 * i + j];
            v += bb * bb * thf[P_C2 + 4 * i + j];
        }
        const float el = expf(m + 0.5f * v), el2 = expf(2.f * m + 2.f * v), em = expm1f(v);
        if (live && (lane == npsf || lane == npsf + 1)) {
            T[2 + 2 * i] = el;
            T[3 + 2 * i] = el2;
            T[8 + i] = em;
            elv[i] = el;
            elv[2 + i] = el2;
        }
    }
    if (lane == npsf + 2) {
        Af[0] = a0; Af[1] = a1; Af[2] = a2; Af[3] = a3;
    }
    if (live && lane == npsf + 2) {
        T[0] = thf[P_A];
        T[1] = thf[P_A + 1];
        T[6] = iota;
        T[7] = ed;
        T[10] = 1.f - ed;
        T[11] = (float)band;
        T[12] = a0; T[13] = a1; T[14] = a2; T[15] = a3;
    }
    {
        // dG = A dW A^T, dW = d(Wxx, Wxy, Wyy) / d(e_axis, e_angle, e_scale)
        const float bh = 0.5f * sg * sg * (1.f - rho * rho);
        float dW[3][3];
        float da = sg * sg * rho, db = -sg * sg * rho;
        dW[0][0] = da + db * c2; dW[0][1] = db * s2; dW[0][2] = da - db * c2;
        dW[1][0] = -2.f * bh * s2; dW[1][1] = 2.f * bh * c2; dW[1][2] = 2.f * bh * s2;
        da = sg * (1.f + rho * rho); db = sg * (1.f - rho * rho);
        dW[2][0] = da + db * c2; dW[2][1] = db * s2; dW[2][2] = da - db * c2;
        if (live && lane == npsf + 3) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float ux = dW[q][0], uxy = dW[q][1], uy = dW[q][2];
                dgs[3 * q + 0] = a0 * a0 * ux + 2.f * a0 * a1 * uxy + a1 * a1 * uy;
                dgs[3 * q + 1] = a0 * a2 * ux + (a0 * a3 + a1 * a2) * uxy + a1 * a3 * uy;
                dgs[3 * q + 2] = a2 * a2 * ux + 2.f * a2 * a3 * uxy + a3 * a3 * uy;
            }
        }
    }
    // the coefficients of each (PSF component k, component slot): lane r takes slots r,
    // r + LP, ..., whose constants are read before the wait for phase one (LP = 32)
    const int npe = (n_exp + 1) >> 1, nslot = 2 * (npe + ((n_dev + 1) >> 1));
    constexpr int NR = (MAXPSF * 2 * ZMAXPAIR + LP - 1) / LP;   // rounds of LP slots
    constexpr int NA = LP == 32 ? NR : 1;                       // rounds read ahead
    const float inv_nslot = __frcp_rn((float)nslot);
    int sk[NA], ss[NA], sj[NA];
    float snu[NA], slw[NA], ssg[NA], scs[NA];
    auto constants = [&](int u, int e) {
        const int r = lane + LP * u;
        // r / nslot (r + 1/2 is no multiple of nslot and r < 2^7, so the product cannot round across one)
        const int k = (int)(((float)r + 0.5f) * inv_nslot), slot = r - k * nslot;
        int j = -1;   // slot -> profile component j (or a padding slot)
        if (r < npsf * nslot) {
            if (slot < 2 * npe) {
                if (slot < n_exp) j = slot;
            } else if (slot - 2 * npe < n_dev) {
                j = n_exp + slot - 2 * npe;
            }
        }
        sk[e] = k;
        ss[e] = slot;
        sj[e] = j;
        snu[e] = j >= 0 ? md.prof_nu_f[j] : 0.f;
        slw[e] = j >= 0 ? md.prof_lw_f[j] : 0.f;
        ssg[e] = r < npsf * nslot ? im.psf_sg[k] : 0.f;
        scs[e] = r < npsf * nslot ? im.psf_cs[k] : 0.f;
    };
    if (NA > 1) {
#pragma unroll
        for (int u = 0; u < NA; ++u) constants(u, u);
    }
    __syncwarp();
#pragma unroll(NA > 1 ? NR : 1)
    for (int u_ = 0; u_ < NR; ++u_) {
        const int u = NA > 1 ? u_ : 0;
        if (!live || lane + LP * u_ >= npsf * nslot) break;
        if (NA == 1) constants(u_, 0);
        const int k = sk[u], slot = ss[u], q = slot >> 1, h = slot & 1, j = sj[u];
        const bool dev = j >= n_exp;
        float A = 0.f, B = 0.f, C = -1e30f, U1 = 0.f, U2 = 0.f, Wa = 0.f, Wb = 0.f, W12 = 0.f, Va = 0.f, Vb = 0.f;
        if (j >= 0) {
            const float nu = snu[u];
            const float l1 = __frcp_rn(1.f + nu * dscr[2 * k]), l2 = __frcp_rn(1.f + nu * dscr[2 * k + 1]);
            const float sgn = ssg[u] * (dev ? ed : 1.f - ed);
            A = HL * l1;
            B = HL * l2;
            C = scs[u] + slw[u] + 0.5f * (__log2f(l1) + __log2f(l2));
            U1 = sgn * l1;
            U2 = sgn * l2;
            const float snu_ = sgn * nu;
            Wa = snu_ * l1 * l1;
            Wb = -snu_ * l1;
            W12 = snu_ * l1 * l2;
            Va = snu_ * l2 * l2;
            Vb = -snu_ * l2;
        }
        float* pv = T + VH + k * VK + VKH + q * VPAIR + h;
        pv[0] = A; pv[2] = B; pv[4] = C; pv[6] = U1;
        float* pq = T + VFULL + k * GK + GKH + q * GPAIR + h;
        pq[0] = U2; pq[2] = Wa; pq[4] = Wb; pq[6] = W12; pq[8] = Va; pq[10] = Vb;
    }
    // the chain-rule record: column j of dy/dtheta for this patch
#pragma unroll 1
    for (int j = lane; live && j < ZCHAIN; j += LP) {
        int y0, y1, y2;
        float k0, k1, k2;
        chain_column<float>(j, band, Af, elv, elv + 2, reinterpret_cast<const float(*)[3]>(dgs), &y0, &k0, &y1, &k1, &y2, &k2);
        zchain[(size_t)patch * ZCHAIN + j] = make_float4(k0, k1, k2, __int_as_float(y0 | (y1 << 4) | (y2 << 8)));
    }
}

// Ready flags of the tables (one int per patch, 0 before the launch): the building warp
// publishes its table and chain record with a release (fence, then the flag) and counts
// it in `built`; a reader acquires the flag, waiting at most ~1 s of SM clock (or less
// once another wait has given up), after which it records CELESTE_ERR_TIMEOUT and goes on.
__device__ __forceinline__ void publish_ready(int32_t* flag, int32_t* built) {
    asm volatile("st.release.gpu.global.s32 [%0], 1;" ::"l"(flag) : "memory");
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(built) : "memory");
}

__device__ __forceinline__ int load_acquire(const int32_t* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// another wait of the launch gave up, or a bounds check failed: waits end at once
__device__ __forceinline__ bool timed_out(const int32_t* status) {
    const int32_t v = *reinterpret_cast<const volatile int32_t*>(status);
    return v == (int32_t)CELESTE_ERR_TIMEOUT || v == (int32_t)CELESTE_ERR_BOUNDS;
}

// a wait that gave up records CELESTE_ERR_TIMEOUT unless an error is recorded already
__device__ __forceinline__ void record_timeout(int32_t* status) {
    atomicCAS(status, 0, (int32_t)CELESTE_ERR_TIMEOUT);
}

__device__ __forceinline__ void wait_ready(const int32_t* flag, int32_t* status) {
    if (load_acquire(flag)) return;
    const long long t0 = clock64();
    for (int i = 0; i < (1 << 24); ++i) {
        __nanosleep(64);
        if (load_acquire(flag)) return;
        if (timed_out(status) || clock64() - t0 > MBAR_MAX_CYCLES) break;
    }
    record_timeout(status);
}

// an mbarrier wait that also gives up once another wait of the launch has
__device__ __forceinline__ bool mbar_wait_launch(uint64_t* bar, unsigned parity, int32_t* status) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (int i = 0; i < MBAR_MAX_POLLS; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63) == 63 && timed_out(status)) break;
        if (clock64() - t0 > MBAR_MAX_CYCLES) break;
    }
    record_timeout(status);
    return false;
}

// A warp that gave up on a wait at item i: let the copies that its CTA has in flight (the stages and
// the records ahead of items i and i + 1) land before it leaves, as the shared memory is another
// CTA's next.  A barrier that nothing is on its way to costs the limit, about 10 ms.
__device__ __forceinline__ void drain(uint64_t* full, uint64_t* fetched, int i) {
#pragma unroll 1
    for (int e = 0; e < 4; ++e) {
        const int x = i + (e >> 1);
        uint64_t* bar = (e & 1 ? fetched : full) + (x & 1);
        const long long t0 = clock64();
        for (int n = 0; n < MBAR_MAX_POLLS && clock64() - t0 < MBAR_MAX_CYCLES / 100; ++n)
            if (mbar_try_wait(bar, (x >> 1) & 1)) break;
    }
}

__device__ __forceinline__ void mbar_arrive_plain(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_arrive(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
// one bulk copy completing on bar (whose expected bytes were announced already)
__device__ __forceinline__ void bulk_g2s_tx(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
// order this thread's earlier (acquired) view of global memory before its async-proxy reads
__device__ __forceinline__ void fence_proxy_async_global() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
}

// ---------------------------------------------------------------------------------
// per-pixel evaluation: PX pixels per thread; a packed FP32x2 operation covers two
// profile components of one pixel

// E_s and Var_s of a source at a pixel from its profile sums (every rounding written out,
// the same wherever a source's E_s is formed):
//   f_i = iota E[l_i] g_i,  E_s = a0 f0 + a1 f1,
//   Var_s = a0 f0^2 em0 + a1 f1^2 em1 + a0 (1 - a0) f0^2 + a1 (1 - a1) f1^2 - 2 a0 a1 f0 f1
__device__ __forceinline__ void source_ev(const float* H, float G0, float G1, float& f0, float& f1,
                                          float& es, float& vs) {
    const float a0 = H[0], a1 = H[1], iota = H[6];
    f0 = __fmul_rn(__fmul_rn(iota, H[2]), G0);
    f1 = __fmul_rn(__fmul_rn(iota, H[4]), G1);
    es = __fadd_rn(__fmul_rn(a0, f0), __fmul_rn(a1, f1));
    const float f00 = __fmul_rn(f0, f0), f11 = __fmul_rn(f1, f1);
    float v = __fmul_rn(__fmul_rn(a0, f00), H[8]);
    v = __fadd_rn(v, __fmul_rn(__fmul_rn(a1, f11), H[9]));
    v = __fadd_rn(v, __fmul_rn(__fmul_rn(a0, __fsub_rn(1.f, a0)), f00));
    v = __fadd_rn(v, __fmul_rn(__fmul_rn(a1, __fsub_rn(1.f, a1)), f11));
    vs = __fsub_rn(v, __fmul_rn(__fmul_rn(2.f, __fmul_rn(a0, a1)), __fmul_rn(f0, f1)));
}

// the profile sums g0 (star), g1 (galaxy) of one patch at PX pixels from its value part
// (an item's own table or another patch's value record: the same layout)
template <int NPE, int NPD>
__device__ __forceinline__ void profile_value(const float* H, int npsf, int npe_rt, int npd_rt,
                                              const float (&X)[PX], const float (&Y)[PX], float (&G0)[PX],
                                              float (&G1)[PX]) {
    const int npe = NPE >= 0 ? NPE : npe_rt, npd = NPD >= 0 ? NPD : npd_rt;
    float ge[PX], gd[PX];
#pragma unroll
    for (int p = 0; p < PX; ++p) G0[p] = ge[p] = gd[p] = 0.f;
    for (int k = 0; k < npsf; ++k) {
        const float* K = H + VH + k * VK;
        const float4 h0 = ld4(K), h1 = ld4(K + 4);
        float2 Z1[PX], Z2[PX], xe[PX], xd[PX];
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            const float dx = __fadd_rn(X[p], h0.x), dy = __fadd_rn(Y[p], h0.y);
            const float z1 = __fmaf_rn(h1.x, dx, __fmul_rn(h1.y, dy));
            const float z2 = __fmaf_rn(h1.z, dx, __fmul_rn(h1.w, dy));
            const float q1 = __fmul_rn(z1, z1), q2 = __fmul_rn(z2, z2);
            const float es = ex2f(__fmaf_rn(HL, __fadd_rn(q1, q2), h0.z));
            G0[p] = __fmaf_rn(h0.w, es, G0[p]);
            Z1[p] = dup(q1);
            Z2[p] = dup(q2);
            xe[p] = xd[p] = dup(0.f);
        }
        const float* Q = K + VKH;
        auto pair = [&](int q, bool is_exp) {
            const float4 ab = ld4(Q + q * VPAIR), cc = ld4(Q + q * VPAIR + 4);
            const float2 A = make_float2(ab.x, ab.y), B = make_float2(ab.z, ab.w), C = make_float2(cc.x, cc.y);
#pragma unroll
            for (int p = 0; p < PX; ++p) {
                const float2 e = ex2x2(__ffma2_rn(A, Z1[p], __ffma2_rn(B, Z2[p], C)));
                if (is_exp) xe[p] = __fadd2_rn(xe[p], e);
                else xd[p] = __fadd2_rn(xd[p], e);
            }
        };
        if (NPE >= 0) {
#pragma unroll
            for (int q = 0; q < (NPE >= 0 ? NPE + NPD : 0); ++q) pair(q, q < NPE);
        } else {
            for (int q = 0; q < npe + npd; ++q) pair(q, q < npe);
        }
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            ge[p] = __fmaf_rn(h0.w, __fadd_rn(xe[p].x, xe[p].y), ge[p]);
            gd[p] = __fmaf_rn(h0.w, __fadd_rn(xd[p].x, xd[p].y), gd[p]);
        }
    }
#pragma unroll
    for (int p = 0; p < PX; ++p) G1[p] = __fmaf_rn(H[10], ge[p], __fmul_rn(H[7], gd[p]));
}

struct ProfileGrad {
    float g0, gx0, gy0, g1, gx1, gy1, de, sxx, sxy, syy;
};
static_assert(sizeof(ProfileGrad) == PG_F * sizeof(float), "ProfileGrad layout");

// the profile sums and their derivatives of the item's own patch at PX pixels; g0 and g1
// are formed with exactly the operations of profile_value (UNR: unroll factor of the
// loop over component pairs)
template <int NPE, int NPD, int UNR>
__device__ __forceinline__ void profile_grad(const float* H, int npsf, int npe_rt, int npd_rt,
                                             const float (&X)[PX], const float (&Y)[PX],
                                             ProfileGrad (&o)[PX]) {
    const int npe = NPE >= 0 ? NPE : npe_rt, npd = NPD >= 0 ? NPD : npd_rt;
    float ge[PX], gd[PX];
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        o[p].g0 = o[p].gx0 = o[p].gy0 = o[p].gx1 = o[p].gy1 = o[p].sxx = o[p].sxy = o[p].syy = 0.f;
        ge[p] = gd[p] = 0.f;
    }
    for (int k = 0; k < npsf; ++k) {
        const float* K = H + VH + k * VK;
        const float* KG = H + VFULL + k * GK;
        const float4 h0 = ld4(K), h1 = ld4(K + 4);
        float z1[PX], z2[PX];
        float2 Z1[PX], Z2[PX], xe[PX], xd[PX], u1[PX], u2[PX], w11[PX], w12[PX], w22[PX];
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            const float dx = __fadd_rn(X[p], h0.x), dy = __fadd_rn(Y[p], h0.y);
            z1[p] = __fmaf_rn(h1.x, dx, __fmul_rn(h1.y, dy));
            z2[p] = __fmaf_rn(h1.z, dx, __fmul_rn(h1.w, dy));
            const float q1 = __fmul_rn(z1[p], z1[p]), q2 = __fmul_rn(z2[p], z2[p]);
            const float es = ex2f(__fmaf_rn(HL, __fadd_rn(q1, q2), h0.z));
            o[p].g0 = __fmaf_rn(h0.w, es, o[p].g0);
            // star: d/dmean = sign alpha N T^T z
            const float ge_ = __fmul_rn(h0.w, es);
            const float su = __fmul_rn(ge_, z1[p]), sv = __fmul_rn(ge_, z2[p]);
            o[p].gx0 = __fmaf_rn(h1.x, su, __fmaf_rn(h1.z, sv, o[p].gx0));
            o[p].gy0 = __fmaf_rn(h1.y, su, __fmaf_rn(h1.w, sv, o[p].gy0));
            Z1[p] = dup(q1);
            Z2[p] = dup(q2);
            xe[p] = xd[p] = u1[p] = u2[p] = w11[p] = w12[p] = w22[p] = dup(0.f);
        }
        const float* Q = K + VKH;
        const float* QG = KG + GKH;
        auto pair = [&](int q, bool is_exp) {
            const float4 c0 = ld4(Q + q * VPAIR), c1 = ld4(Q + q * VPAIR + 4);
            const float* cg = QG + q * GPAIR;
            const float4 c2 = ld4(cg), c3 = ld4(cg + 4), c4 = ld4(cg + 8);
            const float2 A = make_float2(c0.x, c0.y), B = make_float2(c0.z, c0.w);
            const float2 C = make_float2(c1.x, c1.y), U1 = make_float2(c1.z, c1.w);
            const float2 U2 = make_float2(c2.x, c2.y), Wa = make_float2(c2.z, c2.w);
            const float2 Wb = make_float2(c3.x, c3.y), W12 = make_float2(c3.z, c3.w);
            const float2 Va = make_float2(c4.x, c4.y), Vb = make_float2(c4.z, c4.w);
#pragma unroll
            for (int p = 0; p < PX; ++p) {
                const float2 e = ex2x2(__ffma2_rn(A, Z1[p], __ffma2_rn(B, Z2[p], C)));
                if (is_exp) xe[p] = __fadd2_rn(xe[p], e);
                else xd[p] = __fadd2_rn(xd[p], e);
                u1[p] = __ffma2_rn(U1, e, u1[p]);
                u2[p] = __ffma2_rn(U2, e, u2[p]);
                w11[p] = __ffma2_rn(__ffma2_rn(Wa, Z1[p], Wb), e, w11[p]);
                w12[p] = __ffma2_rn(W12, e, w12[p]);
                w22[p] = __ffma2_rn(__ffma2_rn(Va, Z2[p], Vb), e, w22[p]);
            }
        };
        if (NPE >= 0) {
#pragma unroll (UNR)
            for (int q = 0; q < (NPE >= 0 ? NPE + NPD : 0); ++q) pair(q, q < NPE);
        } else {
            for (int q = 0; q < npe + npd; ++q) pair(q, q < npe);
        }
        // finish component k: map the whitened sums back with T
        const float4 f0 = ld4(KG), f1 = ld4(KG + 4);
        const float f8 = KG[8];
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            ge[p] = __fmaf_rn(h0.w, __fadd_rn(xe[p].x, xe[p].y), ge[p]);
            gd[p] = __fmaf_rn(h0.w, __fadd_rn(xd[p].x, xd[p].y), gd[p]);
            const float a = __fmul_rn(z1[p], __fadd_rn(u1[p].x, u1[p].y));
            const float b = __fmul_rn(z2[p], __fadd_rn(u2[p].x, u2[p].y));
            o[p].gx1 = __fmaf_rn(h1.x, a, __fmaf_rn(h1.z, b, o[p].gx1));
            o[p].gy1 = __fmaf_rn(h1.y, a, __fmaf_rn(h1.w, b, o[p].gy1));
            const float W11 = __fadd_rn(w11[p].x, w11[p].y);
            const float W12 = __fmul_rn(__fmul_rn(z1[p], z2[p]), __fadd_rn(w12[p].x, w12[p].y));
            const float W22 = __fadd_rn(w22[p].x, w22[p].y);
            o[p].sxx = __fmaf_rn(f0.x, W11, __fmaf_rn(f0.y, W12, __fmaf_rn(f0.z, W22, o[p].sxx)));
            o[p].sxy = __fmaf_rn(f0.w, W11, __fmaf_rn(f1.x, W12, __fmaf_rn(f1.y, W22, o[p].sxy)));
            o[p].syy = __fmaf_rn(f1.z, W11, __fmaf_rn(f1.w, W12, __fmaf_rn(f8, W22, o[p].syy)));
        }
    }
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        o[p].g1 = __fmaf_rn(H[10], ge[p], __fmul_rn(H[7], gd[p]));
        o[p].de = __fsub_rn(gd[p], ge[p]);
    }
}

// ll = x (log E - Var / (2 E^2)) - E and its weights c_E = x (1/E + Var/E^3) - 1,
// c_V = -x / (2 E^2)
__device__ __forceinline__ float pix_ll(float x, float E, float V) {
    const float iE = __frcp_rn(E), iE2 = __fmul_rn(iE, iE);
    return __fsub_rn(__fmul_rn(x, __fsub_rn(logf(E), __fmul_rn(__fmul_rn(0.5f, V), iE2))), E);
}
__device__ __forceinline__ void pix_weights(float x, float E, float V, float& cE, float& cV) {
    const float iE = __frcp_rn(E), iE2 = __fmul_rn(iE, iE);
    cE = __fsub_rn(__fmul_rn(x, __fadd_rn(iE, __fmul_rn(V, __fmul_rn(iE2, iE)))), 1.f);
    cV = __fmul_rn(__fmul_rn(-0.5f, x), iE2);
}

// the item's own source at this thread's pixels: E_s, Var_s, f_i and (gradient) the
// profile sums with their derivatives
template <int MODE, int NPE, int NPD, int UNR>
__device__ __forceinline__ void own_source(const float* H, int npsf, int npe, int npd, const float (&X)[PX],
                                           const float (&Y)[PX], float (&Es)[PX], float (&Vs)[PX],
                                           float (&f0)[PX], float (&f1)[PX], ProfileGrad (&pg)[PX]) {
    if constexpr (MODE == MODE_LL) {
        float G0[PX], G1[PX];
        profile_value<NPE, NPD>(H, npsf, npe, npd, X, Y, G0, G1);
#pragma unroll
        for (int p = 0; p < PX; ++p) source_ev(H, G0[p], G1[p], f0[p], f1[p], Es[p], Vs[p]);
    } else {
        profile_grad<NPE, NPD, UNR>(H, npsf, npe, npd, X, Y, pg);
#pragma unroll
        for (int p = 0; p < PX; ++p) source_ev(H, pg[p].g0, pg[p].g1, f0[p], f1[p], Es[p], Vs[p]);
    }
}

// the pixel's expected log-likelihood into v[0] and (gradient) its adjoint wrt the twelve
// y of the item's patch into v[1 ..]
template <int MODE, int NV>
__device__ __forceinline__ void pixel_terms(const float* H, float x, float E, float V, float Es, float f0,
                                            float f1, const ProfileGrad& q, float (&v)[NV], float& ll) {
    ll = pix_ll(x, E, V);
    v[0] += ll;
    if constexpr (MODE >= MODE_GRAD) {
        const float a0 = H[0], a1 = H[1], iota = H[6];
        const float el0 = H[2], el20 = H[3], el1 = H[4], el21 = H[5];
        const float i2 = iota * iota;
        float cE, cV;
        pix_weights(x, E, V, cE, cV);
        const float w1 = cE - 2.f * cV * Es, w2 = cV;
        const float s0 = i2 * q.g0 * q.g0, s1 = i2 * q.g1 * q.g1;
        v[1 + Y_A0] += w1 * f0 + w2 * el20 * s0;
        v[1 + Y_A1] += w1 * f1 + w2 * el21 * s1;
        v[1 + Y_EL0] += w1 * a0 * iota * q.g0;
        v[1 + Y_EL20] += w2 * a0 * s0;
        v[1 + Y_EL1] += w1 * a1 * iota * q.g1;
        v[1 + Y_EL21] += w2 * a1 * s1;
        const float u0 = a0 * iota * (w1 * el0 + 2.f * w2 * iota * el20 * q.g0);
        const float u1 = a1 * iota * (w1 * el1 + 2.f * w2 * iota * el21 * q.g1);
        v[1 + Y_MX] += u0 * q.gx0 + u1 * q.gx1;
        v[1 + Y_MY] += u0 * q.gy0 + u1 * q.gy1;
        v[1 + Y_EDEV] += u1 * q.de;
        v[1 + Y_GXX] += 0.5f * u1 * q.sxx;
        v[1 + Y_GXY] += u1 * q.sxy;
        v[1 + Y_GYY] += 0.5f * u1 * q.syy;
    }
}

// ---------------------------------------------------------------------------------
// launch arguments

struct ItemArgs {
    const ZTask* tasks;
    int n_task;
    const ZBuild* torder;      // the patches' build records, in the order the items first read them
    const ZCand* cands;
    const float4* px;          // pixel records (column, row in the patch, counts, sky)
    const ModelDev* md;
    const double* theta;
    float* ztbl;               // [patch][ZFULL] tables
    float4* zchain;            // [patch][ZCHAIN] chain-rule records
    int32_t* ready;            // [patch] table ready flags, then the queue counter and the
                               // count of built tables; all 0 between evaluations
    const ImgMeta* img_tab;
    double* part;              // [item][16] sums: ll, owned ll, d ll / d y
    const int32_t* item_off;   // [n_patch + 1] first item of each patch
    int ne, nd;                // exp / dev profile components
    int n_patch, n_src;
    int64_t n_sp;              // pixel records (bounds checks)
    int n_zcand, n_sitem, n_img_rec;
    double* kl;
    double* kl_grad;
    int32_t* status;           // the evaluation's status, 0 between evaluations
    int32_t* status_out;       // where the epilogue kernel leaves it
    int mode;
    const int32_t* patch_off;  // [n_src + 1] first patch of each source
    int32_t* grp_done;         // [0]: finished sources of the epilogue kernel, 0 between evaluations
    double* src_total;         // [n_src] each source's share of the total (epilogue kernel)
    double* local_out;
    double* grad_out;
    double* total_out;
};

// ---------------------------------------------------------------------------------
// per-source epilogue and the total

__device__ __forceinline__ double warp_dsum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// an arrival counter increment with release (this thread's, and what it has seen of its
// CTA's, writes become visible first) and acquire (the other arrivals' writes become
// visible to the caller) at gpu scope; returns the count before it
__device__ __forceinline__ int arrive_acq_rel(int32_t* ctr) {
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(ctr) : "memory");
    return old;
}


// ---------------------------------------------------------------------------------
// tasks of the compute warps

// The sums over a warp's lanes of N <= 16 values, each along the same tree (FP32); value j is
// returned on the lanes 2 j and 2 j + 1.  Halving the values with each exchange takes 16 shuffles
// for 16 values instead of 80.
template <int N>
__device__ __forceinline__ float warp_sums(const float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    float r[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) r[j] = j < N ? v[j] : 0.f;
#pragma unroll
    for (int h = 8; h >= 1; h >>= 1) {
        const bool up = lane & (2 * h);
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const float keep = up ? r[j + h] : r[j], send = up ? r[j] : r[j + h];
            r[j] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, 2 * h));
        }
    }
    return __fadd_rn(r[0], __shfl_xor_sync(0xffffffffu, r[0], 1));
}

// float -> double without the FP64 pipe (whose conversions take as long as its arithmetic)
// unless a lane holds a denormal, an infinity or a NaN.  Every lane calls it.
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f), e = b & 0x7f800000u;
    if (__any_sync(0xffffffffu, e == 0x7f800000u || (e == 0 && (b << 1) != 0))) return (double)f;
    const unsigned hi = ((b & 0x7fffffffu) >> 3) + 0x38000000u;
    return __hiloint2double((int)((b & 0x80000000u) | (e ? hi : 0u)), (int)(b << 29));
}

// An item's record from its chunks' sums: FP64, lanes c and c + 16 column c of every other
// chunk, then the two added
template <int MODE>
__device__ __forceinline__ void item_record(const ItemArgs& a, int out, const float* red, int nch) {
    const int lane = threadIdx.x & 31, col = lane & 15, half = lane >> 4;
    constexpr int NS = (MODE == MODE_LL) ? 2 : 2 + NY;
    float r[Lay::nch / 2];
#pragma unroll
    for (int u = 0; u < Lay::nch / 2; ++u) r[u] = col < NS && 2 * u + half < nch ? red[(2 * u + half) * 16 + col] : 0.f;
    double y = widen(r[0]);
#pragma unroll
    for (int u = 1; u < Lay::nch / 2; ++u)
        if (2 * u < nch) y += widen(r[u]);
    y += __shfl_xor_sync(0xffffffffu, y, 16);
    if (lane < NS) a.part[(size_t)out * 16 + lane] = y;
}

// One chunk of an item on a warp: the 32 PX pixels from c0 on (PX consecutive ones per
// thread).  A chunk that holds multiply covered pixels (warp-uniform) stashes its derivatives
// in shared memory while the other covering patches are evaluated.  The chunk's FP32 sums
// (ll, owned ll, d ll / d y) go to rec.
template <int MODE, int NPE, int NPD, int UNR>
__device__ __forceinline__ void chunk_compute(const ItemArgs& a, const ZItem& it, const uint8_t* stage, int c0,
                                              float* spg, float* rec) {
    constexpr int NV = (MODE == MODE_LL) ? 1 : 1 + NY;   // ll (+ d ll / d y)
    const int lane = threadIdx.x & 31;
    const int n = it.n_nm & 0xffff, nm = it.n_nm >> 16;
    const int npsf = it.nc_npsf >> 24, nc = it.nc_npsf & 0xffffff;
    const int npe = (a.ne + 1) >> 1, npd = (a.nd + 1) >> 1;
    const float* T = reinterpret_cast<const float*>(stage + ST_TBL);
    const float4* pxr = reinterpret_cast<const float4*>(stage + ST_PX);
    const ZCand* zc = reinterpret_cast<const ZCand*>(stage + ST_ZC);
    const float* vrec = reinterpret_cast<const float*>(stage + ST_VREC);
    float X[PX], Y[PX], xv[PX], sky[PX];
    bool ok[PX];
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        const int l = c0 + lane * PX + p;
        ok[p] = l < n;
        const float4 r = pxr[ok[p] ? l : n - 1];
        X[p] = r.x;
        Y[p] = r.y;
        xv[p] = r.z;
        sky[p] = r.w;
    }
    float Es[PX], Vs[PX], f0[PX], f1[PX];
    ProfileGrad pg[PX];
    own_source<MODE, NPE, NPD, UNR>(T, npsf, npe, npd, X, Y, Es, Vs, f0, f1, pg);
    float E[PX], V[PX];
    bool owner[PX];
    if (c0 < nm) {
        // E and Var over every covering source in ascending source order; the item's
        // own source enters at its place
        if constexpr (MODE >= MODE_GRAD) {
#pragma unroll
            for (int p = 0; p < PX; ++p) {
                const float* q = reinterpret_cast<const float*>(&pg[p]);
#pragma unroll
                for (int f = 0; f < PG_F; ++f) spg[(p * PG_F + f) * NTC] = q[f];
            }
        }
        bool added = false;
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            E[p] = sky[p];
            V[p] = 0.f;
            owner[p] = true;
        }
        for (int ci = 0; ci < nc; ++ci) {
            const ZCand c = ci < ZSTAGE ? zc[ci] : a.cands[it.c0 + ci];
            const float* R = ci < ZSTAGE ? vrec + ci * VFULL : a.ztbl + (size_t)c.patch * ZFULL;
            if (!added && c.src > it.src) {
#pragma unroll
                for (int p = 0; p < PX; ++p) {
                    E[p] = __fadd_rn(E[p], Es[p]);
                    V[p] = __fadd_rn(V[p], Vs[p]);
                }
                added = true;
            }
            float Xc[PX], Yc[PX];
            bool in[PX], any = false;
#pragma unroll
            for (int p = 0; p < PX; ++p) {
                const int xx = (int)X[p] - c.dx, yy = (int)Y[p] - c.dy;
                in[p] = ok[p] && xx >= 0 && xx < c.w && yy >= 0 && yy < c.h;
                Xc[p] = (float)xx;
                Yc[p] = (float)yy;
                any = any || in[p];
                if (in[p] && c.src < it.src) owner[p] = false;
            }
            if (!__any_sync(0xffffffffu, any)) continue;
            float G0[PX], G1[PX];
            profile_value<NPE, NPD>(R, c.npsf, npe, npd, Xc, Yc, G0, G1);
#pragma unroll
            for (int p = 0; p < PX; ++p) {
                float q0, q1, ec, vc;
                source_ev(R, G0[p], G1[p], q0, q1, ec, vc);
                if (in[p]) {
                    E[p] = __fadd_rn(E[p], ec);
                    V[p] = __fadd_rn(V[p], vc);
                }
            }
        }
        if (!added)
#pragma unroll
            for (int p = 0; p < PX; ++p) {
                E[p] = __fadd_rn(E[p], Es[p]);
                V[p] = __fadd_rn(V[p], Vs[p]);
            }
        if constexpr (MODE >= MODE_GRAD) {
#pragma unroll
            for (int p = 0; p < PX; ++p) {
                float* q = reinterpret_cast<float*>(&pg[p]);
#pragma unroll
                for (int f = 0; f < PG_F; ++f) q[f] = spg[(p * PG_F + f) * NTC];
            }
        }
    } else {
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            E[p] = __fadd_rn(sky[p], Es[p]);
            V[p] = Vs[p];
            owner[p] = true;
        }
    }
    float v[NV + 1];
#pragma unroll
    for (int i = 0; i <= NV; ++i) v[i] = 0.f;
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        if (!ok[p]) continue;
        float vv[NV], ll;
#pragma unroll
        for (int i = 0; i < NV; ++i) vv[i] = v[i];
        pixel_terms<MODE, NV>(T, xv[p], E[p], V[p], Es[p], f0[p], f1[p], pg[p], vv, ll);
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = vv[i];
        if (owner[p]) v[NV] += ll;
    }
    float c[NV + 1];
    c[0] = v[0];
    c[1] = v[NV];
#pragma unroll
    for (int i = 1; i < NV; ++i) c[1 + i] = v[i];
    const float r = warp_sums(c);
    if (!(lane & 1) && (lane >> 1) <= NV) rec[lane >> 1] = r;
}

// the KL value and gradient of source s on one warp (with the domain check of its theta)
__device__ __forceinline__ void kl_task(const ItemArgs& a, int s, float* scr) {
    const int lane = threadIdx.x & 31;
    double* kth = reinterpret_cast<double*>(scr);
    double* kg = kth + NP;
    float* kthr = reinterpret_cast<float*>(kg + NP);
    for (int i = lane; i < NP; i += 32) {
        const double v = a.theta[(size_t)NP * s + i];
        kth[i] = v;
        kthr[i] = (float)v;
        theta_domain_check(i, v, a.status);
    }
    __syncwarp();
    const double v = kl_warp<float>(*a.md, kth, kthr, kg);
    __syncwarp();
    if (lane == 0) a.kl[s] = v;
    for (int i = lane; i < NP; i += 32) a.kl_grad[(size_t)NP * s + i] = kg[i];
}

// ---------------------------------------------------------------------------------
// staging the items

// the 64-byte record of queue slot q, a quarter per lane 0 .. 3 (past the end: an end
// marker)
__device__ __forceinline__ int4 load_task(const ItemArgs& a, int q) {
    const int lane = threadIdx.x & 31;
    if (q >= a.n_task) return make_int4(ZT_END, 0, 0, 0);
    return lane < 4 ? __ldcg(reinterpret_cast<const int4*>(a.tasks + q) + lane) : make_int4(0, 0, 0, 0);
}

// Put a task record (lanes 0 .. 3) in a stage and, for an item, wait for the tables it
// reads and start the bulk copies of its data into the stage; the stage's full barrier
// completes when they land (at once for the end marker).  Whole warp, every lane one of
// the item's patches (lane 0 its own, lane 1 + e candidate e), so that the patch ids,
// the ready flags and the copies of the candidates' value records take one memory round
// trip each instead of one per candidate.  all_built (every lane): every table was seen
// built, so no flag need be read.
template <int MODE>
__device__ void prepare(const ItemArgs& a, int4 rec, uint8_t* stage, ZTask* tk, uint64_t* full, bool& all_built) {
    const int lane = threadIdx.x & 31;
    const unsigned fullmask = 0xffffffffu;
    if (lane < 4) reinterpret_cast<int4*>(tk)[lane] = rec;
    __syncwarp();
    if (tk->kind != ZT_ITEM) {
        if (lane == 0) mbar_arrive_plain(full);
        return;
    }
    const ZItem it = tk->item;
    const int n = it.n_nm & 0xffff, nc = it.nc_npsf & 0xffffff, nc0 = nc < ZSTAGE ? nc : ZSTAGE;
    // candidate e's patch: named in the record for e < ZMAXC, else in the candidate list
    auto cand_patch = [&](int e) { return e < ZMAXC ? tk->cand[e] : a.cands[it.c0 + e].patch; };
#ifdef CELESTE_CHECK_BOUNDS
    {
        // the record's offsets into the pixel records, candidates, tables and item records;
        // a bad record ends this CTA's work (the status tells the caller)
        const int nm = it.n_nm >> 16, npsf = it.nc_npsf >> 24;
        bool ok = it.patch >= 0 && it.patch < a.n_patch && n >= 1 && n <= ZIMAX && nm <= n && it.pix >= 0 &&
                  it.pix + n <= a.n_sp && it.c0 >= 0 && (int64_t)it.c0 + nc <= a.n_zcand && it.out >= 0 &&
                  it.out < a.n_sitem && it.src >= 0 && it.src < a.n_src && npsf >= 1 && npsf <= MAXPSF;
        for (int j = lane; ok && j <= nc; j += 32) {
            const int pe = j == 0 ? it.patch : cand_patch(j - 1);
            ok = pe >= 0 && pe < a.n_patch;
        }
        ok = __all_sync(fullmask, ok);
        if (!ok) {
            if (lane == 0) {
                CEL_IN_BOUNDS(false, a.status);
                tk->kind = ZT_END;
                mbar_arrive_plain(full);
            }
            return;
        }
    }
#endif
    // this lane's patch: 0 the item's own, 1 + e candidate e (staged ones: e < nc0 <= 31)
    const int pl = lane == 0 ? it.patch : (lane - 1 < nc ? cand_patch(lane - 1) : -1);
    if (!all_built) {
        // lane 0 reads the built counter while the lanes read the flags of their patches
        bool built = false;
        if (lane == 0) built = load_acquire(a.ready + a.n_patch + 1) >= a.n_patch;
        else if (pl >= 0) wait_ready(a.ready + pl, a.status);
        for (int j = lane + 32; j <= nc; j += 32) wait_ready(a.ready + cand_patch(j - 1), a.status);
        if (lane == 0 && !built) wait_ready(a.ready + it.patch, a.status);
        all_built = __shfl_sync(fullmask, built, 0);
    }
    __syncwarp();
    // lane 0 announces the bytes before any copy is issued
    const unsigned tbl_bytes = MODE == MODE_LL ? VFULL * 4 : ZFULL * 4;
    if (lane == 0) {
        const unsigned bytes =
            tbl_bytes + (unsigned)n * 16u + (unsigned)nc0 * (unsigned)(sizeof(ZCand) + VFULL * 4);
        mbar_expect_arrive(full, bytes);
    }
    __syncwarp();
    fence_proxy_async_global();
    fence_proxy_async_smem();   // the stage was last read through the generic proxy
    if (lane == 0) {
        bulk_g2s_tx(stage + ST_TBL, a.ztbl + (size_t)it.patch * ZFULL, tbl_bytes, full);
        bulk_g2s_tx(stage + ST_PX, a.px + it.pix, (unsigned)n * 16u, full);
        if (nc0 > 0) bulk_g2s_tx(stage + ST_ZC, a.cands + it.c0, (unsigned)nc0 * (unsigned)sizeof(ZCand), full);
    } else if (lane - 1 < nc0) {
        bulk_g2s_tx(stage + ST_VREC + (lane - 1) * VFULL * 4, a.ztbl + (size_t)pl * ZFULL, VFULL * 4, full);
    }
}

// ---------------------------------------------------------------------------------
// the kernels

// Tables and KL terms, a warp each in turn while there are both: the tables and chain-rule
// records of the patches torder[0 .. n_patch) (the patches in the order the items first read
// them), 32 / LP per warp, published when built; the KL terms of a source (with the domain check
// of its theta).  The item kernel is launched as this kernel's programmatic dependent and
// waits for each table's flag, not for this kernel.
// Bound by instruction issue where a warp builds one table (most of its lanes repeat the same
// set-up) and, once the patches are more than the chip's warps, by the KL terms' FP64 pipe time,
// which therefore runs beside the tables and not behind them.  A warp for four patches takes 2.4
// times fewer instructions per patch but is slower for each.  Stage times: 15,625 patches of
// 3,125 sources 47 us with a warp per patch and the KL terms last, 38 with both in turn, 31 with
// four patches per warp too; 8,000 patches of 100 sources 26, 21, 20; 2,500 patches of 500
// sources 15.4 with one patch per warp, 16.7 with four.
template <int LP>
__global__ void __launch_bounds__(128) k_tables(ItemArgs a) {
    __shared__ __align__(16) float scr[4][SCR_W / 4 * (LP == 32 ? 1 : 2)];
    constexpr int PW = 32 / LP;   // patches per warp
    static_assert(PW * 96 * 4 <= sizeof(scr[0]), "scratch of the warp's patches");
    pdl_trigger();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_warp = (a.n_patch + PW - 1) / PW, both = 2 * min(n_warp, a.n_src), v = (int)blockIdx.x * 4 + w;
    const bool table = v < both ? !(v & 1) : n_warp > a.n_src;
    const int u = v < both ? v >> 1 : v - (both >> 1);
    if (table && u < n_warp) {
        const int t = u * PW + lane / LP;
        const ZBuild g = a.torder[min(t, a.n_patch - 1)];
        const bool live = t < a.n_patch && CEL_IN_BOUNDS(g.patch >= 0 && g.patch < a.n_patch && g.img >= 0 &&
                                                             g.img < a.n_img_rec && g.src >= 0 && g.src < a.n_src,
                                                         a.status);
        if (!__any_sync(0xffffffffu, live)) return;
        ZBuild gs = g;
        if (!live) gs = ZBuild{0, 0, 0, 0, 0.0, 0.0};   // (indices in range; nothing is stored)
        build_patch_table<LP>(a.theta, gs, live, a.img_tab, *a.md, a.ztbl, a.zchain, scr[w] + 96 * (lane / LP));
        __syncwarp();
        if (live && lane % LP == 0) publish_ready(a.ready + g.patch, a.ready + a.n_patch + 1);
    } else if (!table && u < a.n_src) {
        kl_task(a, u, scr[w]);
    }
}

// The per-source epilogues and the total, after every item: the item kernel's
// programmatic dependent, waiting for it to finish.  One CTA of W warps per source:
// warp w takes the source's patches w, w + W, ...: the FP64 sums of the patch's item records
// (lanes c and c + 16 column c of every other item, then the two added), then the patch's
// chain rule (lane j < ZCHAIN: column j of d ll / d theta += sum_e k_e d ll / d y_{y_e};
// the next two lanes the ll and the owned ll).  The CTA then adds the warps' sums in warp order
// and subtracts the KL: the local objective and gradient, and the source's share of the total
// (the ll of the pixels its items own, minus its KL).  The last CTA to finish adds the shares
// in source order (its warps over contiguous ranges, lanes strided, then warp order).  The
// kernel leaves the flags, counters and the status word of the evaluation at 0 for the next one
// (the status goes to the caller's word), so an evaluation is three kernels and nothing else:
// two fills of a few bytes ahead of them cost an evaluation 2 us.
//
// Bound by the latency of its loads and of about ten dependent FP64 operations per patch; the next
// patch's records are loaded ahead.  The chain rule stands here, once per patch, and not in the
// item kernel, once per item, where its ~30 FP64 operations delayed the warp that has to
// stage the next item.
// W warps per CTA: on one source (SHARED), or each on a source of its own.  FIN_C: item records
// loaded ahead per lane.
template <int W, int FIN_C, bool SHARED>
__global__ void __launch_bounds__(32 * W, 32 / W) k_finish(ItemArgs a) {
    __shared__ double sh[W][32];
    __shared__ int s_last;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = SHARED ? (int)blockIdx.x : (int)blockIdx.x * W + w;
    constexpr int STEP = SHARED ? W : 1;   // this warp's patches: p0 + w (SHARED) or p0, STEP apart
    const bool grad = a.mode >= MODE_GRAD;
    const int col = lane & 15, half = lane >> 4;
    const bool used = col < (grad ? 2 + NY : 2), valid = s < a.n_src;
    int p0 = valid ? a.patch_off[s] : 0, p1 = valid ? a.patch_off[s + 1] : 0;
    if (!CEL_IN_BOUNDS(p0 >= 0 && p0 <= p1 && p1 <= a.n_patch, a.status)) p0 = p1 = 0;
    if (SHARED) p0 += w;
    int o0 = 0, o1 = 0;   // the items of patch pl, one of this warp's next 32
    auto offsets = [&](int pl) {
        o0 = o1 = 0;
        if (pl >= p1) return;
        o0 = a.item_off[pl];
        o1 = a.item_off[pl + 1];
        if (!CEL_IN_BOUNDS(o0 >= 0 && o0 <= o1 && o1 <= a.n_sitem, a.status)) o0 = o1 = 0;
    };
    offsets(p0 + STEP * lane);
    if (threadIdx.x == 0) s_last = 0;
    if (!SHARED) __syncthreads();
    pdl_wait();
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); i < a.n_patch + 2; i += (int)(gridDim.x * blockDim.x))
        a.ready[i] = 0;
    // (the KL terms, asked for early)
    double klv = 0.0, kg0 = 0.0, kg1 = 0.0;
    if (valid && (!SHARED || w == 0)) {
        const double* kg = a.kl_grad + (size_t)NP * s;
        klv = __ldcg(a.kl + s);
        if (grad) {
            kg0 = __ldcg(kg + lane);
            if (lane < NP - ZCHAIN) kg1 = __ldcg(kg + ZCHAIN + lane);
        }
    }
    double acc = 0.0;
    for (int pb = p0; pb < p1; pb += 32 * STEP) {
        const int np = min(32, (p1 - pb + STEP - 1) / STEP);
        if (pb != p0) offsets(pb + STEP * lane);
        double x[FIN_C];
        float4 ch;
        auto records = [&](int c0, int c1, double (&v)[FIN_C]) {
#pragma unroll
            for (int u = 0; u < FIN_C; ++u) {
                const int c = c0 + 2 * u + half;
                v[u] = used && c < c1 ? __ldcg(a.part + (size_t)c * 16 + col) : 0.0;
            }
        };
        auto load = [&](int i) {
            records(__shfl_sync(0xffffffffu, o0, i), __shfl_sync(0xffffffffu, o1, i), x);
            ch = make_float4(lane < ZCHAIN ? 0.f : 1.f, 0.f, 0.f, 0.f);
            if (grad && lane < ZCHAIN) ch = __ldcg(a.zchain + (size_t)(pb + STEP * i) * ZCHAIN + lane);
        };
        load(0);
        for (int i = 0; i < np; ++i) {
            const int c0 = __shfl_sync(0xffffffffu, o0, i), c1 = __shfl_sync(0xffffffffu, o1, i);
            const float4 k = ch;
            double v[FIN_C];
#pragma unroll
            for (int u = 0; u < FIN_C; ++u) v[u] = x[u];
            if (i + 1 < np) load(i + 1);
            double y = v[0];
#pragma unroll
            for (int u = 1; u < FIN_C; ++u)
                if (c0 + 2 * u < c1) y += v[u];
            for (int b = c0 + 2 * FIN_C; b < c1; b += 2 * FIN_C) {   // patches of more items
                records(b, c1, v);
#pragma unroll
                for (int u = 0; u < FIN_C; ++u)
                    if (b + 2 * u < c1) y += v[u];
            }
            if (c1 - c0 > 1) y += __shfl_xor_sync(0xffffffffu, y, 16);
            const int yy = __float_as_int(k.w);
            const bool lls = lane >= ZCHAIN;   // the ll and the owned ll: columns 0 and 1
            const double y0 = __shfl_sync(0xffffffffu, y, lls ? (lane - ZCHAIN) & 1 : 2 + (yy & 15));
            const double y1 = __shfl_sync(0xffffffffu, y, 2 + ((yy >> 4) & 15));
            const double y2 = __shfl_sync(0xffffffffu, y, 2 + ((yy >> 8) & 15));
            const double k0 = widen(k.x), k1 = widen(k.y), k2 = widen(k.z);
            acc = fma(k0, y0, acc);
            if (!lls) acc = fma(k2, y2, fma(k1, y1, acc));
        }
    }
    if (SHARED) {
        sh[w][lane] = acc;
        __syncthreads();
    }
    if (valid && (!SHARED || w == 0)) {
        double t = acc;
        if (SHARED) {
            double r[W];
#pragma unroll
            for (int v = 0; v < W; ++v) r[v] = sh[v][lane];
#pragma unroll
            for (int h = W / 2; h >= 1; h >>= 1)
#pragma unroll
                for (int v = 0; v < h; ++v) r[v] += r[v + h];
            t = r[0];
        }
        if (lane == ZCHAIN && a.local_out) a.local_out[s] = t - klv;
        if (grad && a.grad_out) {
            double* g = a.grad_out + (size_t)NP * s;
            if (lane < ZCHAIN) g[lane] = t - kg0;
            if (lane < NP - ZCHAIN) g[ZCHAIN + lane] = -kg1;
        }
        if (lane == ZCHAIN + 1) {
            if (a.total_out) a.src_total[s] = t - klv;
            if (SHARED) s_last = arrive_acq_rel(a.grp_done) == (int)gridDim.x - 1;
        }
    }
    if (!SHARED) {
        __syncthreads();
        if (threadIdx.x == 0) s_last = arrive_acq_rel(a.grp_done) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    if (threadIdx.x == 0) {
        *a.status_out = *reinterpret_cast<volatile int32_t*>(a.status);
        *a.status = 0;
        a.grp_done[0] = 0;
    }
    if (!a.total_out) return;
    const int n = a.n_src, per = (n + W - 1) / W;
    const int b0 = w * per, b1 = min(n, b0 + per);
    double tot = 0.0;
    for (int c0 = b0; c0 < b1; c0 += 32 * 16) {
        double x[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int i = c0 + lane + 32 * u;
            x[u] = i < b1 ? __ldcg(a.src_total + i) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) tot += x[u];
    }
    tot = warp_dsum(tot);
    __syncthreads();   // every warp is past its reads of sh
    if (lane == 0) sh[w][0] = tot;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int v = 0; v < W; ++v) t += sh[v][0];
        *a.total_out = t;
    }
}

// Fetch the record of queue slot q ahead (lane 0): a bulk copy into rec completing on bar, or
// an end marker past the end.
__device__ __forceinline__ void fetch_record(const ItemArgs& a, int q, ZTask* rec, uint64_t* bar) {
    if (q >= a.n_task) {
        rec->kind = ZT_END;
        mbar_arrive_plain(bar);
        return;
    }
    fence_proxy_async_smem();   // rec was last read through the generic proxy
    mbar_expect_arrive(bar, (unsigned)sizeof(ZTask));
    bulk_g2s_tx(rec, a.tasks + q, (unsigned)sizeof(ZTask), bar);
}

// The items, on persistent CTAs of four warps that keep the next two items in two stages.
// The warps take an item's chunks in turn from a counter in shared memory and go on to the next
// item when none is left; the one that leaves item i last puts item i + 2, whose record was
// fetched before, in that stage and fetches the record of item i + 3.  CTA c's first two items are slots c and c + G
// (G CTAs); later slots come from the queue counter.
//
// Bound by the FMA pipe and by instruction issue (60% and 67% busy).  Four CTAs per SM at 128
// registers hold 16 computing warps, and the 7 component pairs of 2 pixels still unroll without
// spilling.  For 8.7 million source-pixels in a dense field: two CTAs per SM of four warps and a
// fifth for the staging and the records 444 us; the fifth warp's work on the warp that finishes
// last, three CTAs, chunks dealt out by warp number 434 (a quarter of the warps' time went on
// waiting for the slowest); chunks taken in turn 391; four CTAs 360; whole chunks per item 354;
// pixels grouped by covering set 336; the chain rule moved to k_finish 328.
template <int MODE, int NPE, int NPD, int MINB, int UNR>
__global__ void __launch_bounds__(NTC) __maxnreg__(regs_for(MINB)) k_items(ItemArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    using L = Lay;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::bar);
    uint64_t* fetched = full + 2;
    ZTask* tasks = reinterpret_cast<ZTask*>(smem + L::task);
    float* red = reinterpret_cast<float*>(smem + L::red);
    ZTask* next = reinterpret_cast<ZTask*>(smem + L::next);
    int* cnt = reinterpret_cast<int*>(smem + L::cnt);
    int* taken = cnt + 2;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    pdl_trigger();   // the epilogue kernel may start (it waits for this grid to finish)
    if (t == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&full[b], 1);
            mbar_init(&fetched[b], 1);
            cnt[b] = taken[b] = 0;
        }
        mbar_init_fence();
    }
    __syncthreads();
    int32_t* queue = a.ready + a.n_patch;
    // slots 0 .. 2 G - 1 (G CTAs) are dealt out, one per stage of every CTA, so that a queue
    // of few items spreads over all CTAs; the rest are claimed one at a time
    const int G = (int)gridDim.x, base = 2 * G;
    bool all_built = false;
    if (w < 2)
        prepare<MODE>(a, load_task(a, (int)blockIdx.x + w * G), smem + w * ST_BYTES, &tasks[w], &full[w], all_built);
    else if (w == 2 && lane == 0)
        fetch_record(a, base + atomicAdd(queue, 1), &next[0], &fetched[0]);
    float* spg = reinterpret_cast<float*>(smem + L::pg) + t;
    int stopped = -1;   // the item at which a wait gave up
    for (int i = 0;; ++i) {
        const int b = i & 1;
        __syncwarp();
        if (!mbar_wait_launch(&full[b], (i >> 1) & 1, a.status)) {
            stopped = i;
            break;
        }
        if (tasks[b].kind == ZT_END) break;
        const ZItem it = tasks[b].item;
        uint8_t* stage = smem + b * ST_BYTES;
        float* rb = red + b * L::nch * 16;
        const int nch = ((it.n_nm & 0xffff) + ZCHUNK - 1) / ZCHUNK;
        for (;;) {
            int c = 0;
            if (lane == 0) c = atomicAdd(&taken[b], 1);
            c = __shfl_sync(0xffffffffu, c, 0);
            if (c >= nch) break;
            chunk_compute<MODE, NPE, NPD, UNR>(a, it, stage, c * ZCHUNK, spg, rb + c * 16);
        }
        __syncwarp();
        int last = 0;
        if (lane == 0) {
            __threadfence_block();
            last = atomicAdd(&cnt[b], 1) == NWC - 1;
            if (last) cnt[b] = taken[b] = 0;
            __threadfence_block();
        }
        if (!__shfl_sync(0xffffffffu, last, 0)) continue;
        int q = 0;
        if (lane == 0) q = base + atomicAdd(queue, 1);
        item_record<MODE>(a, it.out, rb, nch);
        if (!mbar_wait_launch(&fetched[b], (i >> 1) & 1, a.status)) {
            stopped = i;
            break;
        }
        const int4 rec = lane < 4 ? reinterpret_cast<const int4*>(&next[b])[lane] : make_int4(0, 0, 0, 0);
        __syncwarp();
        prepare<MODE>(a, rec, stage, &tasks[b], &full[b], all_built);
        if (lane == 0) fetch_record(a, q, &next[b ^ 1], &fetched[b ^ 1]);
    }
    if (stopped >= 0) drain(full, fetched, stopped);
    // this grid completes only after the table kernel (and its KL terms) has, so the epilogue
    // kernel that waits for this grid sees both
    if (w == 0) pdl_wait();
}

// ---------------------------------------------------------------------------------
// launch

template <int MODE, int NPE, int NPD, int MINB, int UNR>
struct ItemsKernel {
    // Resident CTAs per SM on the current device, its shared-memory limit raised first (both are
    // a device's own: the limit holds on the device it was set on).  0: an error, in *err.
    static int per_sm(cudaError_t* err) {
        static PerDevice on;
        *err = cudaSuccess;
        return on.get([&](int) {
            auto* fn = k_items<MODE, NPE, NPD, MINB, UNR>;
            cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay::bytes);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
            int per = 0;
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, NTC, Lay::bytes);
            *err = e;
            return e != cudaSuccess ? 0 : per > 0 ? per : 1;
        });
    }
    // a programmatic dependent launch of the table kernel before it on st
    static cudaError_t launch(const ItemArgs& a, int n_sm, cudaStream_t st) {
        cudaError_t e;
        int grid = per_sm(&e) * n_sm;
        if (e != cudaSuccess) return e;
        if (grid > a.n_task) grid = a.n_task;
        if (grid < 1) return cudaSuccess;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(NTC);
        cfg.dynamicSmemBytes = Lay::bytes;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, k_items<MODE, NPE, NPD, MINB, UNR>, a);
    }
};
// the model of the synthetic workloads and of the paper (6 exp + 8 dev profile
// components: 3 + 4 pairs) gets its loops unrolled for those counts
template <int MODE, int MINB, int UNR>
cudaError_t items_launch_v(const ItemArgs& a, int n_sm, cudaStream_t st) {
    if ((a.ne + 1) / 2 == 3 && (a.nd + 1) / 2 == 4) return ItemsKernel<MODE, 3, 4, MINB, UNR>::launch(a, n_sm, st);
    return ItemsKernel<MODE, -1, -1, MINB, 1>::launch(a, n_sm, st);
}

#define CEL_ITEM_VARIANTS(X) \
    X(1, 4, 7)               \
    X(2, 3, 7)               \
    X(3, 4, 2)               \
    X(4, 4, 3)               \
    X(5, 3, 3)
// variant codes (code, CTAs per SM, unroll of the component-pair loop)
template <int MODE>
cudaError_t items_launch(const ItemArgs& a, int code, int n_sm, cudaStream_t st) {
    switch (code) {
#define CEL_CASE(c, minb, unr) \
    case c: return items_launch_v<MODE, minb, unr>(a, n_sm, st);
        CEL_ITEM_VARIANTS(CEL_CASE)
#undef CEL_CASE
        default: return items_launch_v<MODE, 4, 7>(a, n_sm, st);
    }
}

template <int MODE>
cudaError_t items_setup_mode() {
    cudaError_t e = cudaSuccess;
#define CEL_SETUP(c, minb, unr)                                                    \
    if (e == cudaSuccess) ItemsKernel<MODE, 3, 4, minb, unr>::per_sm(&e);            \
    if (e == cudaSuccess) ItemsKernel<MODE, -1, -1, minb, 1>::per_sm(&e);
    CEL_ITEM_VARIANTS(CEL_SETUP)
#undef CEL_SETUP
    return e;
}

}  // namespace

// shared-memory limits and resident CTAs of every item-kernel variant on the current device, set
// once per device outside any stream capture
cudaError_t prime_items_kernels() {
    cudaError_t e = items_setup_mode<MODE_LL>();
    if (e == cudaSuccess) e = items_setup_mode<MODE_GRAD>();
    return e;
}

static cudaError_t launch_stage(const DevProblem& P, int stage, int mode, cudaStream_t st, const double* d_theta,
                                double* d_local, double* d_grad, double* d_total) {
    if (P.n_src == 0 || !P.ztasks) return cudaSuccess;
    ItemArgs a{};
    a.tasks = P.ztasks;
    a.n_task = P.n_task;
    a.torder = P.ztorder;
    a.cands = P.zcands;
    a.px = P.zpx;
    a.md = P.model;
    a.theta = d_theta;
    a.ztbl = P.ztbl;
    a.zchain = P.zchain;
    a.ready = P.zready;
    a.img_tab = P.img;
    a.part = P.zpart;
    a.item_off = P.zitem_off;
    a.ne = P.model_ne;
    a.nd = P.model_nd;
    a.n_patch = P.n_patch;
    a.n_src = P.n_src;
    a.n_sp = P.n_sp;
    a.n_zcand = P.n_zcand;
    a.n_sitem = P.n_sitem;
    a.n_img_rec = P.n_img_rec;
    a.kl = P.kl;
    a.kl_grad = P.kl_grad;
    a.status = P.zf_done + 1;
    a.status_out = P.status;
    a.mode = mode;
    a.patch_off = P.patch_off;
    a.grp_done = P.zf_done;
    a.src_total = P.src_total;
    a.local_out = d_local;
    a.grad_out = mode >= MODE_GRAD ? d_grad : nullptr;
    a.total_out = d_total;
    if (stage == 0) {
        // a warp per patch up to one wave of warps (36 per SM), four patches per warp beyond
        const int pw = P.n_patch > 36 * sm_count() ? 4 : 1, n_warp = (P.n_patch + pw - 1) / pw + P.n_src;
        if (pw == 4) k_tables<8><<<(n_warp + 3) / 4, 128, 0, st>>>(a);
        else k_tables<32><<<(n_warp + 3) / 4, 128, 0, st>>>(a);
        return cudaGetLastError();
    }
    if (stage == 1) {
        const int n_sm = sm_count();
        return mode == MODE_LL ? items_launch<MODE_LL>(a, P.tune_items, n_sm, st)
                               : items_launch<MODE_GRAD>(a, P.tune_items, n_sm, st);
    }
    cudaLaunchConfig_t cfg{};
    // Sixteen warps on a source of many images (a source of 80 images with four: 22 us, sixteen 19),
    // eight on one of a few.  Beyond four waves of eight-warp CTAs a warp takes a source of its own
    // (3125 sources of 5 images: 30 -> 26 us; 1200 sources: 12 -> 17 us, so not below).
    const bool wide = P.n_patch > 8 * (int64_t)P.n_src, shared = wide || P.n_src <= 16 * sm_count();
    cfg.gridDim = dim3((unsigned)(shared ? P.n_src : (P.n_src + 7) / 8));
    cfg.blockDim = dim3(32 * (wide ? 16 : 8));
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (wide) return cudaLaunchKernelEx(&cfg, k_finish<16, 4, true>, a);
    return shared ? cudaLaunchKernelEx(&cfg, k_finish<8, 2, true>, a) : cudaLaunchKernelEx(&cfg, k_finish<8, 2, false>, a);
}

cudaError_t launch_items_stage(const DevProblem& P, int stage, int mode, cudaStream_t st, const double* d_theta,
                               double* d_local, double* d_grad, double* d_total) {
    const cudaError_t e = launch_stage(P, stage, mode, st, d_theta, d_local, d_grad, d_total);
    // tables published without an epilogue kernel behind them must not pass for the next call's (the
    // first stage too: the error that it reports can be one that an earlier call left)
    if (e != cudaSuccess && P.ztasks) {
        cudaMemsetAsync(P.zready, 0, sizeof(int32_t) * ((size_t)P.n_patch + 2), st);
        cudaMemsetAsync(P.zf_done, 0, 2 * sizeof(int32_t), st);
    }
    return e;
}

}  // namespace cel
