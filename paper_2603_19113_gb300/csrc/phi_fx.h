// The fundamental solution phi_kappa (Sec. 3.1, eq. FundamentalSol) to FP64
// accuracy in 64-bit fixed point on the integer multipliers.  Host and device
// code.
//
// GB300 does 32 32x32+64-bit integer multiply-adds per clock and SM (measured)
// and 2 FP64 ones, so a 64 x 64 -> 64 (high half) product from three of them
// costs a fifth of one FP64 multiply-add and keeps more bits.  Distances are taken relative to one source body: with its
// reference point c, radius rho and a target t, D = t - c (FP64, once per
// target and body) and 2^e > |D| + rho, every length is a fraction of 2^e in
// [0, 1) with 62 bits, so the phase kappa r carries 2^-62 kappa 2^e, against
// 2^-53 kappa r of an FP64 product.  Phases are counted in turns modulo 1, so
// the reduction of the argument is the wrap-around of 64-bit integers.
//
// Notation: x62 is a value times 2^62.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "bessel_coeffs.h"

#if defined(__CUDACC__)
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

typedef long long fx_i64;
typedef unsigned long long fx_u64;

// a = h 2^32 + l with both parts signed, as the multiplier takes them
struct fx2 {
    int h, l;
};

FX_HD int fx_hi(fx_i64 a) { return (int)(a >> 32); }
FX_HD unsigned fx_hiu(fx_u64 a) { return (unsigned)(a >> 32); }
// a b + c and the high half of a b.  On the device as explicit wide
// multiply-adds (32 a clock and SM), whatever a compiler makes of 64-bit
// expressions.
FX_HD fx_i64 fx_madw(int a, int b, fx_i64 c) {
#if defined(__CUDA_ARCH__)
    fx_i64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (fx_i64)a * b + c;
#endif
}
FX_HD fx_i64 fx_mulw(int a, int b) {
#if defined(__CUDA_ARCH__)
    fx_i64 d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (fx_i64)a * b;
#endif
}
FX_HD fx_u64 fx_mulwu(unsigned a, unsigned b) {
#if defined(__CUDA_ARCH__)
    fx_u64 d;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (fx_u64)a * b;
#endif
}
FX_HD unsigned fx_mulhu(unsigned a, unsigned b) { return (unsigned)(fx_mulwu(a, b) >> 32); }
FX_HD fx2 fx_split(fx_i64 a) { return fx2{(int)((a + 0x80000000ll) >> 32), (int)a}; }
// a b / 2^64, error below 2; |a| <= 2^62 or |b| <= 2^62
FX_HD fx_i64 fx_mulhi(fx2 a, fx2 b) {
    const fx_i64 m = fx_madw(a.h, b.l, fx_mulw(a.l, b.h));
    return fx_madw(a.h, b.h, fx_hi(m));
}

// a^2 / 2^64, error below 3, not negative
FX_HD fx_i64 fx_square(fx2 a) { return fx_madw(a.h, a.h, fx_madw(fx_hi(fx_mulw(a.h, a.l)), 2, 1)); }

FX_HD float fx_rsqrt(float a) {
#if defined(__CUDA_ARCH__)
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a));
    return y;
#else
    const float y = 1.0f / sqrtf(a);
#if defined(FX_RSQRT_ULP)
    static unsigned n = 0;  // errors of the device's approximation, for the host-side check
    n = n * 1664525u + 1013904223u;
    return y * (1.0f + (float)((int)(n >> 8) % (FX_RSQRT_ULP + 1) - FX_RSQRT_ULP / 2) * 0x1p-24f);
#else
    return y;
#endif
#endif
}
FX_HD int fx_rint(float a) {
#if defined(__CUDA_ARCH__)
    return __float2int_rn(a);
#else
    return (int)lrintf(a);
#endif
}

// 2^e for -1000 < e < 1000, and the e with a < 2^e <= 2 a (normal a > 0)
FX_HD double fx_exp2(int e) {
    const fx_i64 bits = (fx_i64)(e + 1023) << 52;
#if defined(__CUDA_ARCH__)
    return __longlong_as_double(bits);
#else
    double d;
    memcpy(&d, &bits, 8);
    return d;
#endif
}
FX_HD int fx_exponent(double a) {
#if defined(__CUDA_ARCH__)
    const fx_i64 bits = __double_as_longlong(a);
#else
    fx_i64 bits;
    memcpy(&bits, &a, 8);
#endif
    return (int)(bits >> 52) - 1022;
}
FX_HD fx_i64 fx_round(double a) {
#if defined(__CUDA_ARCH__)
    return __double2ll_rn(a);
#else
    return llrint(a);
#endif
}

// a - b = the returned value + lo exactly
FX_HD double fx_diff(double a, double b, double& lo) {
    const double d = a - b, t = d - a;
    lo = (a - (d - t)) - (b + t);
    return d;
}

// 1024 steps of cos and sin of a turn, at 2^62, split
constexpr int FX_TAB = 1024;
struct FxEntry {
    int ch, cl, sh, sl;
};

// Constants of one wavenumber: kappa / (2 pi) = kturn62 2^(kturn_e - 62) and
// 1 / kappa = kinv62 2^(kinv_e - 62), mantissas in [2^61, 2^62)
struct FxKappa {
    fx_i64 kturn62, kinv62;
    int kturn_e, kinv_e;
    double kappa;
    double amp;  // 2D: (1/4) sqrt(2 / (pi kappa)); 3D: 1 / (4 pi)
};

// Per target and source body.
template <int DIM>
struct FxBody {
    fx_i64 X[DIM];  // (t - c) 2^(63 - e) + 2^31 (the rounding of fx_split)
    int sh;         // source offsets are stored at 2^(63 - es): shift by e - es
    fx2 K;          // kappa 2^e / (2 pi), as a mantissa at 2^62
    int ksh;        // left shift of r K to turns at 2^64
    fx2 Ki;         // 2D: 1 / (kappa 2^e) at 2^66
    int up;         // left shift that brings the largest amplitude near 2^61
};

// Lengths below 2^-4 of 2^e would leave the integer formats: such bodies
// (2^e is 2 to 4 times the radius there, so targets within an eighth to a quarter
// of the radius of the hull) and the ranges below go to the FP64 evaluation
// instead.
constexpr double FX_RMIN = 0.0626;  // least r / 2^e

// Constants of a body at offset D + Dl from the target (|D| = R), radius rho, with
// the stored exponent es (rho < 2^es); false: not in the range of the formats.
// scale: phi = scale * (the integers of fx_phi).
template <int DIM>
FX_HD bool fx_body(const FxKappa& k, const double* D, const double* Dl, double R, double rho, int es, FxBody<DIM>& b, double& scale) {
    const double rmax = (R + rho) * (1.0 + 1e-6);
    if (!(rmax > 1e-17 && rmax < 1e18)) return false;  // R comes from FP32 squares, R > rho: normal numbers
    int e = fx_exponent(rmax);
    if (e < es) e = es;
    const double rmin = (R - rho) * (1.0 - 1e-6);
    if (!(rmin >= FX_RMIN * fx_exp2(e))) return false;
    const int j = e + 1 - fx_exponent(rmin);  // r / 2^e >= 2^-j, 1 <= j <= 4
    b.up = DIM == 2 ? (j <= 1 ? 2 : j <= 3 ? 1 : 0) : 5 - j;
    const int ksh = k.kturn_e + e + 4;  // (2^62 2^62 2^-64) 2^ksh = 2^64 / 2^(kturn_e + e)
    if (ksh < -30 || ksh > 40) return false;  // kappa 2^e between 2^-34 and 2^36 turns
    if (DIM == 2) {
        // 1 / (kappa 2^e) at 2^66 below 2^62: kappa 2^e > 16
        const int s = k.kinv_e - e + 4;
        if (s > 0 || s < -40) return false;
        b.Ki = fx_split(k.kinv62 >> -s);
    }
    const double up = fx_exp2(63 - e);
#pragma unroll
    for (int a = 0; a < DIM; ++a) b.X[a] = fx_round(D[a] * up) + fx_round(Dl[a] * up) + 0x80000000ll;
    b.sh = e - es > 63 ? 63 : e - es;
    b.ksh = ksh > 0 ? ksh : 0;
    b.K = fx_split(ksh < 0 ? k.kturn62 >> -ksh : k.kturn62);
    // fx_phi returns the amplitude relative to that at r = 2^e times 2^(56 + up) (2D) or 2^(54 + up) (3D)
    if (DIM == 2)
        scale = k.amp * ((e & 1) ? 0.70710678118654752440 * fx_exp2(-(e - 1) / 2 - 56 - b.up) : fx_exp2(-e / 2 - 56 - b.up));
    else
        scale = k.amp * fx_exp2(-e - 54 - b.up);
    return true;
}

// Two polynomials in u (|u| <= 1, at 2^62) with coefficients at 2^62, highest
// first; side by side, so that each hides the other's latency
FX_HD void fx_horner2(const fx_i64* cf, const fx_i64* cg, int deg, fx2 u, fx_i64& f, fx_i64& g) {
    f = cf[0];
    g = cg[0];
#pragma unroll 2
    for (int k = 1; k <= deg; ++k) {
        f = (fx_mulhi(fx_split(f), u) << 2) + cf[k];
        g = (fx_mulhi(fx_split(g), u) << 2) + cg[k];
    }
}

#if defined(__CUDACC__)
#define FX_CONST __device__ __constant__ const
#else
#define FX_CONST static const
#endif
// fits of bessel_coeffs.h, f - 1 and g / 2 pi, at 2^62
template <int N>
struct FxTab {
    fx_i64 c[N];
};
template <int N>
constexpr FxTab<N> fx_table(const double (&d)[N], double scale, double last) {
    FxTab<N> t{};
    for (int k = 0; k < N; ++k) {
        const double v = (d[k] + (k == N - 1 ? last : 0.0)) * scale * 4611686018427387904.0;
        t.c[k] = (fx_i64)(v + (v < 0 ? -0.5 : 0.5));
    }
    return t;
}
constexpr double kFx16F[] = MBS_F64_X16_F, kFx16G[] = MBS_F64_X16_G;
constexpr double kFx4F[] = MBS_F64_X4_F, kFx4G[] = MBS_F64_X4_G;
constexpr double FX_INV2PI = 0.15915494309189533577;
FX_CONST FxTab<MBS_F64_X16_DEG + 1> c_fx16F = fx_table(kFx16F, 1.0, -1.0);
FX_CONST FxTab<MBS_F64_X16_DEG + 1> c_fx16G = fx_table(kFx16G, FX_INV2PI, 0.0);
FX_CONST FxTab<MBS_F64_X4_DEG + 1> c_fx4F = fx_table(kFx4F, 1.0, -1.0);
FX_CONST FxTab<MBS_F64_X4_DEG + 1> c_fx4G = fx_table(kFx4G, FX_INV2PI, 0.0);

// kappa r >= 64: with s = 1 / x, v = s^2, f = 1 - v/16 + v^2 F(v) and
// g = -s/8 + s v G(v) (Hankel's expansion, leading terms exact, F and G fitted
// on v <= 2^-12; errors 3e-18 and 4e-17)
constexpr double kFx64F[] = MBS_FX_X64_F, kFx64G[] = MBS_FX_X64_G;  // signs alternate
constexpr unsigned FX_F0 = (unsigned)(kFx64F[0] * 0x1p34 + 0.5);
constexpr unsigned FX_F1 = (unsigned)(-kFx64F[1] * 0x1p23 + 0.5);
constexpr unsigned FX_F2 = (unsigned)(kFx64F[2] * 0x1p12 + 0.5);
constexpr unsigned FX_G0 = (unsigned)(kFx64G[0] * FX_INV2PI * 0x1p37 + 0.5);
constexpr unsigned FX_G1 = (unsigned)(-kFx64G[1] * FX_INV2PI * 0x1p26 + 0.5);
constexpr unsigned FX_G2 = (unsigned)(kFx64G[2] * FX_INV2PI * 0x1p15 + 0.5);

// e^{2 pi i theta} at 2^62, theta in turns at 2^64: the nearest of 1024 steps,
// times cos t + i sin t of the rest |t| <= pi / 1024
FX_HD void fx_cis(fx_u64 theta, const FxEntry* tab, fx_i64& dc, fx_i64& ds) {
    const fx_u64 th = theta + (1ull << 53);
    const FxEntry k = tab[(int)(th >> 54)];
    const fx_i64 z = (fx_i64)(th & ((1ull << 54) - 1)) - ((fx_i64)1 << 53);
    const fx_i64 tt = fx_mulhi(fx_split(z << 4), fx_split(7244019458077122842ll));  // 2 pi at 2^60: t at 2^64
    const fx2 ts = fx_split(tt);
    const fx_i64 t2 = fx_square(ts);  // t^2 at 2^64
    const unsigned t2s = (unsigned)(t2 >> 18);                                       // at 2^46
    const unsigned t4 = fx_mulhu(t2s, t2s);                                          // at 2^60
    const fx_i64 c1 = (fx_i64)fx_mulhu(t4, 2863311531u) - (t2 >> 1);                 // cos t - 1 at 2^64 (2^36 / 24)
    const unsigned p = fx_mulhu(t2s, 2863311531u - fx_mulhu(t2s, 8738u));            // t^2/6 - t^4/120 at 2^48 (2^34 / 6, 2^20 / 120)
    const fx_i64 sn = tt - ((fx_i64)fx_hi(fx_mulw((int)(tt >> 25), (int)p)) << 9);   // sin t at 2^64
    const fx2 C = fx_split(c1), S = fx_split(sn);
    // (k.c + i k.s)(1 + c1 + i sn) at 2^62
    const int nsh = -k.sh, nsl = -k.sl;
    const fx_i64 mc = fx_madw(k.ch, C.l, fx_madw(k.cl, C.h, fx_madw(nsh, S.l, fx_mulw(nsl, S.h))));
    const fx_i64 mi = fx_madw(k.sh, C.l, fx_madw(k.sl, C.h, fx_madw(k.ch, S.l, fx_mulw(k.cl, S.h))));
    dc = fx_madw(k.ch, C.h, fx_madw(nsh, S.h, ((fx_i64)k.ch << 32) + k.cl + (fx_i64)fx_hi(mc)));
    ds = fx_madw(k.sh, C.h, fx_madw(k.ch, S.h, ((fx_i64)k.sh << 32) + k.sl + (fx_i64)fx_hi(mi)));
}

// phi for one source at stored offset dj: the integers re, im, with
// phi = scale (re + i im) and |re|, |im| <= 2^59.  2D: false below kappa r = 4
// (the caller evaluates those pairs in FP64).  tab: cos and sin of k / 1024 turns.
template <int DIM>
FX_HD bool fx_phi(const FxBody<DIM>& b, const fx_i64* dj, const FxEntry* tab, fx_i64& re, fx_i64& im) {
    // r^2 at 2^62
    fx_i64 H = 0, M = 0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const fx_i64 dx = b.X[a] - (dj[a] >> b.sh);
        const int h = fx_hi(dx), l = (int)((unsigned)dx ^ 0x80000000u);
        H = fx_madw(h, h, H);
        M = fx_madw(h, l, M);
    }
    const fx_i64 A = fx_madw(fx_hi(M), 2, H);
    // r: an FP32 root r0 (24 bits, exact at 2^31) and two corrections from the
    // exact residuals of r0 and r0 + c
    const float af = (float)fx_hi(A) * 0x1p-30f;
    const float y = fx_rsqrt(af);
    const float r0f = af * y;
    const int r0 = fx_rint(r0f * 0x1p31f);
    const fx_i64 eps = fx_madw(-r0, r0, A);
    const float cf = (float)(int)(eps >> 20) * (y * 256.0f);
    const int c = fx_rint(cf);                               // at 2^51
    const fx_i64 t = fx_madw(-2 * c, r0, eps << 20);         // at 2^82, c^2 still to be taken off
    const int c2 = fx_rint(fmaf(cf, cf * -0x1p-34f, (float)(int)(t >> 14)) * (y * 0x1p-7f));  // at 2^62
    const fx_i64 cc = fx_madw(c, 2048, c2);
    const fx_i64 r = ((fx_i64)r0 << 31) + cc;
    // 1 / sqrt(r) = q0 (1 - w)^{-1/2}, w = 1 - q0^2 r: the residual of q0^2 r0
    // exactly modulo 2^64 (at 2^83), less q0^2 (r - r0); w at 2^75.  r - r0 counts to
    // its last bit: rounded at 2^-51, near pairs ended at 1.2e-15 instead of 2.4e-16
    // (1 % less time)
    const int q0 = fx_rint(fx_rsqrt(r0f) * 0x1p28f);
    const fx_u64 Q = fx_mulwu(q0, q0);  // 1 / r to 2^-22, at 2^56
    const unsigned rs = (unsigned)r0 >> 4;
    const fx_i64 w0 = -(fx_i64)(fx_mulwu((unsigned)Q, rs) + ((fx_u64)(fx_hiu(Q) * rs) << 32));
    const fx2 Qs = fx_split((fx_i64)Q);
    const int ch = (int)(cc >> 11), cl = (int)cc & 2047;
    const fx_i64 w = (w0 >> 8) - fx_madw(Qs.h, ch, fx_hi(fx_mulw(Qs.l, ch))) - (fx_mulw(Qs.h, cl) >> 11);
    const int w32 = (int)(w >> 25);               // at 2^50
    const int w2 = fx_hi(fx_mulw(w32, w32));      // w^2 at 2^68
    fx_i64 amp;                                   // 2D at 2^(58 + up), 3D at 2^(56 + up)
    fx_u64 theta;                                 // turns at 2^64
    {
        const fx_i64 p = fx_mulhi(fx_split(r), b.K);
        theta = (fx_u64)p << b.ksh;
    }
    if (DIM == 3) {
        const fx2 ws = fx_split(w);
        const fx_i64 qw = fx_mulhi(Qs, ws) + (fx_mulw(Qs.h, w2) >> 25);  // Q (w + w^2) at 2^67
        amp = ((fx_i64)Q + (qw >> 11)) << b.up;
    } else {
        const fx_i64 rinv =
            (fx_i64)Q + (fx_madw(Qs.h, w32, fx_hi(fx_mulw(Qs.l, w32)) + (fx_mulw(Qs.h, w2) >> 18)) >> 18);
        const fx_i64 s = fx_mulhi(fx_split(rinv), b.Ki);  // 1 / (kappa r) at 2^58
        fx_i64 f1, g;                                     // f - 1 at 2^62, g / 2 pi at 2^64
        if (s <= (fx_i64)1 << 52) {                       // kappa r >= 64
            const fx2 ss = fx_split(s);
            const fx_i64 v = fx_square(ss);  // at 2^52
            const unsigned s32 = (unsigned)(s >> 21), v32 = (unsigned)(v >> 9);
            const unsigned F = FX_F0 - fx_mulhu(v32, FX_F1 - fx_mulhu(v32, FX_F2));
            const unsigned G = FX_G0 - fx_mulhu(v32, FX_G1 - fx_mulhu(v32, FX_G2));
            f1 = ((fx_i64)fx_mulhu(fx_mulhu(v32, v32), F) << 6) - (v << 6);
            g = ((fx_i64)fx_mulhu(fx_mulhu(s32, v32), G) << 11) -
                (fx_mulhi(ss, fx_split(5871781006564002453ll)) << 2);  // 1 / (16 pi) at 2^68
        } else if (s <= (fx_i64)1 << 54) {  // kappa r >= 16: u = 32 s - 1
            const fx2 u = fx_split((s << 9) - ((fx_i64)1 << 62));
            fx_horner2(c_fx16F.c, c_fx16G.c, MBS_F64_X16_DEG, u, f1, g);
            g <<= 2;
        } else if (s <= (fx_i64)1 << 56) {  // kappa r >= 4: u = 8 s - 1
            const fx2 u = fx_split((s << 7) - ((fx_i64)1 << 62));
            fx_horner2(c_fx4F.c, c_fx4G.c, MBS_F64_X4_DEG, u, f1, g);
            g <<= 2;
        } else {
            re = im = 0;
            return false;
        }
        theta += (fx_u64)g + (1ull << 61);  // + pi / 4
        // f (1 - w)^{-1/2} at 2^62
        const fx_i64 m = ((fx_i64)1 << 62) + (w >> 14) + ((3 * w2) >> 9) + f1 +
                         (fx_mulw(w32, (int)(f1 >> 24)) >> 27);
        const fx2 ms = fx_split(m);
        amp = fx_madw(q0 << b.up, ms.h, fx_hi(fx_mulw(q0 << b.up, ms.l)));
    }
    fx_i64 dc, ds;
    fx_cis(theta, tab, dc, ds);
    const fx2 as = fx_split(amp);
    re = fx_mulhi(as, fx_split(dc));
    im = fx_mulhi(as, fx_split(ds));
    return true;
}
