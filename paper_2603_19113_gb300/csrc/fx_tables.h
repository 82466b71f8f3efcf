// Host tables of the fixed-point kernels (phi_fx.h): the steps of cos and sin
// and the constants of a wavenumber, from 128-bit integer arithmetic.
#pragma once

#include "phi_fx.h"

// a b / 2^64, rounded down, from 32-bit products (constant expressions of host
// and device compilers alike)
constexpr fx_u64 fx_umul64(fx_u64 a, fx_u64 b) {
    const fx_u64 al = a & 0xffffffffu, ah = a >> 32, bl = b & 0xffffffffu, bh = b >> 32;
    const fx_u64 m1 = ah * bl + ((al * bl) >> 32);
    const fx_u64 m2 = al * bh + (m1 & 0xffffffffu);
    return ah * bh + (m1 >> 32) + (m2 >> 32);
}

struct FxSteps {
    FxEntry e[FX_TAB];
};

// cos and sin of k / 1024 turns at 2^62: Taylor series on the first eighth of a
// turn, then the symmetries
constexpr FxSteps fx_steps() {
    FxSteps t{};
    fx_i64 cs[FX_TAB / 8 + 1] = {}, sn[FX_TAB / 8 + 1] = {};
    for (int j = 0; j <= FX_TAB / 8; ++j) {
        // angle 2 pi j / 1024 at 2^64 (below 0.79): 2 pi at 2^61 times j 2^-7
        const fx_u64 a = fx_umul64(14488038916154245685ull, (fx_u64)j << 56) << 1;
        const fx_u64 a2 = fx_umul64(a, a);
        // cos a = 1 - a2/2 (1 - a2/12 (1 - ...)), sin a = a (1 - a2/6 (1 - ...)), at 2^63
        fx_u64 c = 1ull << 63, s = 1ull << 63;
        for (int n = 22; n >= 2; n -= 2) {
            c = (1ull << 63) - fx_umul64(c, a2) / (fx_u64)(n * (n - 1));
            s = (1ull << 63) - fx_umul64(s, a2) / (fx_u64)(n * (n + 1));
        }
        cs[j] = (fx_i64)((c + 1) >> 1);
        sn[j] = (fx_i64)((fx_umul64(s, a) + 1) >> 1);
    }
    for (int k = 0; k < FX_TAB; ++k) {
        const int oct = k / (FX_TAB / 8), rest = k % (FX_TAB / 8);
        const int j = (oct & 1) ? FX_TAB / 8 - rest : rest;  // eighth turns alternate in direction
        const bool swap = (oct & 3) == 1 || (oct & 3) == 2;
        const fx_i64 u = swap ? sn[j] : cs[j], w = swap ? cs[j] : sn[j];
        const fx_i64 x = (oct >= 2 && oct <= 5) ? -u : u, y = oct >= 4 ? -w : w;
        t.e[k].ch = (int)((x + 0x80000000ll) >> 32);
        t.e[k].cl = (int)(unsigned)((fx_u64)x & 0xffffffffu);
        t.e[k].sh = (int)((y + 0x80000000ll) >> 32);
        t.e[k].sl = (int)(unsigned)((fx_u64)y & 0xffffffffu);
    }
    return t;
}

// Mantissas at 2^62 in [2^61, 2^62) of kappa / (2 pi) and 1 / kappa
inline FxKappa fx_kappa(int dim, double kappa) {
    FxKappa k{};
    k.kappa = kappa;
    int e;
    const fx_u64 m = (fx_u64)ldexp(frexp(kappa, &e), 53);  // kappa = m 2^(e - 53), m in [2^52, 2^53)
    const fx_u64 inv2pi66 = 11743562013128004906ull;       // 1 / (2 pi) at 2^66 (0.159 2^66 in [2^63, 2^64))
    const unsigned __int128 p = (unsigned __int128)m * inv2pi66;               // kappa / 2 pi = p 2^(e - 119), p in [2^115, 2^117)
    const int up = (p >> 116) ? 1 : 0;
    k.kturn62 = (fx_i64)(((p >> (53 + up)) + 1) >> 1);
    k.kturn_e = e - 119 + 54 + up + 62;
    const unsigned __int128 q = ((unsigned __int128)1 << 115) / m;             // 1 / kappa = q 2^(-62 - e), q in (2^62, 2^63]
    k.kinv62 = (fx_i64)((q + 1) >> 1);
    k.kinv_e = 1 - e;
    k.amp = dim == 2 ? 0.25 * sqrt(2.0 / (3.14159265358979323846 * kappa)) : 0.07957747154594766788;
    return k;
}
