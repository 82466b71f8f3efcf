// Host entry points of csrc/phi_fx.h for tests/test_phi_fx.py.
#include "../paper_2603_19113_gb300/csrc/fx_tables.h"
#include "../paper_2603_19113_gb300/csrc/phi_fx.h"

static const FxSteps steps = fx_steps();

// phi of n (target offset D, source offset dj at 2^(63 - es)) pairs; ok[i] = 0:
// outside the formats, 2: below kappa r = 4; raw: the integers, scaled: phi
template <int DIM>
static void run(double kappa, int n, const double* D, const double* rho, const int* es, const long long* dj,
                double* out, int* ok, long long* raw) {
    const FxKappa k = fx_kappa(DIM, kappa);
    const double zero[3] = {0.0, 0.0, 0.0};
    for (int i = 0; i < n; ++i) {
        double R = 0.0, scale = 0.0;
        for (int a = 0; a < DIM; ++a) R += D[i * DIM + a] * D[i * DIM + a];
        FxBody<DIM> b;
        fx_i64 re = 0, im = 0;
        ok[i] = fx_body<DIM>(k, D + DIM * i, zero, sqrt(R), rho[i], es[i], b, scale) ? 1 : 0;
        if (ok[i] && !fx_phi<DIM>(b, dj + DIM * i, steps.e, re, im)) ok[i] = 2;
        raw[2 * i] = re;
        raw[2 * i + 1] = im;
        out[2 * i] = scale * (double)re;
        out[2 * i + 1] = scale * (double)im;
    }
}

extern "C" void phi_fx_batch(int dim, double kappa, int n, const double* D, const double* rho, const int* es,
                             const long long* dj, double* out, int* ok, long long* raw) {
    if (dim == 2)
        run<2>(kappa, n, D, rho, es, dj, out, ok, raw);
    else
        run<3>(kappa, n, D, rho, es, dj, out, ok, raw);
}

extern "C" void cis_fx_batch(int n, const unsigned long long* theta, long long* c, long long* s) {
    for (int i = 0; i < n; ++i) {
        fx_i64 x, y;
        fx_cis(theta[i], steps.e, x, y);
        c[i] = x;
        s[i] = y;
    }
}
