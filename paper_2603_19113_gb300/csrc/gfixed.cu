// FP64-accurate all-pairs sums in 64-bit fixed point on the integer
// multipliers (Sec. 1 eq. Gmtx-entries; Sec. 2.2; Sec. 4.1 eq. out_skel):
// y_i = sum over the skeleton sources j of other bodies of phi(t_i - x_j) q_j,
// for FP64 operators, refinement residuals and field evaluation.
//
// phi comes from phi_fx.h (73 wide integer multiply-adds a pair in 2D, against
// about 50 FP64 operations that take 16 times as long each); the product with
// the right-hand sides, integers of 60 bits relative to the largest |q| of a
// source body, takes 4 wide multiply-adds and 8 FP32 ones a pair and right-hand
// side, and goes into FP64 sums once per 64 sources.  The FP32 ones are the cross
// terms of high words (27 bits of phi, 28 of q) and low ones, 2^-28 of a product
// of the largest entries: their 24 bits end near 2^-52 of it, up to 8 times
// coarser in a sum of 16.  237 bodies of 64
// points, 5 right-hand sides: 4.40 ms, 42 ms on the FP64 pipe; 1000 bodies and
// 4096 targets, 8 right-hand sides: 5.7 ms and 53.6 ms.  The wide multiply-adds
// alone, 32 a clock and SM, would take 2.1 ms of the 4.40; issue slots are 57 %
// busy, the ALU 52 %, and warps wait for dispatch, busy pipes and dependent
// results in about equal parts.
//
// g_fx_pack_kernel, one CTA per body, turns the offsets from the body's centre
// and the right-hand sides into integers scaled by the body's own radius and
// largest entry.  A body with a non-finite entry, or entries outside
// 1e-270..1e270, is marked and its sums are formed in FP64 from the caller's
// values; so are bodies outside the formats of phi_fx.h (targets close to the
// hull of a body, extreme kappa or sizes) and 2D pairs below kappa r = 4.
#include <type_traits>

#include "bessel.cuh"
#include "common.cuh"
#include "fx_tables.h"
#include "phi_fx.h"

namespace {

__device__ const FxSteps g_fx_steps = fx_steps();

constexpr int FXT = 128;     // threads per CTA
constexpr int FX_SB = 32;    // sources staged per round
constexpr int FX_FLUSH = 64; // sources per integer sum
constexpr int FX_QBITS = 60;  // right-hand sides are integers below 2^60: 64 products stay below 2^62 in an integer sum
constexpr int FX_CROSS = 4;   // sources per FP32 sum of cross terms (below 2^63: its integer part fits 32 bits)
constexpr int FX_BAD = INT_MIN;  // stored exponent of a body whose values need FP64

__device__ __forceinline__ double fx_block_max(double v, double* s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    double m = s[0];
#pragma unroll
    for (int w = 1; w < FXT / 32; ++w) m = fmax(m, s[w]);
    return m;
}

template <int DIM>
__global__ void __launch_bounds__(FXT) g_fx_pack_kernel(const int64_t N, const int T, const int64_t* __restrict__ off,
                                                        const double* __restrict__ xw,
                                                        const double* __restrict__ centres, const int nrhs,
                                                        const double2* __restrict__ q, FxPacked P) {
    __shared__ double s_red[FXT / 32];
    const int b = blockIdx.x;
    const int64_t j0 = off[b], j1 = off[b + 1];
    double c[DIM], r2 = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) c[a] = centres[3 * b + a];
    for (int64_t j = j0 + threadIdx.x; j < j1; j += FXT) {
        double s = 0.0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            const double d = xw[a * N + j] - c[a];
            s = fma(d, d, s);
        }
        r2 = fmax(r2, s);
    }
    const double rho = sqrt(fx_block_max(r2, s_red)) * (1.0 + 1e-6);
    const int es = fx_exponent(fmin(fmax(rho, 1e-80), 1e80));
    const double up = fx_exp2(63 - es);
    bool bad = !(rho < 1e80);
    for (int64_t j = j0 + threadIdx.x; j < j1; j += FXT)
#pragma unroll
        for (int a = 0; a < DIM; ++a) P.d[a * N + j] = bad ? 0 : fx_round((xw[a * N + j] - c[a]) * up);
    // one warp per right-hand side: no barriers between them (one body of 64
    // points, 8 right-hand sides, as one loop of the CTA: 26 us more)
    const int lane = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < nrhs; r += FXT / 32) {
        double m = 0.0;
        bool odd = false;
        for (int64_t j = j0 + lane; j < j1; j += 32) {
            const double2 v = q[(int64_t)r * N + j];
            m = fmax(m, fmax(fabs(v.x), fabs(v.y)));
            odd = odd || !isfinite(v.x) || !isfinite(v.y);
        }
        if (odd) m = HUGE_VAL;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        const bool out = !(m < 1e270) || (m > 0.0 && m < 1e-270);
        bad = bad || out;
        const int ex = fx_exponent(out || m == 0.0 ? 1.0 : m);
        const double sc = fx_exp2(FX_QBITS - ex);
        for (int64_t j = j0 + lane; j < j1; j += 32) {
            const double2 v = q[(int64_t)r * N + j];
            const fx2 re = fx_split(out ? 0 : fx_round(v.x * sc)), im = fx_split(out ? 0 : fx_round(v.y * sc));
            P.qh[(int64_t)r * N + j] = make_int2(re.h, im.h);
            P.ql[(int64_t)r * N + j] = make_float4((float)re.h, (float)re.l, (float)im.h, (float)im.l);
        }
        if (lane == 0) P.qs[(int64_t)r * T + b] = fx_exp2(ex + 64 - FX_QBITS);  // of sums kept at 2^-64
    }
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        P.rho[b] = (float)rho * 1.000001f;
        P.es[b] = bad ? FX_BAD : es;
    }
}

// phi in FP64 where the fixed-point evaluation does not apply
template <int DIM>
__device__ __noinline__ double2 fx_phi_f64(double kappa, double r2) {
    return phi_f64_r2<DIM>(kappa, r2);
}

// One thread per target; SG groups of FXT / SG threads take SG-th parts of the
// staged sources of the same targets (small problems, where the sources of a
// body would otherwise be one long chain per thread).  4 CTAs per SM with two
// sources in flight a thread: 5 with one source 3 % slower (4.50 ms, 237 bodies, 5
// right-hand sides), 5 with two 2 %, 6 with one 4 % (8 right-hand sides: 12 %).
template <int DIM, int NR, int SG>
__global__ void __launch_bounds__(FXT, 4)
    g_fx_kernel(const FxKappa kap, const int64_t Nt, const double* __restrict__ tgt, const int* __restrict__ tbody,
                const int64_t N, const int T, const double* __restrict__ xw, const int64_t* __restrict__ off,
                const double* __restrict__ centres, const FxPacked P, const int nrhs, const int r0,
                const double2* __restrict__ q, double2* __restrict__ part, const int* __restrict__ split_body) {
    constexpr int TG = FXT / SG;
    __shared__ FxEntry s_tab[FX_TAB];
    __shared__ fx_i64 s_d[FX_SB][DIM];
    __shared__ int2 s_qh[FX_SB][NR];    // high words of re q, im q
    __shared__ float4 s_ql[FX_SB][NR];  // re high, re low, im high, im low as floats
    __shared__ double2 s_acc[NR][FXT];
    const int tid = threadIdx.x, grp = tid / TG;
    for (int k = tid; k < FX_TAB; k += FXT) s_tab[k] = g_fx_steps.e[k];
    const int64_t i = (int64_t)blockIdx.x * TG + tid % TG;
    const bool valid = i < Nt;
    const int tb = (valid && tbody) ? tbody[i] : -1;
    double x[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) x[a] = valid ? tgt[a * Nt + i] : 0.0;
#pragma unroll
    for (int r = 0; r < NR; ++r) s_acc[r][tid] = make_double2(0.0, 0.0);
    const int sb0 = split_body[blockIdx.y], sb1 = split_body[blockIdx.y + 1];
    for (int sb = sb0; sb < sb1; ++sb) {
        const int64_t js = off[sb], je = off[sb + 1];
        const bool act = valid && tb != sb;  // zero diagonal blocks of G_hat
        const int es = P.es[sb];
        FxBody<DIM> B;
        double D[DIM], Dl[DIM], scale = 0.0;
        float R2 = 0.f;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            D[a] = fx_diff(x[a], centres[3 * sb + a], Dl[a]);
            R2 = fmaf((float)D[a], (float)D[a], R2);
        }
        const bool fast = act && es != FX_BAD && fx_body<DIM>(kap, D, Dl, sqrtf(R2), P.rho[sb], es, B, scale);
        fx_i64 ar[NR], ai[NR];
        float mr[NR], mi[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            ar[r] = ai[r] = 0;
            mr[r] = mi[r] = 0.f;
        }
        // the cross terms into the integer sums, every few sources: their FP32
        // sum rounds at 2^-24 of its own size
        auto carry = [&]() {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                ar[r] += __float2int_rn(mr[r] * 0x1p-32f);
                ai[r] += __float2int_rn(mi[r] * 0x1p-32f);
                mr[r] = mi[r] = 0.f;
            }
        };
        auto flush = [&]() {
#pragma unroll
            for (int r = 0; r < NR; ++r)
                if (r0 + r < nrhs) {
                    const double f = scale * P.qs[(int64_t)(r0 + r) * T + sb];
                    double2 a = s_acc[r][tid];
                    a.x = fma((double)ar[r], f, a.x);
                    a.y = fma((double)ai[r], f, a.y);
                    s_acc[r][tid] = a;
                    ar[r] = ai[r] = 0;
                }
        };
        int since = 0;
        for (int64_t jc = js; jc < je; jc += FX_SB) {
            const int n = (int)min((int64_t)FX_SB, je - jc);
            __syncthreads();
            for (int k = tid; k < n * DIM; k += FXT) s_d[k % n][k / n] = P.d[(int64_t)(k / n) * N + jc + k % n];
            for (int k = tid; k < n * NR; k += FXT) {
                const int r = k / n, j = k - r * n;
                const bool in = r0 + r < nrhs;
                s_qh[j][r] = in ? P.qh[(int64_t)(r0 + r) * N + jc + j] : make_int2(0, 0);
                s_ql[j][r] = in ? P.ql[(int64_t)(r0 + r) * N + jc + j] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            __syncthreads();
            const int part_n = (n + SG - 1) / SG;
            const int k0 = grp * part_n, k1 = min(n, k0 + part_n);
            if (fast) {
#pragma unroll 2
                for (int j = k0; j < k1; ++j) {
                    fx_i64 pr, pi;
                    if (!fx_phi<DIM>(B, s_d[j], s_tab, pr, pi)) {  // 2D, kappa r < 4
                        double r2 = 0.0;
#pragma unroll
                        for (int a = 0; a < DIM; ++a) {
                            const double e = x[a] - xw[a * N + jc + j];
                            r2 = fma(e, e, r2);
                        }
                        const double2 p = fx_phi_f64<DIM>(kap.kappa, r2);
                        pr = fx_round(p.x / scale);
                        pi = fx_round(p.y / scale);
                    }
                    // high x high words exactly on the integer multipliers; the
                    // cross terms, 2^-32 of them, in FP32 beside them
                    const fx2 a = fx_split(pr), b = fx_split(pi);
                    const int nh = -b.h;
                    const float ah = (float)a.h, al = (float)a.l, bh = (float)b.h, bl = (float)b.l;
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const int2 v = s_qh[j][r];
                        const float4 w = s_ql[j][r];
                        ar[r] = fx_madw(a.h, v.x, fx_madw(nh, v.y, ar[r]));
                        ai[r] = fx_madw(a.h, v.y, fx_madw(b.h, v.x, ai[r]));
                        mr[r] = fmaf(ah, w.y, fmaf(al, w.x, fmaf(-bh, w.w, fmaf(-bl, w.z, mr[r]))));
                        mi[r] = fmaf(ah, w.w, fmaf(al, w.z, fmaf(bh, w.y, fmaf(bl, w.x, mi[r]))));
                    }
                    if ((j - k0) % FX_CROSS == FX_CROSS - 1) carry();
                }
                carry();
                since += FX_SB;
                if (since == FX_FLUSH || jc + FX_SB >= je) {
                    flush();
                    since = 0;
                }
            } else if (act) {
#pragma unroll 1
                for (int j = k0; j < k1; ++j) {
                    double r2 = 0.0;
#pragma unroll
                    for (int a = 0; a < DIM; ++a) {
                        const double e = x[a] - xw[a * N + jc + j];
                        r2 = fma(e, e, r2);
                    }
                    const double2 p = fx_phi_f64<DIM>(kap.kappa, r2);
#pragma unroll 1
                    for (int r = 0; r < NR; ++r)
                        if (r0 + r < nrhs) s_acc[r][tid] = cfma(p, q[(int64_t)(r0 + r) * N + jc + j], s_acc[r][tid]);
                }
            }
        }
    }
    if (SG > 1) __syncthreads();
    if (!valid || grp > 0) return;
    double2* out = part + (int64_t)blockIdx.y * nrhs * Nt;
#pragma unroll
    for (int r = 0; r < NR; ++r)
        if (r0 + r < nrhs) {
            double2 a = s_acc[r][tid];
#pragma unroll
            for (int g = 1; g < SG; ++g) a = cadd(a, s_acc[r][g * TG + tid]);
            out[(int64_t)(r0 + r) * Nt + i] = a;
        }
}

template <int DIM, int SG>
void launch_fx(const GLayout& L, const double* centres, const FxKappa& k, int64_t Nt, const double* tgt, const int* tbody,
               int nrhs, const double2* q, const FxPacked& P, double2* part, int nsplit, const int* sb, cudaStream_t st) {
    const dim3 grid((unsigned)((Nt + FXT / SG - 1) / (FXT / SG)), (unsigned)nsplit);
    auto pass = [&](auto width, int r0) {
        g_fx_kernel<DIM, decltype(width)::value, SG>
            <<<grid, FXT, 0, st>>>(k, Nt, tgt, tbody, L.N, L.T, L.xw64, L.off, centres, P, nrhs, r0, q, part, sb);
        MBS_CHECK_LAUNCH();
        return r0 + decltype(width)::value;
    };
    // a right-hand side of padding costs about 4 % of a pair
    for (int r0 = 0; r0 < nrhs;) {
        const int left = nrhs - r0;
        r0 = left > 6    ? pass(std::integral_constant<int, 8>{}, r0)
             : left > 4  ? pass(std::integral_constant<int, 6>{}, r0)
             : left == 4 ? pass(std::integral_constant<int, 4>{}, r0)
             : left == 3 ? pass(std::integral_constant<int, 3>{}, r0)
             : left == 2 ? pass(std::integral_constant<int, 2>{}, r0)
                         : pass(std::integral_constant<int, 1>{}, r0);
    }
}

}  // namespace

size_t fx_pack_bytes(int dim, int64_t N, int T, int nrhs) {
    return (size_t)N * nrhs * (sizeof(int2) + sizeof(float4)) + (size_t)nrhs * T * sizeof(double) +
           (size_t)dim * N * sizeof(fx_i64) + (size_t)T * (sizeof(float) + sizeof(int));
}

FxPacked fx_packed(void* p, int dim, int64_t N, int T, int nrhs) {
    unsigned char* c = static_cast<unsigned char*>(p);
    FxPacked P;
    P.ql = reinterpret_cast<float4*>(c);
    c += (size_t)N * nrhs * sizeof(float4);
    P.qh = reinterpret_cast<int2*>(c);
    c += (size_t)N * nrhs * sizeof(int2);
    P.qs = reinterpret_cast<double*>(c);
    c += (size_t)nrhs * T * sizeof(double);
    P.d = reinterpret_cast<fx_i64*>(c);
    c += (size_t)dim * N * sizeof(fx_i64);
    P.rho = reinterpret_cast<float*>(c);
    c += (size_t)T * sizeof(float);
    P.es = reinterpret_cast<int*>(c);
    return P;
}

void launch_G_fx(const GLayout& L, const double* d_centres, double kappa, int64_t Nt, const double* tgt,
                 const int* tbody, int nrhs, const double2* q, double2* y, double2* part, int nsplit,
                 const int* d_split_body, void* pack, cudaStream_t st, cudaEvent_t ev0, cudaEvent_t ev1) {
    if (Nt == 0 || L.N == 0 || nrhs == 0) return;
    const FxKappa k = fx_kappa(L.dim, kappa);
    const FxPacked P = fx_packed(pack, L.dim, L.N, L.T, nrhs);
    if (ev0) record_event(ev0, st);
    if (L.dim == 2)
        g_fx_pack_kernel<2><<<L.T, FXT, 0, st>>>(L.N, L.T, L.off, L.xw64, d_centres, nrhs, q, P);
    else
        g_fx_pack_kernel<3><<<L.T, FXT, 0, st>>>(L.N, L.T, L.off, L.xw64, d_centres, nrhs, q, P);
    MBS_CHECK_LAUNCH();
    const bool wide = fx_groups(Nt, L.T) > 1;
    if (L.dim == 2 && wide)
        launch_fx<2, 4>(L, d_centres, k, Nt, tgt, tbody, nrhs, q, P, part, nsplit, d_split_body, st);
    else if (L.dim == 2)
        launch_fx<2, 1>(L, d_centres, k, Nt, tgt, tbody, nrhs, q, P, part, nsplit, d_split_body, st);
    else if (wide)
        launch_fx<3, 4>(L, d_centres, k, Nt, tgt, tbody, nrhs, q, P, part, nsplit, d_split_body, st);
    else
        launch_fx<3, 1>(L, d_centres, k, Nt, tgt, tbody, nrhs, q, P, part, nsplit, d_split_body, st);
    if (ev1) record_event(ev1, st);
    launch_reduce_splits64(part, nsplit, Nt * nrhs, y, st);
}

// Four groups of threads share the sources of a target when 128-target tiles
// and one split per body would leave SMs without a CTA or two (4 right-hand
// sides, bodies of 64: 95 us instead of 142 for 10 bodies, 226 for 259 for 40,
// 622 for 620 for 80, 2114 for 2019 for 160).
int fx_groups(int64_t Nt, int T) {
    const int64_t tiles = (Nt + FXT - 1) / FXT;
    return tiles * std::min(T, 64) < 8LL * mbs_num_sms() ? 4 : 1;
}

int fx_outside(int dim, double kappa, const double* x, int own, int T, const double* centres, const double* rho) {
    const FxKappa k = fx_kappa(dim, kappa);
    int n = 0;
    for (int t = 0; t < T; ++t) {
        if (t == own) continue;
        double D[3] = {0.0, 0.0, 0.0}, Dl[3] = {0.0, 0.0, 0.0}, R2 = 0.0, scale = 0.0;
        for (int a = 0; a < dim; ++a) {
            D[a] = x[a] - centres[3 * t + a];
            R2 += D[a] * D[a];
        }
        FxBody<2> b2;
        FxBody<3> b3;
        const int es = fx_exponent(rho[t]);
        n += dim == 2 ? !fx_body<2>(k, D, Dl, sqrt(R2), rho[t], es, b2, scale)
                      : !fx_body<3>(k, D, Dl, sqrt(R2), rho[t], es, b3, scale);
    }
    return n;
}

int fx_tile(int64_t Nt, int T) { return FXT / fx_groups(Nt, T); }
