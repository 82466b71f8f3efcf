// Batched FP64 construction of the local scattering matrices (Sec. 4.2-4.5).
//
// One CTA per distinct shape does the whole local computation in FP64 on
// matrices kept in global memory (L2-resident for the sizes used here):
//
//  phase 1   B(i,j) = phi(z_i - x_j)  (p x m, eq. B-matrix)
//            D(i,j) = phi(z_i - y_j)  (p x n)         A(i,j) = phi(x_i - y_j)  (m x n)
//            Householder QR of B with column pivoting (largest remaining
//            column norm, recomputed in full after every step; ties within a
//            relative 1e-10 go to the lowest original column index), with the
//            same reflectors applied to D.  The skeleton count k is fixed or
//            the first step at which the largest remaining column norm is at
//            most eps times the largest initial one; the factorisation goes on
//            to the numerical rank r_B (largest remaining column norm above
//            10 ls_rcond, see B_QR_CUT) for the least-squares solve below.
//            Randomized ID (option id_sketch): the skeleton and Z* come instead
//            from the pivoted QR of the sketch Y = Omega B (k + oversampling
//            rows, Omega a complex Gaussian test matrix from Philox4x32-10
//            keyed by the seed and the shape index, Box-Muller); B's own
//            pivoted QR then serves the least-squares solve for C only.
//  phase 2   Z* = [I_k | R11^{-1} R12] in pivot order (ID, eq. B_fac);
//            C = minimum-norm least-squares solution of B C = D on the rank r_B
//            of that factorisation (Sec. 4.4): a complete orthogonal
//            decomposition R_B Z^H = [T 0] by reflectors from the right (RZ
//            reduction of the trapezoidal R_B), then
//            C P_B = Z^H [T^{-1} (Q_B^H D)(1:r_B, :); 0];
//            U = (Z*)^T (Sec. 4.2) and the pivoted QR of A with its reflectors
//            applied to U, run to the rounding level (0.01 ls_rcond).
//  phase 3   truncated SVD of A (Sec. 3.1, "truncated SVD"): one-sided Jacobi
//            (Hestenes) on X = R_A^H, the columns of X J mutually orthogonal,
//            so R_A = J Sigma V^H with V = (X J) Sigma^{-1} and
//            A P_A = (Q_A J) Sigma V^H.  Singular values at most ls_rcond times
//            the largest are dropped, as in the oracle, so that
//            A^+ = P_A V_r Sigma_r^{-1} J_r^H Q_A^H, and
//            S = (Z* C P_A V_r Sigma_r^{-1}) (J_r^H (Q_A^H U)(1:r_A, :))
//            (eq. scattering-matrix).  The division by the small singular
//            values acts on the columns of Z* C P_A V_r before the product with
//            the projections of U, which keeps the rounding of the
//            ill-conditioned MFS solve out of S.  Pivoted QR ahead of the
//            Jacobi sweeps (Drmac & Veselic 2008) leaves X with strongly graded
//            columns, so few sweeps converge.
//
// The right-hand side b = Z* C A^+ v (Sec. 4.5) is formed right to left from
// the stored factors (rhs_kernel): Q_A^H v, J_r^H, the scaled right singular
// vectors, C, then Z*.
#include <algorithm>

#include "bessel.cuh"
#include "common.cuh"
#include "sbuild.cuh"

namespace {

constexpr int SBT_MAX = 512;      // largest CTA size (threads per shape CTA: 128, 256 or 512)
constexpr int NW_MAX = SBT_MAX / 32;
constexpr double TIE = 1e-10;
// The rank of B for the least-squares solve of C: the pivoted QR stops where
// its largest remaining column norm falls to B_QR_CUT * ls_rcond.  A pivoted
// QR's diagonal overestimates the singular values it tracks; cut at 10 x
// ls_rcond it keeps the rank of the truncated SVD at ls_rcond to within 0-2
// on the test shapes (2D smooth, corner-refined and 3D), where a cut at
// ls_rcond itself keeps 4-11 more, noise-level directions.
constexpr double B_QR_CUT = 10.0;

// warps of the CTA (the block size is chosen at launch)
__device__ __forceinline__ int nwarps() { return (int)(blockDim.x >> 5); }

// The CTAs that build one shape together: one, or a thread-block cluster when
// there are fewer shapes than SMs.  Columns and entries are dealt out over the
// team's warps and threads; what decides the course of a factorisation is
// computed by every CTA from the same values (or by CTA 0 alone), and every sum
// is formed by one warp or one CTA in the same order as with one CTA, so the
// results do not depend on the team's size.
struct Team {
    int rank, size;
    __device__ __forceinline__ int warp() const { return rank * nwarps() + (int)(threadIdx.x >> 5); }
    __device__ __forceinline__ int warps() const { return size * nwarps(); }
    __device__ __forceinline__ int64_t thread() const { return (int64_t)rank * blockDim.x + threadIdx.x; }
    __device__ __forceinline__ int64_t threads() const { return (int64_t)size * blockDim.x; }
    // all writes of the team to global memory before the call are visible after it
    __device__ __forceinline__ void sync() const {
        __syncthreads();
        if (size > 1) {
            __threadfence();
            asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        }
    }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double2 warp_sum2(double2 v) {
    return make_double2(warp_sum(v.x), warp_sum(v.y));
}

struct Red {
    double d[NW_MAX];
    double d2[NW_MAX];
    int i[NW_MAX];
    int j[NW_MAX];
};

// Block-wide sum of a double (every thread gets the result).
__device__ double block_sum(double v, Red& r) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) r.d[w] = v;
    __syncthreads();
    double t = 0.0;
    const int nw = nwarps();
    for (int k = 0; k < nw; ++k) t += r.d[k];
    return t;
}

__device__ double block_max(double v, Red& r) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) r.d[w] = v;
    __syncthreads();
    double t = r.d[0];
    const int nw = nwarps();
    for (int k = 1; k < nw; ++k) t = fmax(t, r.d[k]);
    return t;
}

// Block-wide argmin of key (ties: smaller idx); returns idx.
__device__ int block_argmin(int key, int idx, Red& r) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int k2 = __shfl_xor_sync(0xffffffffu, key, o);
        const int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
        if (k2 < key || (k2 == key && i2 < idx)) {
            key = k2;
            idx = i2;
        }
    }
    __syncthreads();
    if (lane == 0) {
        r.i[w] = key;
        r.j[w] = idx;
    }
    __syncthreads();
    int bk = r.i[0], bi = r.j[0];
    const int nw = nwarps();
    for (int k = 1; k < nw; ++k)
        if (r.i[k] < bk || (r.i[k] == bk && r.j[k] < bi)) {
            bk = r.i[k];
            bi = r.j[k];
        }
    return bi;
}

template <int DIM>
__device__ void fill_kernel_matrix(const Team& tm, double2* M, int ld, const double* T, int nt, const double* S,
                                   int ns, double kappa) {
    for (int64_t e = tm.thread(); e < (int64_t)nt * ns; e += tm.threads()) {
        const int i = (int)(e % nt), j = (int)(e / nt);
        double r2 = 0.0;
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
            const double d = T[c * nt + i] - S[c * ns + j];
            r2 = fma(d, d, r2);
        }
        M[(int64_t)j * ld + i] = phi_f64<DIM>(kappa, sqrt(r2));
    }
}

// Step j of a Householder QR of A (rows x ncols columns, leading dimension
// ld): the unit reflector v of column j (rows j..rows-1) replaces the column
// there (H = I - 2 v v^H), diag[j] = R_jj, and H is applied to columns
// j+1 .. ntot-1 (one warp per column).  With nrm2 given, the squared norms of
// rows j+1.. of columns j+1 .. ncols-1 are refreshed in full.  Every CTA of the
// team forms the reflector; CTA 0 stores it once all have read the column.
__device__ void householder_step(const Team& tm, double2* A, int ld, int rows, int j, int ncols, int ntot,
                                 double2* diag, double* nrm2, double2* s_v, Red& red) {
    const int lane = threadIdx.x & 31;
    double2* cj = A + (int64_t)j * ld;
    double sl = 0.0;
    for (int i = j + threadIdx.x; i < rows; i += blockDim.x) sl += cabs2(cj[i]);
    const double nx2 = block_sum(sl, red);
    const double2 x0 = cj[j];
    const double ax0 = sqrt(cabs2(x0));
    const double2 ph = ax0 > 0.0 ? make_double2(x0.x / ax0, x0.y / ax0) : make_double2(1.0, 0.0);
    const double nx = sqrt(nx2);
    const double2 alpha = make_double2(-ph.x * nx, -ph.y * nx);
    const double2 v0 = csub(x0, alpha);
    const double nv2 = nx2 - ax0 * ax0 + cabs2(v0);
    const double inv = nv2 > 0.0 ? 1.0 / sqrt(nv2) : 0.0;
    __syncthreads();
    for (int i = j + threadIdx.x; i < rows; i += blockDim.x) {
        s_v[i - j] = (i == j) ? cscale(v0, inv) : cscale(cj[i], inv);
    }
    if (tm.rank == 0 && threadIdx.x == 0) diag[j] = alpha;
    __syncthreads();
    for (int c = j + 1 + tm.warp(); c < ntot; c += tm.warps()) {
        double2* cc = A + (int64_t)c * ld;
        double2 d = make_double2(0.0, 0.0);
        for (int i = j + lane; i < rows; i += 32) d = cfmac(s_v[i - j], cc[i], d);
        d = warp_sum2(d);
        d = cscale(d, 2.0);
        double s = 0.0;
        for (int i = j + lane; i < rows; i += 32) {
            const double2 nv = cfms(s_v[i - j], d, cc[i]);
            cc[i] = nv;
            if (i > j) s = abs2_acc(nv, s);
        }
        if (nrm2 && c < ncols) {
            s = warp_sum(s);
            if (lane == 0) nrm2[c] = s;
        }
    }
    tm.sync();
    if (tm.rank == 0)
        for (int i = j + threadIdx.x; i < rows; i += blockDim.x) cj[i] = s_v[i - j];
}

// One-sided Jacobi (Hestenes 1958) on the r columns of X (rows x r, leading
// dimension ldx): plane rotations from the right until every pair of columns
// is orthogonal to tol relative to the product of their norms; X J = W with
// orthogonal columns, J (r x r, leading dimension ldj, starts as I)
// accumulating the rotations.  Pairs are taken in round-robin tournament
// order, so every round rotates r/2 disjoint pairs; the result does not depend
// on how they are dealt out.  Returns the sweeps run (maxsweep + 1 if the last
// one still rotated).
//
// The FP64 pipe bounds this (a warp instruction takes 16 clocks of the SM
// whatever its lanes do), and of the ~230 FP64 instructions that a pair of 64
// rows took when one warp did all of it, 150 were the angle's square roots,
// divisions and hypotenuses, the same in all lanes.  So a round has three parts:
// warps sum the three products of up to four pairs at a time (the 16 partial
// sums of a lane halve in number while they are added, 16 additions instead of
// 80, in the same tree); one thread per pair finds the angle; warps rotate.
// The phase for 3 shapes of 64 MFS sources: 28.1 ms to 6.3 ms with 8 CTAs a
// shape; for 300 shapes of 35 to 105, one CTA each: 202 ms to 106 ms.
constexpr int JP = 256;  // pairs in flight (larger rounds are taken in parts)

struct Rot {
    double cs, sn, px, py;
    int on, i, j;
};

struct JacobiShared {
    double sums[JP][4];  // |x_i|^2, |x_j|^2, re and im of x_i^H x_j
    Rot rot[JP];
};

__device__ __forceinline__ void jacobi_pair(int pi, int rho, int re, int& i, int& j) {
    if (pi == 0) {
        i = rho;
        j = re - 1;
    } else {
        i = (rho + pi) % (re - 1);
        j = (rho - pi + re - 1) % (re - 1);
    }
    if (i > j) {
        const int t = i;
        i = j;
        j = t;
    }
}

__device__ int cta_jacobi(const Team& tm, double2* X, int ldx, int rows, int r, double2* Jm, int ldj, double tol,
                          int maxsweep, int* flag, JacobiShared& sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = nwarps();
    const int re = r + (r & 1);  // with a dummy column when r is odd
    const int half = re / 2;
    // this CTA's pairs of a round: a contiguous part of them
    const int per = (half + tm.size - 1) / tm.size;
    const int p0 = min(half, tm.rank * per), p1 = min(half, p0 + per);
    for (int sweep = 0; sweep < maxsweep; ++sweep) {
        if (tm.rank == 0 && threadIdx.x == 0) flag[sweep & 1] = 0;
        tm.sync();
        for (int rho = 0; rho < re - 1; ++rho) {
            for (int q0 = p0; q0 < p1; q0 += JP) {
                const int np = min(JP, p1 - q0);
                for (int g = 4 * w; g < np; g += 4 * nw) {
                    const double2 *xi[4], *xj[4];
                    double v[16];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        int i = 0, j = 0;
                        const bool in = g + u < np;
                        if (in) jacobi_pair(q0 + g + u, rho, re, i, j);
                        xi[u] = in && j < r ? X + (int64_t)i * ldx : nullptr;
                        xj[u] = X + (int64_t)(j < r ? j : 0) * ldx;
                        v[4 * u] = v[4 * u + 1] = v[4 * u + 2] = v[4 * u + 3] = 0.0;
                    }
                    for (int l = lane; l < rows; l += 32)
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (xi[u]) {
                                const double2 a = xi[u][l], b = xj[u][l];
                                v[4 * u] = abs2_acc(a, v[4 * u]);
                                v[4 * u + 1] = abs2_acc(b, v[4 * u + 1]);
                                const double2 c = cfmac(a, b, make_double2(v[4 * u + 2], v[4 * u + 3]));
                                v[4 * u + 2] = c.x;
                                v[4 * u + 3] = c.y;
                            }
#pragma unroll
                    for (int n = 16, o = 16; n > 1; n >>= 1, o >>= 1) {
                        const bool up = (lane & o) != 0;
#pragma unroll
                        for (int k = 0; k < n / 2; ++k) {
                            const double keep = up ? v[k + n / 2] : v[k], send = up ? v[k] : v[k + n / 2];
                            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                        }
                    }
                    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
                    // lanes 2 k and 2 k + 1 hold value k % 4 of pair k / 4
                    if (!(lane & 1) && g + (lane >> 3) < np) sh.sums[g + (lane >> 3)][(lane >> 1) & 3] = v[0];
                }
                __syncthreads();
                for (int q = threadIdx.x; q < np; q += blockDim.x) {
                    Rot R;
                    R.on = 0;
                    jacobi_pair(q0 + q, rho, re, R.i, R.j);
                    if (R.j < r) {
                        const double a = sh.sums[q][0], b = sh.sums[q][1];
                        const double2 c = make_double2(sh.sums[q][2], sh.sums[q][3]);
                        const double ac = sqrt(cabs2(c));
                        if (!(!(ac > 0.0) || ac <= tol * sqrt(a) * sqrt(b))) {
                            // x_j' = e^{-i arg c} x_j makes the pair's inner product real and
                            // positive; then the real rotation with t = tan(theta) the
                            // smaller root of t^2 + 2 zeta t - 1 = 0
                            R.on = 1;
                            R.px = c.x / ac;
                            R.py = -c.y / ac;
                            const double zeta = (b - a) / (2.0 * ac);
                            const double t = copysign(1.0, zeta) / (fabs(zeta) + hypot(1.0, zeta));
                            R.cs = 1.0 / hypot(1.0, t);
                            R.sn = R.cs * t;
                            flag[sweep & 1] = 1;
                        }
                    }
                    sh.rot[q] = R;
                }
                __syncthreads();
                for (int q = w; q < np; q += nw) {
                    const Rot R = sh.rot[q];
                    if (!R.on) continue;
                    const double cs = R.cs, sn = R.sn;
                    const double2 ph = make_double2(R.px, R.py);
                    double2* xi = X + (int64_t)R.i * ldx;
                    double2* xj = X + (int64_t)R.j * ldx;
                    for (int l = lane; l < rows; l += 32) {
                        const double2 u = xi[l], v = cmul(ph, xj[l]);
                        xi[l] = make_double2(cs * u.x - sn * v.x, cs * u.y - sn * v.y);
                        xj[l] = make_double2(sn * u.x + cs * v.x, sn * u.y + cs * v.y);
                    }
                    double2* ji = Jm + (int64_t)R.i * ldj;
                    double2* jj = Jm + (int64_t)R.j * ldj;
                    for (int l = lane; l < r; l += 32) {
                        const double2 u = ji[l], v = cmul(ph, jj[l]);
                        ji[l] = make_double2(cs * u.x - sn * v.x, cs * u.y - sn * v.y);
                        jj[l] = make_double2(sn * u.x + cs * v.x, sn * u.y + cs * v.y);
                    }
                }
                __syncthreads();
            }
            if (tm.size > 1) tm.sync();
        }
        tm.sync();
        const int more = *(volatile int*)(flag + (sweep & 1));
        if (!more) return sweep + 1;
    }
    return maxsweep + 1;
}

// Pivoted Householder QR of the first `cols` columns of A (rows x cols,
// leading dimension ld); `extra` further columns are transformed by the same
// reflectors but never pivoted.  Column j of the result holds the unit
// reflector v_j in rows j..rows-1 (H_j = I - 2 v v^H), diag[j] = R_jj, and
// rows < j of later columns hold R.  Stops at step j when
//   j == min(rows, cols), or
//   the skeleton count is known, j >= it, and the largest remaining column
//   norm is <= rcond * (largest initial norm).
// kfix > 0: skeleton count kfix; else the first j with max norm <= eps * max0.
// The outputs are written by CTA 0 and visible to the team on return; ctl: a
// flag of the team in global memory.
__device__ void cta_cpqr(const Team& tm, double2* A, int ld, int rows, int cols, int extra, int* perm,
                         double2* diag, double* nrm2, double2* s_v, int kfix, double eps,
                         double rcond, Red& red, int* out_rank, int* out_k, double* out_eps, int* ctl) {
    const int lane = threadIdx.x & 31;
    for (int64_t c = tm.thread(); c < cols; c += tm.threads()) perm[c] = (int)c;
    for (int c = tm.warp(); c < cols; c += tm.warps()) {
        double s = 0.0;
        for (int i = lane; i < rows; i += 32) s += cabs2(A[(int64_t)c * ld + i]);
        s = warp_sum(s);
        if (lane == 0) nrm2[c] = s;
    }
    tm.sync();
    double m0 = 0.0;
    for (int c = threadIdx.x; c < cols; c += blockDim.x) m0 = fmax(m0, nrm2[c]);
    const double max0 = block_max(m0, red);
    const int kmax = min(rows, cols);
    int kskel = -1;
    double eps_ach = 0.0;
    int j = 0;
    for (; j < kmax; ++j) {
        // CTA 0 picks the pivot and brings it to column j
        if (tm.rank == 0) {
            double mloc = 0.0;
            for (int c = j + threadIdx.x; c < cols; c += blockDim.x) mloc = fmax(mloc, nrm2[c]);
            const double mx = block_max(mloc, red);
            if (kskel < 0) {
                if (kfix > 0 && j == kfix) {
                    kskel = j;
                    eps_ach = sqrt(mx / max0);
                } else if (kfix <= 0 && mx <= eps * eps * max0) {
                    kskel = j;
                    eps_ach = sqrt(mx / max0);
                }
            }
            const bool stop = (kskel >= 0 && j >= kskel && mx <= rcond * rcond * max0) || mx <= 0.0;
            if (!stop) {
                // pivot: lowest original index among the columns within TIE of the max
                const double thr = (1.0 - TIE) * (1.0 - TIE) * mx;
                int key = INT_MAX, idx = INT_MAX;
                for (int c = j + threadIdx.x; c < cols; c += blockDim.x)
                    if (nrm2[c] >= thr && perm[c] < key) {
                        key = perm[c];
                        idx = c;
                    }
                const int q = block_argmin(key, idx, red);
                if (q != j) {
                    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
                        const double2 t = A[(int64_t)j * ld + i];
                        A[(int64_t)j * ld + i] = A[(int64_t)q * ld + i];
                        A[(int64_t)q * ld + i] = t;
                    }
                    __syncthreads();
                    if (threadIdx.x == 0) {
                        const int tp = perm[j];
                        perm[j] = perm[q];
                        perm[q] = tp;
                        const double tn = nrm2[j];
                        nrm2[j] = nrm2[q];
                        nrm2[q] = tn;
                    }
                }
            }
            if (threadIdx.x == 0) *(volatile int*)ctl = stop ? 1 : 0;
        }
        tm.sync();
        if (*(volatile int*)ctl) break;
        householder_step(tm, A, ld, rows, j, cols, cols + extra, diag, nrm2, s_v, red);
    }
    if (tm.rank == 0 && threadIdx.x == 0) {
        if (kskel < 0) {
            kskel = (kfix > 0) ? min(kfix, j) : j;
            eps_ach = 0.0;
        }
        *out_rank = j;
        *out_k = kskel;
        *out_eps = eps_ach;
    }
    tm.sync();
}

// X(0:n, c) = R(0:n, 0:n)^{-1} Bm(0:n, c) for c < ncols, R upper triangular stored
// above the diagonal of Rm (leading dimension ldr) with its diagonal in diag.
// One thread per right-hand-side column.  X may alias Bm.
__device__ void cta_backsub(const Team& tm, const double2* Rm, int ldr, const double2* diag, int n,
                            const double2* Bm, int ldb, int ncols, double2* X, int ldx) {
    for (int64_t c = tm.thread(); c < ncols; c += tm.threads()) {
        for (int i = n - 1; i >= 0; --i) {
            double2 s = Bm[(int64_t)c * ldb + i];
            for (int l = i + 1; l < n; ++l)
                s = cfms(Rm[(int64_t)l * ldr + i], X[(int64_t)c * ldx + l], s);
            const double2 d = diag[i];
            const double id = 1.0 / cabs2(d);
            X[(int64_t)c * ldx + i] = cscale(cmulc(d, s), id);  // s / d
        }
    }
    tm.sync();
}

}  // namespace

// ----------------------------------------------------------------------------
// phase 1: fill B | D and A, pivoted QR of B (with D)
// ----------------------------------------------------------------------------
// Philox4x32 with 10 rounds (Salmon, Moraes, Dror & Shaw, SC'11).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const unsigned lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const unsigned lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// Entry (i, l) of the complex Gaussian test matrix: counter (l, i, 0, 0), key
// (seed, shape); two 53-bit uniforms in (0, 1) and the Box-Muller transform,
// scaled to unit variance (the same definition as the oracle's).
__device__ __forceinline__ double2 sketch_entry(int i, int l, unsigned seed, int shape) {
    const uint4 w = philox4x32_10(make_uint4((unsigned)l, (unsigned)i, 0u, 0u), make_uint2(seed, (unsigned)shape));
    const double u1 = (double)(((unsigned long long)w.x << 21) + (w.y >> 11)) * 0x1p-53 + 0x1p-54;
    const double u2 = (double)(((unsigned long long)w.z << 21) + (w.w >> 11)) * 0x1p-53 + 0x1p-54;
    const double rad = sqrt(-2.0 * log(u1));
    const double th = 6.283185307179586 * u2;
    const double is2 = 0.70710678118654752440;
    return make_double2(rad * cos(th) * is2, rad * sin(th) * is2);
}

template <int DIM>
__device__ __forceinline__ void sbuild_phase1(const Team& tm, SBuildJob& J, double kappa, double rcond, Red& red,
                                              double2* s_v) {
    fill_kernel_matrix<DIM>(tm, J.BD, J.p, J.z, J.p, J.x, J.m, kappa);
    fill_kernel_matrix<DIM>(tm, J.BD + (int64_t)J.m * J.p, J.p, J.z, J.p, J.y, J.n, kappa);
    fill_kernel_matrix<DIM>(tm, J.AU, J.m, J.x, J.m, J.y, J.n, kappa);
    tm.sync();
    if (J.sketch_d > 0) {
        const int d = J.sketch_d, p = J.p, m = J.m;
        for (int64_t e = tm.thread(); e < (int64_t)d * p; e += tm.threads())
            J.OM[e] = sketch_entry((int)(e % d), (int)(e / d), J.seed, J.shape_index);
        tm.sync();
        for (int64_t e = tm.thread(); e < (int64_t)d * m; e += tm.threads()) {
            const int i = (int)(e % d), j = (int)(e / d);
            double2 sum = make_double2(0.0, 0.0);
            for (int l = 0; l < p; ++l) sum = cfma(J.OM[(int64_t)l * d + i], J.BD[(int64_t)j * p + l], sum);
            J.Y[e] = sum;
        }
        tm.sync();
        // the ID from the sketch: halted at k (a cutoff above every column norm)
        cta_cpqr(tm, J.Y, d, d, m, 0, J.permY, J.diagY, J.nrm2, s_v, J.kfix, 0.0, 2.0, red, &J.rankB, &J.k,
                 &J.eps_ach, J.ctl);
        // B's own factorisation, for the least-squares solve of C
        cta_cpqr(tm, J.BD, J.p, J.p, J.m, J.n, J.permB, J.diagB, J.nrm2, s_v, J.kfix, J.eps, B_QR_CUT * rcond, red,
                 &J.rankB, J.ctl + 1, (double*)(J.ctl + 2), J.ctl);
        return;
    }
    cta_cpqr(tm, J.BD, J.p, J.p, J.m, J.n, J.permB, J.diagB, J.nrm2, s_v, J.kfix, J.eps, B_QR_CUT * rcond, red,
             &J.rankB, &J.k, &J.eps_ach, J.ctl);
}

// ----------------------------------------------------------------------------
// phase 2: Z*, C (minimum norm), U, pivoted QR of A (with U)
// ----------------------------------------------------------------------------
__device__ __forceinline__ void sbuild_phase2(const Team& tm, SBuildJob& J, double rcond, Red& red, double2* s_v) {
    const int m = J.m, n = J.n, p = J.p, k = J.k, rB = J.rankB;
    // the ID's factorisation: B's own pivoted QR, or the sketch's
    const bool sk = J.sketch_d > 0;
    const double2* RI = sk ? J.Y : J.BD;
    const int ldi = sk ? J.sketch_d : p;
    const int* permI = sk ? J.permY : J.permB;
    const double2* diagI = sk ? J.diagY : J.diagB;
    // skeleton indices
    for (int64_t i = tm.thread(); i < k; i += tm.threads()) J.skel[i] = permI[i];
    // Z* (k x m, ld k): identity on the skeleton, T = R11^{-1} R12 elsewhere
    for (int64_t e = tm.thread(); e < (int64_t)k * m; e += tm.threads()) J.Zs[e] = make_double2(0.0, 0.0);
    tm.sync();
    for (int64_t i = tm.thread(); i < k; i += tm.threads())
        J.Zs[(int64_t)permI[i] * k + i] = make_double2(1.0, 0.0);
    // T columns: solve into the work area W1 (k x (m-k), ld k)
    cta_backsub(tm, RI, ldi, diagI, k, RI + (int64_t)k * ldi, ldi, m - k, J.W1, k);
    for (int64_t e = tm.thread(); e < (int64_t)k * (m - k); e += tm.threads()) {
        const int i = (int)(e % k), c = (int)(e / k);
        J.Zs[(int64_t)permI[k + c] * k + i] = J.W1[e];
    }
    // C (m x n, ld m): minimum-norm solution of R_B (C P_B) = (Q_B^H D)(0:rB, :) with
    // R_B = [R11 R12] (rB x m, upper trapezoidal, pivot order).  Complete
    // orthogonal decomposition by reflectors from the right (the RZ reduction):
    // for rows i = rB-1 .. 0 a reflector P_i on column i and columns rB..m-1
    // zeroes row i of R12, so R_B P_{rB-1} ... P_0 = [T 0] with T upper
    // triangular; then C P_B = P_{rB-1} ... P_0 [T^{-1} (Q_B^H D)(0:rB, :); 0].
    // A reflector has 1 + m - rB entries (m - rB is small when B is close to
    // full rank), so this costs O(rB^2 (m - rB)), not the O(m rB^2) of a QR of
    // R_B^H.  V (1 + m - rB) x rB in XB holds the unit reflectors.
    {
        const int L = m - rB + 1;
        double2* V = J.XB;
        const int lane = threadIdx.x & 31;
        // entry l of row r's reduced vector: column r (l = 0) or column rB + l - 1
        auto col_of = [&](int r, int l) { return l == 0 ? r : rB + l - 1; };
        if (L > 1) {
            for (int i = rB - 1; i >= 0; --i) {
                double sl = 0.0;
                for (int l = threadIdx.x; l < L; l += blockDim.x)
                    sl += cabs2(l == 0 ? J.diagB[i] : J.BD[(int64_t)col_of(i, l) * p + i]);
                const double nx2 = block_sum(sl, red);
                // a = conj(u) with u = row i's vector; P a = alpha e1, so u P = conj(alpha) e1
                const double2 u0 = J.diagB[i];
                const double2 a0 = make_double2(u0.x, -u0.y);
                const double ax0 = sqrt(cabs2(a0));
                const double2 ph = ax0 > 0.0 ? make_double2(a0.x / ax0, a0.y / ax0) : make_double2(1.0, 0.0);
                const double nx = sqrt(nx2);
                const double2 alpha = make_double2(-ph.x * nx, -ph.y * nx);
                const double2 v0 = csub(a0, alpha);
                const double nv2 = nx2 - ax0 * ax0 + cabs2(v0);
                const double inv = nv2 > 0.0 ? 1.0 / sqrt(nv2) : 0.0;
                for (int l = threadIdx.x; l < L; l += blockDim.x) {
                    double2 v;
                    if (l == 0) {
                        v = cscale(v0, inv);
                    } else {
                        const double2 u = J.BD[(int64_t)col_of(i, l) * p + i];
                        v = cscale(make_double2(u.x, -u.y), inv);
                    }
                    s_v[l] = v;
                }
                __syncthreads();
                // rows r < i: w <- w P_i = w - 2 (w . v) v^H
                for (int r = tm.warp(); r < i; r += tm.warps()) {
                    double2 d = make_double2(0.0, 0.0);
                    for (int l = lane; l < L; l += 32) d = cfma(J.BD[(int64_t)col_of(i, l) * p + r], s_v[l], d);
                    d = cscale(warp_sum2(d), 2.0);
                    for (int l = lane; l < L; l += 32) {
                        double2& x = J.BD[(int64_t)col_of(i, l) * p + r];
                        x = cfmsc(s_v[l], d, x);  // x - conj(v_l) d
                    }
                }
                tm.sync();  // every CTA has read row i and R(i, i)
                if (tm.rank == 0) {
                    for (int l = threadIdx.x; l < L; l += blockDim.x) {
                        V[(int64_t)i * L + l] = s_v[l];
                        if (l > 0) J.BD[(int64_t)col_of(i, l) * p + i] = make_double2(0.0, 0.0);
                    }
                    if (threadIdx.x == 0) J.diagB[i] = make_double2(alpha.x, -alpha.y);
                }
                __syncthreads();
            }
            tm.sync();
        }
        // Y = T^{-1} (Q_B^H D)(0:rB, :) into W2 (rB x n, ld rB), T now in R_B's place
        const int ldy = rB > 0 ? rB : 1;
        cta_backsub(tm, J.BD, p, J.diagB, rB, J.BD + (int64_t)m * p, p, n, J.W2, ldy);
        for (int64_t e = tm.thread(); e < (int64_t)m * n; e += tm.threads()) {
            const int i = (int)(e % m), c = (int)(e / m);
            J.W3[e] = i < rB ? J.W2[(int64_t)c * ldy + i] : make_double2(0.0, 0.0);
        }
        tm.sync();
        // W3 <- P_{rB-1} ... P_0 W3 (P_0 first), P_i x = x - 2 v (v^H x); a column
        // stays with one warp
        if (L > 1) {
            for (int c = tm.warp(); c < n; c += tm.warps()) {
                for (int i = 0; i < rB; ++i) {
                    double2* x = J.W3 + (int64_t)c * m;
                    double2 d = make_double2(0.0, 0.0);
                    for (int l = lane; l < L; l += 32) d = cfmac(V[(int64_t)i * L + l], x[col_of(i, l)], d);
                    d = cscale(warp_sum2(d), 2.0);
                    for (int l = lane; l < L; l += 32)
                        x[col_of(i, l)] = cfms(V[(int64_t)i * L + l], d, x[col_of(i, l)]);
                    __syncwarp();  // x[i] is read by another lane in a later step
                }
            }
            tm.sync();
        }
    }
    for (int64_t e = tm.thread(); e < (int64_t)m * n; e += tm.threads()) {
        const int i = (int)(e % m), c = (int)(e / m);
        J.C[(int64_t)c * m + J.permB[i]] = J.W3[e];
    }
    // U = (Z*)^T into AU columns n..n+k-1 (m x k, ld m)
    tm.sync();
    for (int64_t e = tm.thread(); e < (int64_t)m * k; e += tm.threads()) {
        const int i = (int)(e % m), c = (int)(e / m);
        J.AU[(int64_t)(n + c) * m + i] = J.Zs[(int64_t)i * k + c];
    }
    tm.sync();
    // pivoted QR of A (m x n), reflectors applied to U, run down to the
    // rounding level: the truncation itself is done on the singular values
    const double rq = 0.01 * rcond;
    cta_cpqr(tm, J.AU, m, m, n, k, J.permA, J.diagA, J.nrm2, s_v, -1, rq, rq, red, &J.rankA, J.ctl + 1,
             (double*)(J.ctl + 2), J.ctl);
}

// ----------------------------------------------------------------------------
// phase 3: truncated SVD of A from its pivoted QR (one-sided Jacobi on
// R_A^H), the factors of A^+, and S
// ----------------------------------------------------------------------------
__device__ __forceinline__ void sbuild_phase3(const Team& tm, SBuildJob& J, double rcond, Red& red, int& s_r,
                                              JacobiShared& jac) {
    const int m = J.m, n = J.n, k = J.k, rA = J.rankA;
    const int lane = threadIdx.x & 31;
    // X = R_A^H (n x rA, ld n) and J = I (rA x rA, ld n)
    for (int64_t e = tm.thread(); e < (int64_t)n * rA; e += tm.threads()) {
        const int c = (int)(e % n), i = (int)(e / n);
        double2 v = make_double2(0.0, 0.0);
        if (c == i)
            v = J.diagA[i];
        else if (c > i)
            v = J.AU[(int64_t)c * m + i];
        J.XA[e] = make_double2(v.x, -v.y);
    }
    for (int64_t e = tm.thread(); e < (int64_t)rA * rA; e += tm.threads()) {
        const int l = (int)(e % rA), i = (int)(e / rA);
        J.JA[(int64_t)i * n + l] = make_double2(l == i ? 1.0 : 0.0, 0.0);
    }
    tm.sync();
    const double tol = 2.220446049250313e-16 * sqrt((double)max(n, 1));
    const int sweeps = cta_jacobi(tm, J.XA, n, n, rA, J.JA, n, tol, 60, J.ctl, jac);
    // singular values = column norms of X J
    for (int i = tm.warp(); i < rA; i += tm.warps()) {
        double sum = 0.0;
        for (int l = lane; l < n; l += 32) sum = abs2_acc(J.XA[(int64_t)i * n + l], sum);
        sum = warp_sum(sum);
        if (lane == 0) J.sig[i] = sqrt(sum);
    }
    tm.sync();
    double mloc = 0.0;
    for (int i = threadIdx.x; i < rA; i += blockDim.x) mloc = fmax(mloc, J.sig[i]);
    const double smax = block_max(mloc, red);
    if (threadIdx.x == 0) {
        int r = 0;
        for (int i = 0; i < rA; ++i)
            if (J.sig[i] > rcond * smax) J.keep[r++] = i;
        s_r = r;
        if (tm.rank == 0) {
            J.rankS = r;
            J.sweepsA = sweeps;
        }
    }
    __syncthreads();
    const int r = s_r;
    // F = P_A V_r Sigma_r^{-1} = P_A (X J)(:, kept) Sigma_r^{-2}  (n x r, ld n, rows in
    // the original column order of A)
    for (int64_t e = tm.thread(); e < (int64_t)n * r; e += tm.threads()) {
        const int row = (int)(e % n), slot = (int)(e / n);
        const int i = J.keep[slot];
        const double sg = J.sig[i];
        J.FA[(int64_t)slot * n + J.permA[row]] = cscale(J.XA[(int64_t)i * n + row], 1.0 / (sg * sg));
    }
    // kept columns of J moved to the front, in order (a source column is never
    // the destination of an earlier one)
    for (int slot = 0; tm.rank == 0 && slot < r; ++slot) {
        const int i = J.keep[slot];
        if (i != slot)
            for (int l = threadIdx.x; l < rA; l += blockDim.x)
                J.JA[(int64_t)slot * n + l] = J.JA[(int64_t)i * n + l];
        __syncthreads();
    }
    tm.sync();
    // M = Z* C (k x n, ld k) into W1
    for (int64_t e = tm.thread(); e < (int64_t)k * n; e += tm.threads()) {
        const int i = (int)(e % k), c = (int)(e / k);
        double2 sum = make_double2(0.0, 0.0);
        for (int l = 0; l < m; ++l) sum = cfma(J.Zs[(int64_t)l * k + i], J.C[(int64_t)c * m + l], sum);
        J.W1[e] = sum;
    }
    // H = J_r^H (Q_A^H U)(0:rA, :)  (r x k, ld r) into W3
    const int ldh = r > 0 ? r : 1;
    for (int64_t e = tm.thread(); e < (int64_t)r * k; e += tm.threads()) {
        const int i = (int)(e % ldh), c = (int)(e / ldh);
        double2 sum = make_double2(0.0, 0.0);
        for (int l = 0; l < rA; ++l)
            sum = cfmac(J.JA[(int64_t)i * n + l], J.AU[(int64_t)(n + c) * m + l], sum);
        J.W3[e] = sum;
    }
    tm.sync();
    // G = M F  (k x r, ld k) into XB
    for (int64_t e = tm.thread(); e < (int64_t)k * r; e += tm.threads()) {
        const int i = (int)(e % k), c = (int)(e / k);
        double2 sum = make_double2(0.0, 0.0);
        for (int l = 0; l < n; ++l) sum = cfma(J.W1[(int64_t)l * k + i], J.FA[(int64_t)c * n + l], sum);
        J.XB[e] = sum;
    }
    tm.sync();
    // S = G H  (k x k, ld k), and its Frobenius norm
    for (int64_t e = tm.thread(); e < (int64_t)k * k; e += tm.threads()) {
        const int i = (int)(e % k), c = (int)(e / k);
        double2 sum = make_double2(0.0, 0.0);
        for (int l = 0; l < r; ++l) sum = cfma(J.XB[(int64_t)l * k + i], J.W3[(int64_t)c * ldh + l], sum);
        J.S[e] = sum;
    }
    tm.sync();
    if (tm.rank != 0) return;
    double sq = 0.0;
    for (int64_t e = threadIdx.x; e < (int64_t)k * k; e += blockDim.x) sq += cabs2(J.S[e]);
    sq = block_sum(sq, red);
    if (threadIdx.x == 0) J.snorm = sqrt(sq);
}

// ----------------------------------------------------------------------------
// persistent launches: every CTA takes the next shape from an atomic counter.
// The host orders the shapes by decreasing work, so this is longest-
// processing-time-first scheduling over uneven sizes, and a launch covers the
// whole batch with a grid sized to the GPU.  The three phases stay separate
// kernels (one register allocation each; a fused kernel spilled).
// ----------------------------------------------------------------------------
__device__ __forceinline__ int next_job(int* counter, int* s_job) {
    if (threadIdx.x == 0) *s_job = atomicAdd(counter, 1);
    __syncthreads();
    const int j = *s_job;
    __syncthreads();  // every thread holds j before thread 0 fetches the next one
    return j;
}

// f(team, job) for the jobs of this CTA, or the one job of the cluster of `size`
// CTAs that it belongs to.  One call site: two copies of a phase may contract
// their products and sums differently.
template <typename F>
__device__ __forceinline__ void each_job(int size, int njobs, int* counter, int* s_job, F&& f) {
    const Team tm{size > 1 ? (int)(blockIdx.x % size) : 0, size};
    int j = size > 1 ? (int)(blockIdx.x / size) : next_job(counter, s_job);
    while (j < njobs) {
        f(tm, j);
        j = size > 1 ? njobs : next_job(counter, s_job);
    }
}

template <int DIM>
__global__ void __launch_bounds__(SBT_MAX) sbuild_phase1_kernel(SBuildJob* jobs, int njobs, int* counter, int team,
                                                                double kappa, double rcond) {
    __shared__ Red red;
    __shared__ int s_job;
    extern __shared__ double2 s_v[];
    each_job(team, njobs, counter, &s_job,
             [&](const Team& tm, int j) { sbuild_phase1<DIM>(tm, jobs[j], kappa, rcond, red, s_v); });
}

__global__ void __launch_bounds__(SBT_MAX) sbuild_phase2_kernel(SBuildJob* jobs, int njobs, int* counter, int team,
                                                                double rcond) {
    __shared__ Red red;
    __shared__ int s_job;
    extern __shared__ double2 s_v[];
    each_job(team, njobs, counter, &s_job,
             [&](const Team& tm, int j) { sbuild_phase2(tm, jobs[j], rcond, red, s_v); });
}

__global__ void __launch_bounds__(SBT_MAX) sbuild_phase3_kernel(SBuildJob* jobs, int njobs, int* counter, int team,
                                                                double rcond) {
    __shared__ Red red;
    __shared__ int s_job, s_r;
    __shared__ JacobiShared jac;
    each_job(team, njobs, counter, &s_job,
             [&](const Team& tm, int j) { sbuild_phase3(tm, jobs[j], rcond, red, s_r, jac); });
}

// ----------------------------------------------------------------------------
// right-hand side b_tau = Z* C A^+ v_tau, right to left, one CTA per (body, rhs)
// ----------------------------------------------------------------------------
// qm = A^+ t for one body from the stored factors of the truncated SVD:
// t <- Q_A^H t by the Householder reflectors, z = J_r^H t(0:rA) (r values),
// qm = F z with F = P_A V_r Sigma_r^{-1}.  t (m), z (n) and qm (n) are in
// shared memory; every thread of the block takes part.
__device__ void apply_Apinv(const RhsBody& B, double2* t, double2* z, double2* qm, double* rs,
                            double* rs2) {
    const int m = B.m, n = B.n;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int j = 0; j < B.rankA; ++j) {
        const double2* vj = B.A + (int64_t)j * m;
        double2 d = make_double2(0.0, 0.0);
        for (int i = j + threadIdx.x; i < m; i += blockDim.x) d = cadd(d, cmulc(vj[i], t[i]));
        d = warp_sum2(d);
        __syncthreads();
        if (lane == 0) {
            rs[w] = d.x;
            rs2[w] = d.y;
        }
        __syncthreads();
        double2 tot = make_double2(0.0, 0.0);
        for (int k2 = 0; k2 < nw; ++k2) {
            tot.x += rs[k2];
            tot.y += rs2[k2];
        }
        tot = cscale(tot, 2.0);
        for (int i = j + threadIdx.x; i < m; i += blockDim.x) t[i] = csub(t[i], cmul(vj[i], tot));
        __syncthreads();
    }
    for (int s = threadIdx.x; s < B.rankS; s += blockDim.x) {
        double2 sum = make_double2(0.0, 0.0);
        for (int l = 0; l < B.rankA; ++l) sum = cadd(sum, cmulc(B.J[(int64_t)s * n + l], t[l]));
        z[s] = sum;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double2 sum = make_double2(0.0, 0.0);
        for (int s = 0; s < B.rankS; ++s) sum = cadd(sum, cmul(B.F[(int64_t)s * n + i], z[s]));
        qm[i] = sum;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(256) rhs_kernel(const RhsBody* __restrict__ bodies, int T,
                                                  const double2* __restrict__ v, int64_t Mtot,
                                                  double2* __restrict__ b, int64_t N) {
    __shared__ double rs[8], rs2[8];
    extern __shared__ double2 sm[];
    const int tau = blockIdx.x, r = blockIdx.y;
    const RhsBody B = bodies[tau];
    const int m = B.m, n = B.n, k = B.k;
    double2* t = sm;              // m
    double2* qm = sm + m;         // n
    double2* q = sm + m + n;      // m
    double2* z = sm + 2 * m + n;  // n
    const double2* vin = v + (int64_t)r * Mtot + B.voff;
    for (int i = threadIdx.x; i < m; i += blockDim.x) t[i] = vin[i];
    __syncthreads();
    if (B.W) {  // injected W: b = W v
        for (int i = threadIdx.x; i < k; i += blockDim.x) {
            double2 s = make_double2(0.0, 0.0);
            for (int l = 0; l < m; ++l) s = cadd(s, cmul(B.W[(int64_t)l * k + i], t[l]));
            b[(int64_t)r * N + B.boff + i] = s;
        }
        return;
    }
    apply_Apinv(B, t, z, qm, rs, rs2);
    // q = C q_mfs
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double2 s = make_double2(0.0, 0.0);
        for (int l = 0; l < n; ++l) s = cadd(s, cmul(B.C[(int64_t)l * m + i], qm[l]));
        q[i] = s;
    }
    __syncthreads();
    // b = Z* q
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        double2 s = make_double2(0.0, 0.0);
        for (int l = 0; l < m; ++l) s = cadd(s, cmul(B.Zs[(int64_t)l * k + i], q[l]));
        b[(int64_t)r * N + B.boff + i] = s;
    }
}

// Sec. 4.6: q_mfs = A^+ (v - U w_hat), U(i, a) = Z*(a, i).
__global__ void __launch_bounds__(256) recon_kernel(const RhsBody* __restrict__ bodies, int T,
                                                    const double2* __restrict__ v, int64_t Mtot,
                                                    const double2* __restrict__ w_hat, int64_t N,
                                                    double2* __restrict__ qmfs, int64_t Nm) {
    __shared__ double rs[8], rs2[8];
    extern __shared__ double2 sm[];
    const int tau = blockIdx.x, r = blockIdx.y;
    const RhsBody B = bodies[tau];
    const int m = B.m, n = B.n, k = B.k;
    double2* t = sm;           // m
    double2* qm = sm + m;      // n
    double2* z = sm + m + n;   // n
    const double2* vin = v + (int64_t)r * Mtot + B.voff;
    const double2* wh = w_hat + (int64_t)r * N + B.boff;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double2 s = vin[i];
        for (int a = 0; a < k; ++a) s = csub(s, cmul(B.Zs[(int64_t)i * k + a], wh[a]));
        t[i] = s;
    }
    __syncthreads();
    apply_Apinv(B, t, z, qm, rs, rs2);
    for (int j = threadIdx.x; j < n; j += blockDim.x) qmfs[(int64_t)r * Nm + B.moff + j] = qm[j];
}

// ----------------------------------------------------------------------------
// The same for bodies of at most 256 collocation points: one CTA per body and
// block of up to 8 right-hand sides (rhs_per_cta), one warp per right-hand side through the
// reflectors, then all threads over the entries of the five products.
//
// The FP64 pipe bounds this (64 cycles a warp instruction and scheduler).  The
// kernels above give a right-hand side 8 warps, of which m = 128 rows fill 4;
// every warp spends 10 additions on its part of a dot product and 16 on the
// total, next to 8 for the rows themselves, and three CTA barriers.  Here a
// warp holds all row groups, adds them by a scatter (8 partial sums a lane
// become one in 4 + 2 + 1 additions), and waits for nobody.  Every sum is
// formed in the order of the kernels above (32 consecutive rows from row j by
// the exchange tree, then the groups in order), so the results are the same to
// the bit.  1000 bodies, m = 128, n = k = 64, 8 right-hand sides: 10.5 ms to
// 4.2 ms.
// ----------------------------------------------------------------------------
constexpr int RB = 8;          // right-hand sides per CTA = warps
constexpr int RB_GROUPS = 8;   // groups of 32 rows: m <= 256

// One step of the tree lane ^ 16, 8, 4, 2, 1 for a value that this lane keeps: the
// partner's copy of it is added.
__device__ __forceinline__ double xchg_add(double keep, double send, int o) {
    return keep + __shfl_xor_sync(0xffffffffu, send, o);
}

// Totals over the rows of one reflector step: p[g] are this lane's products of
// row group g; returns sum_g (tree sum of p[g]), groups in order.
template <int G>
__device__ __forceinline__ double2 rows_total(const double2 (&p)[G]) {
    static_assert(G == 4 || G == 8, "row groups");
    const int lane = threadIdx.x & 31;
    double v[2 * G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        v[2 * g] = p[g].x;
        v[2 * g + 1] = p[g].y;
    }
    // halve the values a lane holds while the tree's partners meet: step o adds
    // the partner's copy of the values this lane keeps
    int o = 16;
#pragma unroll
    for (int n = 2 * G; n > 1; n >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const double keep = up ? v[i + n / 2] : v[i], send = up ? v[i] : v[i + n / 2];
            v[i] = xchg_add(keep, send, o);
        }
    }
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    // value i sits in the lanes whose top log2(2 G) bits spell i
    constexpr int W = 32 / (2 * G);
    double2 tot = make_double2(0.0, 0.0);
#pragma unroll
    for (int g = 0; g < G; ++g) {
        tot.x += __shfl_sync(0xffffffffu, v[0], W * (2 * g));
        tot.y += __shfl_sync(0xffffffffu, v[0], W * (2 * g + 1));
    }
    return tot;
}

// t <- Q_A^H t for one right-hand side, by one warp
template <int G>
__device__ __forceinline__ void warp_reflect(const RhsBody& B, double2* t) {
    const int m = B.m, lane = threadIdx.x & 31;
    double2 nxt[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const int i = 32 * g + lane;
        nxt[g] = i < m && B.rankA > 0 ? B.A[i] : make_double2(0.0, 0.0);
    }
    for (int j = 0; j < B.rankA; ++j) {
        double2 vj[G], tt[G], p[G];
#pragma unroll
        for (int g = 0; g < G; ++g) vj[g] = nxt[g];
        if (j + 1 < B.rankA) {
            const double2* vn = B.A + (int64_t)(j + 1) * m;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int i = j + 1 + 32 * g + lane;
                nxt[g] = i < m ? vn[i] : make_double2(0.0, 0.0);
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int i = j + 32 * g + lane;
            tt[g] = i < m ? t[i] : make_double2(0.0, 0.0);
            p[g] = i < m ? cmulc(vj[g], tt[g]) : make_double2(0.0, 0.0);
        }
        const double2 tot = cscale(rows_total<G>(p), 2.0);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int i = j + 32 * g + lane;
            if (i < m) t[i] = csub(tt[g], cmul(vj[g], tot));
        }
        __syncwarp();
    }
}

// Entries e = i + rows * r of an output of `rows` rows for the nr right-hand
// sides: every thread takes whole rows for one right-hand side at a time.
template <typename F>
__device__ __forceinline__ void each_entry(int rows, int nr, F&& f) {
    for (int e = threadIdx.x; e < rows * nr; e += blockDim.x) f(e % rows, e / rows);
}

// qm = A^+ t for the nr right-hand sides (t: [RB][m], z, qm: [RB][n])
__device__ __forceinline__ void block_Apinv(const RhsBody& B, double2* t, double2* z, double2* qm, int nr) {
    const int m = B.m, n = B.n, w = threadIdx.x >> 5;
    if (w < nr) {
        if (m <= 128)
            warp_reflect<4>(B, t + (int64_t)w * m);
        else
            warp_reflect<8>(B, t + (int64_t)w * m);
    }
    __syncthreads();
    each_entry(B.rankS, nr, [&](int s, int r) {
        double2 sum = make_double2(0.0, 0.0);
        for (int l = 0; l < B.rankA; ++l) sum = cadd(sum, cmulc(B.J[(int64_t)s * n + l], t[(int64_t)r * m + l]));
        z[(int64_t)r * n + s] = sum;
    });
    __syncthreads();
    each_entry(n, nr, [&](int i, int r) {
        double2 sum = make_double2(0.0, 0.0);
        for (int s = 0; s < B.rankS; ++s) sum = cadd(sum, cmul(B.F[(int64_t)s * n + i], z[(int64_t)r * n + s]));
        qm[(int64_t)r * n + i] = sum;
    });
    __syncthreads();
}

__global__ void __launch_bounds__(32 * RB) rhs_block_kernel(const RhsBody* __restrict__ bodies, const int nrhs,
                                                            const int rb, const int mmax, const int nmax,
                                                            const double2* __restrict__ v, const int64_t Mtot,
                                                            double2* __restrict__ b, const int64_t N) {
    extern __shared__ double2 sm[];
    const RhsBody B = bodies[blockIdx.x];
    const int r0 = blockIdx.y * rb, nr = min(rb, nrhs - r0);
    const int m = B.m, n = B.n, k = B.k;
    double2* t = sm;                      // [rb][m]; later C q_mfs
    double2* qm = sm + (int64_t)rb * mmax;  // [rb][n]
    double2* z = qm + (int64_t)rb * nmax;   // [rb][n]
    each_entry(m, nr, [&](int i, int r) { t[(int64_t)r * m + i] = v[(int64_t)(r0 + r) * Mtot + B.voff + i]; });
    __syncthreads();
    if (B.W) {  // injected W: b = W v
        each_entry(k, nr, [&](int i, int r) {
            double2 s = make_double2(0.0, 0.0);
            for (int l = 0; l < m; ++l) s = cadd(s, cmul(B.W[(int64_t)l * k + i], t[(int64_t)r * m + l]));
            b[(int64_t)(r0 + r) * N + B.boff + i] = s;
        });
        return;
    }
    block_Apinv(B, t, z, qm, nr);
    // q = C q_mfs
    each_entry(m, nr, [&](int i, int r) {
        double2 s = make_double2(0.0, 0.0);
        for (int l = 0; l < n; ++l) s = cadd(s, cmul(B.C[(int64_t)l * m + i], qm[(int64_t)r * n + l]));
        t[(int64_t)r * m + i] = s;
    });
    __syncthreads();
    // b = Z* q
    each_entry(k, nr, [&](int i, int r) {
        double2 s = make_double2(0.0, 0.0);
        for (int l = 0; l < m; ++l) s = cadd(s, cmul(B.Zs[(int64_t)l * k + i], t[(int64_t)r * m + l]));
        b[(int64_t)(r0 + r) * N + B.boff + i] = s;
    });
}

__global__ void __launch_bounds__(32 * RB) recon_block_kernel(const RhsBody* __restrict__ bodies, const int nrhs,
                                                              const int rb, const int mmax, const int nmax,
                                                              const double2* __restrict__ v, const int64_t Mtot,
                                                              const double2* __restrict__ w_hat, const int64_t N,
                                                              double2* __restrict__ qmfs, const int64_t Nm) {
    extern __shared__ double2 sm[];
    const RhsBody B = bodies[blockIdx.x];
    const int r0 = blockIdx.y * rb, nr = min(rb, nrhs - r0);
    const int m = B.m, n = B.n, k = B.k;
    double2* t = sm;
    double2* qm = sm + (int64_t)rb * mmax;
    double2* z = qm + (int64_t)rb * nmax;
    each_entry(m, nr, [&](int i, int r) {
        double2 s = v[(int64_t)(r0 + r) * Mtot + B.voff + i];
        const double2* wh = w_hat + (int64_t)(r0 + r) * N + B.boff;
        for (int a = 0; a < k; ++a) s = csub(s, cmul(B.Zs[(int64_t)i * k + a], wh[a]));
        t[(int64_t)r * m + i] = s;
    });
    __syncthreads();
    block_Apinv(B, t, z, qm, nr);
    each_entry(n, nr, [&](int i, int r) {
        qmfs[(int64_t)(r0 + r) * Nm + B.moff + i] = qm[(int64_t)r * n + i];
    });
}

template <typename K>
static int blocks_per_sm(K* kern, int threads, size_t sm) {
    if (sm > 48 * 1024)
        MBS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    int nb = 0;
    MBS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, threads, sm));
    return std::max(nb, 1);
}

// Launch of a build phase: a persistent grid of single CTAs, or one cluster of
// `team` CTAs per job.
template <typename... A>
static void launch_phase(void (*kern)(A...), int njobs, int team, int threads, size_t sm, cudaStream_t st, A... args) {
    const int per = blocks_per_sm(kern, threads, sm);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(team > 1 ? njobs * team : std::min(njobs, mbs_num_sms() * per)));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)team;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = team > 1 ? 1 : 0;
    MBS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, args...));
    MBS_CHECK_LAUNCH();
}

void launch_sbuild(int dim, SBuildJob* d_jobs, int njobs, int* d_counter, int rows_max, int threads,
                   double kappa, double rcond, cudaStream_t st) {
    if (njobs == 0) return;
    if (threads != 128 && threads != 256 && threads != 512)
        throw MbsError{MBS_ERR_ARG, "S build: threads per CTA must be 128, 256 or 512"};
    const size_t sm = (size_t)std::max(rows_max, 1) * sizeof(double2);
    // CTAs per shape: a shape alone on an SM is bound by that SM's FP64 pipe and
    // by the latency of its steps, so few shapes are shared out over clusters of
    // up to 8 CTAs (the portable size) while every CTA still finds an SM.  Phases
    // 1, 2 and 3 of 3 shapes with 128 points: 8.7, 5.9, 28.1 ms to 2.6, 3.2,
    // 6.3 ms; of 6 ellipsoids with 192: 17.2, 9.2, 15.7 ms to 4.5, 5.4, 4.3 ms.
    int team = 8;
    while (team > 1 && njobs * team > mbs_num_sms()) team /= 2;
    MBS_CUDA_TRY(cudaMemsetAsync(d_counter, 0, 3 * sizeof(int), st));
    if (dim == 2)
        launch_phase(sbuild_phase1_kernel<2>, njobs, team, threads, sm, st, d_jobs, njobs, d_counter, team, kappa, rcond);
    else
        launch_phase(sbuild_phase1_kernel<3>, njobs, team, threads, sm, st, d_jobs, njobs, d_counter, team, kappa, rcond);
    launch_phase(sbuild_phase2_kernel, njobs, team, threads, sm, st, d_jobs, njobs, d_counter + 1, team, rcond);
    launch_phase(sbuild_phase3_kernel, njobs, team, threads, (size_t)0, st, d_jobs, njobs, d_counter + 2, team, rcond);
}

// Right-hand sides per CTA of the blocked kernels; 0 where the general ones are
// faster.  A CTA takes 260 us for one right-hand side of 128 points and 640 us
// for 8, alone on its SM; so few bodies get as few per CTA as still find an SM
// each (the general kernel: 315 us a round of CTAs), many bodies 8 (1000 bodies,
// 8 right-hand sides: 4.2 ms, general 10.6; but 1 right-hand side: 1.58 ms, 1.48).
// Of 256 points: 770 and 2190 us against 640, so only many bodies with 4 or more
// right-hand sides gain (200 bodies, 8: 4.3 ms, general 5.5).
static int rhs_per_cta(int T, int nrhs, int mmax) {
    if (mmax > 32 * RB_GROUPS) return 0;
    const int64_t sms = mbs_num_sms(), all = (int64_t)T * nrhs;
    if (mmax > 128) return nrhs >= 4 && all >= 4 * sms ? RB : 0;
    for (int rb = 1; rb < RB; rb *= 2)
        if ((int64_t)T * ((nrhs + rb - 1) / rb) <= sms) return rb;
    return nrhs > 1 ? std::min(RB, nrhs) : 0;
}

void launch_rhs(const RhsBody* d_bodies, int T, int nrhs, int mmax, int nmax, const double2* v,
                int64_t Mtot, double2* b, int64_t N, cudaStream_t st) {
    if (T == 0 || nrhs == 0) return;
    if (const int rb = rhs_per_cta(T, nrhs, mmax)) {
        const size_t smb = (size_t)rb * (mmax + 2 * nmax) * sizeof(double2);
        if (smb > 48 * 1024)
            MBS_CUDA_TRY(cudaFuncSetAttribute(rhs_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smb));
        const dim3 gb((unsigned)T, (unsigned)((nrhs + rb - 1) / rb));
        rhs_block_kernel<<<gb, 32 * RB, smb, st>>>(d_bodies, nrhs, rb, mmax, nmax, v, Mtot, b, N);
        MBS_CHECK_LAUNCH();
        return;
    }
    const size_t sm = (size_t)(2 * mmax + 2 * nmax) * sizeof(double2);
    if (sm > 48 * 1024)
        MBS_CUDA_TRY(cudaFuncSetAttribute(rhs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)sm));
    dim3 g((unsigned)T, (unsigned)nrhs);
    rhs_kernel<<<g, 256, sm, st>>>(d_bodies, T, v, Mtot, b, N);
    MBS_CHECK_LAUNCH();
}

void launch_recon(const RhsBody* d_bodies, int T, int nrhs, int mmax, int nmax, const double2* v,
                  int64_t Mtot, const double2* w_hat, int64_t N, double2* qmfs, int64_t Nm,
                  cudaStream_t st) {
    if (T == 0 || nrhs == 0) return;
    if (const int rb = rhs_per_cta(T, nrhs, mmax)) {
        const size_t smb = (size_t)rb * (mmax + 2 * nmax) * sizeof(double2);
        if (smb > 48 * 1024)
            MBS_CUDA_TRY(cudaFuncSetAttribute(recon_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smb));
        const dim3 gb((unsigned)T, (unsigned)((nrhs + rb - 1) / rb));
        recon_block_kernel<<<gb, 32 * RB, smb, st>>>(d_bodies, nrhs, rb, mmax, nmax, v, Mtot, w_hat, N, qmfs, Nm);
        MBS_CHECK_LAUNCH();
        return;
    }
    const size_t sm = (size_t)(mmax + 2 * nmax) * sizeof(double2);
    if (sm > 48 * 1024)
        MBS_CUDA_TRY(cudaFuncSetAttribute(recon_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)sm));
    dim3 g((unsigned)T, (unsigned)nrhs);
    recon_kernel<<<g, 256, sm, st>>>(d_bodies, T, v, Mtot, w_hat, N, qmfs, Nm);
    MBS_CHECK_LAUNCH();
}
