// One-time precomputation of Alg. 1 on the GPU, all in FP64:
//   K4  GS weights/exponents by sinc quadrature (eq. sin_1_x)
//   K5  1D integral tables G, H of eq. (Gten_sep) per axis
//   K6  multiplier M_k = -|kappa|^2 Vhat_k / Ntilde (eqs. Gten_sep, convtheorem)
//   K7  FFT twiddles exp(-2 pi i j / N)
//   and, for passes on lengths F > 2n, the multiplier of period F (sp_embed.cuh)
// K5, K6 and the change of period are contractions over a long index (quadrature nodes, GS
// terms, wavenumbers), each in a tiled FP64 kernel of its shape: k_axis_sums, k_dgemm_nt with
// problem-specific operands and epilogues, k_dgemm_nn along strided axes.
#include <math.h>
#include <stdio.h>

#include <vector>

#include "sp_internal.h"

namespace {

constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr int kGLQ = 16;          // Gauss-Legendre points per panel
constexpr double kFullLine = 40.0; // a L^2 at or above which the full-line forms are used

// ------------------------------------------------------------------------- K4
// tau_s = tau_lo + s h, a_s = exp(2 tau_s), w_s = (1/(8 pi)) (2/sqrt(pi)) h exp(tau_s):
// the trapezoidal rule for 1/(8 pi r) = (1/(8 pi)) (2/sqrt(pi)) int exp(tau - r^2 e^{2tau}) dtau.
__global__ void k_gs_table(double tau_lo, double h, int terms, double* w, double* a)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= terms) return;
    double tau = tau_lo + s * h;
    a[s] = exp(2.0 * tau);
    w[s] = (1.0 / (4.0 * kPi * sqrt(kPi))) * h * exp(tau);
}

// ------------------------------------------------------------------------- K5
// Gauss-Legendre nodes and weights of 16 points on [-1, 1], the positive half in descending
// order: the roots of P_16 and 2 (1 - x^2)/(16 P_15(x))^2, evaluated to 50 digits and rounded
// (Newton's method in FP64 left 3e-16 on the weights' sum, a common factor of G and H).
__constant__ double kGlX[kGLQ / 2] = {0.9894009349916499326, 0.94457502307323257608, 0.86563120238783174388, 0.7554044083550030339,
                                      0.61787624440264374845, 0.45801677765722738634, 0.28160355077925891323, 0.095012509837637440185};
__constant__ double kGlW[kGLQ / 2] = {0.027152459411754094852, 0.062253523938647892863, 0.09515851168249278481, 0.12462897125553387205,
                                      0.14959598881657673208, 0.16915651939500253819, 0.18260341504492358887, 0.18945061045506849629};

// Quadrature nodes of the composite rule: P panels of Q points on [0, L].
// t[j] = (panel + (1 + x_i)/2) position in units of the panel width, wq[j] = weight.
__global__ void k_nodes(int P, double L, double* tpos, double* y, double* wq)
{
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= P * kGLQ) return;
    int panel = j / kGLQ, i = j % kGLQ;
    const int h = i < kGLQ / 2 ? i : kGLQ - 1 - i;
    double t = 0.5 * (1.0 + (i < kGLQ / 2 ? kGlX[h] : -kGlX[h]));
    tpos[j] = t;
    y[j] = L * (panel + t) / P;
    wq[j] = 0.5 * (L / P) * kGlW[h];
}

// Quadrature weights times the integrands, per GS row s and node j:
//   E0 = wq f,  E2 = wq g,  F0 = wq f'''',  F2 = wq g''''
// with f = exp(-a y^2), g = y^2 exp(-a y^2) and their fourth derivatives
//   f'''' = (16a^4y^4 - 48a^3y^2 + 12a^2) f,  g'''' = (16a^4y^6 - 112a^3y^4 + 156a^2y^2 - 24a) f.
__global__ void k_gauss_rows(int rows, int nq, const double* a, const double* y,
                             const double* wq, double* E0, double* E2, double* F0, double* F2)
{
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)rows * nq) return;
    int s = (int)(idx / nq), j = (int)(idx % nq);
    double al = a[s], a2 = al * al, a3 = a2 * al, a4 = a3 * al;
    double yy = y[j] * y[j];
    double e = wq[j] * exp(-al * yy);
    E0[idx] = e;
    E2[idx] = e * yy;
    F0[idx] = (16.0 * a4 * yy * yy - 48.0 * a3 * yy + 12.0 * a2) * e;
    F2[idx] = (16.0 * a4 * yy * yy * yy - 112.0 * a3 * yy * yy + 156.0 * a2 * yy - 24.0 * al) * e;
}

// C[k][j] = cos(pi k y_j / L) = cos(pi ((k panel mod 2P) + k t_j) / P): the integer part
// of the phase is reduced exactly before the floating-point product.
__global__ void k_cos_rows(int nk, int P, int Q, const double* tpos, double* C)
{
    long long nq = (long long)P * Q;
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nk * nq) return;
    int k = (int)(idx / nq);
    int j = (int)(idx % nq);
    int panel = j / Q;
    long long red = ((long long)k * panel) % (2LL * P);
    C[idx] = cospi(((double)red + (double)k * tpos[j]) / (double)P);
}

// Rows with a_s L^2 >= kFullLine: the window cut is below exp(-40) relative, and the
// full-line transforms hold:  G = sqrt(pi/a) e^{-kappa^2/4a},
// H = sqrt(pi)/(2 a^{3/2}) (1 - kappa^2/(2a)) e^{-kappa^2/4a}.
__global__ void k_full_line(int s0, int terms, int nk, double L, const double* a, double* G,
                            double* H)
{
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long rows = terms - s0;
    if (idx >= rows * nk) return;
    int s = s0 + (int)(idx / nk), k = (int)(idx % nk);
    double al = a[s];
    double kap = kPi * k / L;
    double q = kap * kap / (4.0 * al);
    double ex = exp(-q);
    G[(long long)s * nk + k] = sqrt(kPi / al) * ex;
    H[(long long)s * nk + k] = sqrt(kPi) / (2.0 * al * sqrt(al)) * (1.0 - 2.0 * q) * ex;
}

// ------------------------------------------------------------------------- GEMM
// C[m][n] = sum_k A[m][k] B[n][k] (both operands K-contiguous), FP64, 16 x 16 tiles, 64
// threads with 2 x 2 outputs each, K staged through shared memory 16 at a time.  Bound by the
// FP64 pipe (two FMAs a clock an SM), so small tiles cost nothing in shared-memory reads,
// compute less that nobody needs and spread evenly over the SMs.  Column tiles are aligned
// to the last column: n + 1 of them are one more than a multiple of 16 at the usual sizes, and
// the tile that is nearly empty is then the one at column 0, which the symmetric contraction
// needs least.  Multiplier of a 128^3 grid (129 columns): 32 x 32 tiles from column 0 computed
// 2.09 times the entries it needs (1616 us), 32 x 16 from the last 1.19 times (1083 us, 5.6
// tiles an SM), these 1.18 times (955 us).  Row tiles are blockIdx.x (there are up to 65664):
// blocks of one column tile run together, and the skipped ones of the low columns last (columns
// fastest: precompute 1.58 ms instead of 1.40).  The epilogue functor receives (m, n, value);
// skip(m0, n0) names tiles that are not needed.
constexpr int TM = 16, TN = 16, TK = 16, kGemmThreads = 64;

template <class Epi>
__global__ void __launch_bounds__(kGemmThreads) k_dgemm_nt(int M, int N, int K, const double* __restrict__ A,
                                                           long long lda, const double* __restrict__ B,
                                                           long long ldb, Epi epi)
{
    __shared__ double As[TK][TM + 1];
    __shared__ double Bs[TK][TN + 1];
    const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;
    const int m0 = blockIdx.x * TM, n0 = N - TN * ((int)blockIdx.y + 1);  // n0 < 0: partly empty
    if (epi.skip(m0, n0)) return;
    double acc[2][2] = {};
    for (int k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
        for (int l = threadIdx.x; l < TM * TK; l += kGemmThreads) {
            const int r = l / TK, c = l % TK;
            As[c][r] = (m0 + r < M && k0 + c < K) ? A[(long long)(m0 + r) * lda + k0 + c] : 0.0;
        }
#pragma unroll
        for (int l = threadIdx.x; l < TN * TK; l += kGemmThreads) {
            const int r = l / TK, c = l % TK;
            Bs[c][r] = (n0 + r >= 0 && k0 + c < K) ? B[(long long)(n0 + r) * ldb + k0 + c] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < TK; ++c) {
            const double a0 = As[c][ty], a1 = As[c][ty + 8], b0 = Bs[c][tx], b1 = Bs[c][tx + 8];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int gm = m0 + ty + 8 * i, gn = n0 + tx + 8 * j;
            if (gm < M && gn >= 0) epi(gm, gn, acc[i][j]);
        }
}

// The 1D integrals are taken in one of two exact forms per (s, k):
//  direct  (k = 0 or kappa^2 < 4 a_s):  I = int_0^L P(y) cos(kappa y) dy
//  by parts (otherwise): with kappa L = pi k and P even (P'(0) = P'''(0) = 0),
//     I = (-1)^k [P'(L)/kappa^2 - P'''(L)/kappa^4] + (1/kappa^4) int_0^L P''''(y) cos(kappa y) dy,
// which keeps the boundary terms exact where I is small next to the size of P, so that
// G and H have relative (not only absolute) accuracy at high wavenumber.
__device__ __forceinline__ bool by_parts(int k, double kap, double al) { return k > 0 && kap * kap >= 4.0 * al; }

// boundary terms of the by-parts form: 2 (-1)^k (P'(L)/kappa^2 - P'''(L)/kappa^4), plus 2 v / kappa^4
// WHICH 0: P = f = exp(-a y^2); 1: P = g = y^2 exp(-a y^2)
__device__ __forceinline__ double parts_value(int which, int k, double kap, double al, double L, double v)
{
    const double e = exp(-al * L * L), a2 = al * al, a3 = a2 * al, L2 = L * L;
    double d1, d3;
    if (which == 0) {
        d1 = -2.0 * al * L * e;
        d3 = (-8.0 * a3 * L2 * L + 12.0 * a2 * L) * e;
    } else {
        d1 = (2.0 * L - 2.0 * al * L2 * L) * e;
        d3 = (-24.0 * al * L + 36.0 * a2 * L2 * L - 8.0 * a3 * L2 * L2 * L) * e;
    }
    const double sgn = (k & 1) ? -1.0 : 1.0, k2 = kap * kap, k4 = k2 * k2;
    return 2.0 * (sgn * (d1 / k2 - d3 / k4) + v / k4);
}

// The quadrature sums of one axis, all four (direct and by-parts integrands of G and H) in
// one launch: 16 x 8 outputs (s, k) a block, blockIdx.z = 0 for G, 1 for H.  A block runs
// the direct sum, the by-parts sum, or (where the border between them crosses it) both.
// Bound by the FP64 pipe at two FMAs a clock an SM, so the tile is small: it fills the chip
// (918 blocks at n = 128, where 64 x 64 tiles gave 21) and few blocks run both sums, and
// two shared-memory reads an FMA do not show.
constexpr int kAxS = 16, kAxC = 8, kAxK = 32;
__global__ void __launch_bounds__(kAxS * kAxC) k_axis_sums(int rows, int nk, int nq, const double* __restrict__ E,
                                                           const double* __restrict__ C, const double* __restrict__ a, double L,
                                                           double* __restrict__ G, double* __restrict__ H)
{
    __shared__ double As[kAxS][kAxK + 1], Bs[kAxC][kAxK + 1];
    const int which = blockIdx.z, tx = threadIdx.x % kAxC, ty = threadIdx.x / kAxC;
    const int s = blockIdx.y * kAxS + ty, k = blockIdx.x * kAxC + tx;
    const bool in = s < rows && k < nk;
    const double al = in ? a[s] : 1.0, kap = kPi * k / L;
    const bool parts = in && by_parts(k, kap, al);
    const long long rn = (long long)rows * nq;
    for (int form = 0; form < 2; ++form) {  // 0: direct (E0, E2), 1: by parts (F0, F2)
        if (!__syncthreads_or(in && parts == (form == 1))) continue;
        const double* A = E + (2 * form + which) * rn;
        double acc = 0.0;
        for (int q0 = 0; q0 < nq; q0 += kAxK) {
            for (int l = threadIdx.x; l < (kAxS + kAxC) * kAxK; l += kAxS * kAxC) {
                const int r = l / kAxK, c = l % kAxK, q = q0 + c;
                const int gs = blockIdx.y * kAxS + r, gk = blockIdx.x * kAxC + r - kAxS;
                if (r < kAxS) As[r][c] = gs < rows && q < nq ? A[(long long)gs * nq + q] : 0.0;
                else Bs[r - kAxS][c] = gk < nk && q < nq ? C[(long long)gk * nq + q] : 0.0;
            }
            __syncthreads();
            double part = 0.0;  // summed by steps: the rounding of nq terms in a row stays below the rule's
#pragma unroll 8
            for (int c = 0; c < kAxK; ++c) part = fma(As[ty][c], Bs[tx][c], part);
            acc += part;
            __syncthreads();
        }
        if (in && parts == (form == 1)) {
            double* out = which ? H : G;
            out[(long long)s * nk + k] = form ? parts_value(which, k, kap, al, L, acc) : 2.0 * acc;
        }
    }
}

// ------------------------------------------------------------------------- K6
// Rows of the multiplier's contraction: every (k1, k0), or with SYM (axes 0 and 1 share n
// and L, so V is symmetric in them) those with k0 <= k1, numbered k1 (k1 + 1)/2 + k0.
__device__ __forceinline__ void mult_row(int row, int n0p, int sym, int& k0, int& k1)
{
    if (!sym) {
        k1 = row / n0p;
        k0 = row % n0p;
        return;
    }
    k1 = (int)((sqrtf(8.0f * row + 1.0f) - 1.0f) * 0.5f);  // within one: corrected below
    while (k1 * (k1 + 1) / 2 > row) --k1;
    while ((k1 + 1) * (k1 + 2) / 2 <= row) ++k1;
    k0 = row - k1 * (k1 + 1) / 2;
}

// Tables of one axis with the contraction index fastest: B[k][c], c < S: G[c][k], S <= c <
// 2S: H[c - S][k].  The third axis's is the right-hand operand of the contraction, the other
// two are read by the rows of the left-hand one.
__global__ void k_mult_rhs(int S, int nk, const double* G, const double* H, double* B)
{
    const int k = blockIdx.y, c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < 2 * S) B[(long long)k * 2 * S + c] = c < S ? G[(long long)c * nk + k] : H[(long long)(c - S) * nk + k];
}

// A'[row][c], rows [row0, row0 + gridDim.y) (mult_row), from the axes' B tables:
//   c <  S: w_c (H0[c][k0] G1[c][k1] + G0[c][k0] H1[c][k1])
//   c >= S: w_{c-S} G0[c-S][k0] G1[c-S][k1]
__global__ void k_mult_lhs(int row0, int S, int n0p, int sym, const double* w, const double* B0, const double* B1, double* Ap)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= 2 * S) return;
    int k0, k1;
    mult_row(row0 + blockIdx.y, n0p, sym, k0, k1);
    const double *b0 = B0 + (long long)k0 * 2 * S, *b1 = B1 + (long long)k1 * 2 * S;
    const int s = c < S ? c : c - S;
    const double g0 = b0[s], g1 = b1[s];
    Ap[(long long)blockIdx.y * 2 * S + c] = c < S ? w[s] * (b0[S + s] * g1 + g0 * b1[S + s]) : w[s] * (g0 * g1);
}

// Original GS method without near-field correction: A'[row][s] = 2 w_s G0 G1 (the GS of
// 1/(4 pi r) is twice the 1/(8 pi r) table), contracted with the G half of the third axis's
// table: V = sum_s 2 w_s G0 G1 G2.
__global__ void k_plain_lhs(int row0, int S, int n0p, int sym, const double* w, const double* B0, const double* B1, double* Ap)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    int k0, k1;
    mult_row(row0 + blockIdx.y, n0p, sym, k0, k1);
    Ap[(long long)blockIdx.y * S + s] = 2.0 * w[s] * B0[(long long)k0 * 2 * S + s] * B1[(long long)k1 * 2 * S + s];
}

struct EpiMultiplier {  // M[k1][k0][kz] = -(kappa0^2 + kappa1^2 + kappa2^2) V / Ntilde (or V / Ntilde)
    double* M;
    int ldz, row0, n0p;
    int sym, cube;      // symmetric in axes 0, 1; in all three (only kz >= k1 >= k0 is needed)
    double c0, c1, c2;  // (pi / L_p)^2
    double invN;
    int laplacian;      // 1: super-potential (spectral Laplacian applied); 0: plain GS kernel
    // a tile is needed when its last column reaches its first row's k1 (the rows' smallest)
    __device__ bool skip(int m0, int n0) const
    {
        if (!cube) return false;
        int k0, k1;
        mult_row(row0 + m0, n0p, sym, k0, k1);
        return n0 + TN - 1 < k1;
    }
    __device__ void operator()(int m, int n, double v) const
    {
        int k0, k1;
        mult_row(row0 + m, n0p, sym, k0, k1);
        const double k2sum = c0 * (double)k0 * k0 + c1 * (double)k1 * k1 + c2 * (double)n * n;
        const double x = laplacian ? -k2sum * v * invN : v * invN;
        M[((long long)k1 * n0p + k0) * ldz + n] = x;
        if (sym) M[((long long)k0 * n0p + k1) * ldz + n] = x;
    }
};

// The entries of a cube's multiplier with kz below max(k0, k1), from the sorted triple.
__global__ void k_cube_fill(int np, int ldz, double* M)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)np * np * np) return;
    const int kz = (int)(idx % np), k0 = (int)(idx / np % np), k1 = (int)(idx / ((long long)np * np));
    const int hi = k0 > k1 ? k0 : k1, lo = k0 > k1 ? k1 : k0;
    if (kz >= hi) return;
    // sorted: smallest and middle as (k0, k1), hi as the column
    const int a = kz < lo ? kz : lo, b = kz < lo ? lo : kz;
    M[((long long)k1 * np + k0) * ldz + kz] = M[((long long)b * np + a) * ldz + hi];
}

__global__ void k_to_f32(long long count, const double* in, float* out)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = (float)in[i];
}

__global__ void k_to_df(long long count, const double* in, df32* out)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = df_from_double(in[i]);
}

// ------------------------------------------------------------------------- K7
__global__ void k_twiddles(int N, cpx<double>* tw64, cpx<float>* tw32, cpx<df32>* twdf)
{
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    double s, c;
    sincospi(2.0 * (double)j / (double)N, &s, &c);
    if (tw64) tw64[j] = mk(c, -s);
    if (tw32) tw32[j] = mk((float)c, (float)-s);
    if (twdf) twdf[j] = mk(df_from_double(c), df_from_double(-s));
}

// ------------------------------------------------------------------------- period F
// Rows of the change of period of one axis (sp_embed.cuh): the multiplier of period F from
// the one of period N = 2n, through the kernel values it stands for,
//   K_j = sum_{k=0}^{N-1} M_k cos(2 pi jk/N),   M'_q = (1/F) sum_{|j| <= n-1} K_j cos(2 pi jq/F),
// folded over |k|: T[q][k] = (1/F) c_k sum_{|j| <= n-1} cos(2 pi jk/N) cos(2 pi jq/F), c_0 =
// c_n = 1, else 2.  The sum is half of D(b) + D(b') with b, b' = 2 pi (q/F -+ k/N) and the
// Dirichlet kernel D(b) = sin((n - 1/2) b) / sin(b/2) = sum_{|j| <= n-1} cos(jb); with
// b/2 = pi m / (N F), m = q N -+ k F, both phases are reduced as integers.
__device__ __forceinline__ double dirichlet(long long m, long long NF, int n)
{
    // D has period NF in m (both sines change sign); the phases are folded to at most pi/2, so
    // that neither sine is taken near a multiple of pi of a rounded argument
    long long r = m % NF;
    if (2 * r > NF) r -= NF;
    if (2 * r < -NF) r += NF;
    if (r == 0) return (double)(2 * n - 1);
    long long s = (2 * n - 1) * r % (2 * NF);
    if (s > NF) s -= 2 * NF;
    if (s < -NF) s += 2 * NF;
    if (2 * s > NF) s = NF - s;
    if (2 * s < -NF) s = -NF - s;
    return sinpi((double)s / (double)NF) / sinpi((double)r / (double)NF);
}
__global__ void k_period_rows(int n, int F, double* T)
{
    const int nk = n + 1, nq = F / 2 + 1;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nk * nq) return;
    const int q = idx / nk, k = idx % nk;
    const long long N = 2 * n, NF = N * F;
    const double d = dirichlet(q * N - (long long)k * F, NF, n) + dirichlet(q * N + (long long)k * F, NF, n);
    T[idx] = (k == 0 || k == n ? 0.5 : 1.0) * d / (double)F;
}

// C[b][m][j] = sum_k A[m][k] B[b][k][j]: the change of period along a strided axis (FP64).
// B's rows have stride ldb, its batches sb; C's likewise.  Bound by the FP64 pipe; 16 x 16 tiles
// (64 threads, 2 x 2 outputs each) keep the waste at the edges small (F/2 + 1 rows are one more
// than a multiple of 16 at most lengths) and give an 83^3 grid 2400 blocks a launch, where
// 64 x 64 tiles gave 168 to 194, one to two an SM.
constexpr int kNnT = 16;
__global__ void __launch_bounds__(64) k_dgemm_nn(int M, int N, int K, const double* __restrict__ A,
                                                 const double* __restrict__ B, long long ldb, long long sb,
                                                 double* __restrict__ C, long long ldc, long long sc)
{
    __shared__ double As[kNnT][kNnT + 1];
    __shared__ double Bs[kNnT][kNnT];
    const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;
    const int m0 = blockIdx.y * kNnT, n0 = blockIdx.x * kNnT;
    B += blockIdx.z * sb;
    C += blockIdx.z * sc;
    double acc[2][2] = {};
    for (int k0 = 0; k0 < K; k0 += kNnT) {
#pragma unroll
        for (int l = threadIdx.x; l < kNnT * kNnT; l += 64) {
            const int r = l / kNnT, c = l % kNnT;
            As[c][r] = (m0 + r < M && k0 + c < K) ? A[(long long)(m0 + r) * K + k0 + c] : 0.0;
            Bs[r][c] = (k0 + r < K && n0 + c < N) ? B[(long long)(k0 + r) * ldb + n0 + c] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < kNnT; ++c) {
            const double a0 = As[c][ty], a1 = As[c][ty + 8], b0 = Bs[c][tx], b1 = Bs[c][tx + 8];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (m0 + ty + 8 * i < M && n0 + tx + 8 * j < N)
                C[(long long)(m0 + ty + 8 * i) * ldc + n0 + tx + 8 * j] = acc[i][j];
}

struct EpiStore {
    double* C;
    long long ldc;
    __device__ bool skip(int, int) const { return false; }
    __device__ void operator()(int m, int n, double v) const { C[(long long)m * ldc + n] = v; }
};

__device__ __forceinline__ void put(double* p, double v) { *p = v; }
__device__ __forceinline__ void put(float* p, double v) { *p = (float)v; }
__device__ __forceinline__ void put(df32* p, double v) { *p = df_from_double(v); }
// Columns [c0, c0 + cols) of the period-F multiplier into the plan's table (row stride ldf).
template <class R> __global__ void k_put_columns(long long rows, int cols, const double* X, long long ldx, R* M, int c0, int ldf)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * cols) return;
    const long long r = i / cols;
    const int c = (int)(i % cols);
    put(M + r * ldf + c0 + c, X[r * ldx + c]);
}

inline unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// Scratch of one step of the precompute, freed at scope exit (stream-ordered).  Where the
// device has no memory left for it, it lies in the plan's workspace, which no solve uses
// meanwhile (solves are ordered against the precompute) and which a plan on lengths F >= 2n
// holds larger: such a plan leaves less memory free than one on 2n, and its change of period
// wants more (500 x 500 x 20, FP32: 105 MB beside a workspace of 131 MB).
struct Scratch {
    cudaStream_t st;
    unsigned char* room;
    size_t left;
    void* own[8];
    int nown = 0;
    Scratch(sp_plan p, cudaStream_t s) : st(s), room((unsigned char*)p->d_work), left(p->work_bytes) {}
    Scratch(const Scratch&) = delete;
    double* take(long long values)  // NULL: it fits neither
    {
        const size_t bytes = (sizeof(double) * (size_t)values + 255) / 256 * 256;
        void* q = nullptr;
        if (nown < 8 && cudaMallocAsync(&q, bytes, st) == cudaSuccess) return (double*)(own[nown++] = q);
        cudaGetLastError();  // allocation failures are not sticky: clear them
        if (bytes > left) return nullptr;
        q = room;
        room += bytes;
        left -= bytes;
        return (double*)q;
    }
    ~Scratch()
    {
        for (int i = 0; i < nown; ++i) cudaFreeAsync(own[i], st);
    }
};

}  // namespace

// 1D tables of one axis: G, H [S][n+1].
static sp_status setup_axis(sp_plan p, int ax, cudaStream_t st)
{
    const int n = p->n[ax], nk = n + 1, S = p->gs_terms;
    const double L = p->L[ax];
    // split between quadrature rows and full-line rows (a_s increases with s)
    const double* a = p->h_gs_a;
    int s_split = S;
    for (int s = 0; s < S; ++s)
        if (a[s] * L * L >= kFullLine) { s_split = s; break; }
    sp_status rc;
    // full-line rows
    if (s_split < S) {
        k_full_line<<<nblk((long long)(S - s_split) * nk, 256), 256, 0, st>>>(
            s_split, S, nk, L, p->d_gs_a, p->d_G[ax], p->d_H[ax]);
    }
    if (s_split > 0) {
        // panels: a panel spans a phase of at most 3 pi of cos(pi k y / L), k <= n.  The 16-point
        // rule's error is phi^33 (16!)^4 / (33 (32!)^3) of the integrand's 32nd derivative, phi
        // the phase: 5e-23 for the cosine alone, below 1e-17 with the Gaussian's own variation
        // over a panel (a L^2 < 40: at most 4.2 more of phase at n = 33)
        const int P = n > 32 ? (n + 2) / 3 : (n > 8 ? n : 8), Q = kGLQ;
        const long long nq = (long long)P * Q;
        const long long rn = (long long)s_split * nq;
        Scratch scratch(p, st);
        double *tpos = scratch.take(3 * nq), *E0 = scratch.take(4 * rn), *C = scratch.take(nk * nq);
        if (!tpos || !E0 || !C) return sp_fail(SP_ERR_OOM, "setup: quadrature scratch allocation failed");
        double *y = tpos + nq, *wq = tpos + 2 * nq, *E2 = E0 + rn, *F0 = E2 + rn, *F2 = F0 + rn;
        k_nodes<<<nblk(nq, 256), 256, 0, st>>>(P, L, tpos, y, wq);
        k_gauss_rows<<<nblk(rn, 256), 256, 0, st>>>(s_split, (int)nq, p->d_gs_a, y, wq, E0, E2, F0, F2);
        k_cos_rows<<<nblk(nk * nq, 256), 256, 0, st>>>(nk, P, Q, tpos, C);
        dim3 grid(nblk(nk, kAxC), nblk(s_split, kAxS), 2);
        k_axis_sums<<<grid, kAxS * kAxC, 0, st>>>(s_split, nk, (int)nq, E0, C, p->d_gs_a, L, p->d_G[ax], p->d_H[ax]);
        rc = sp_cuda_check(cudaGetLastError(), "setup: 1D integral kernels");
        if (rc) return rc;
    }
    return sp_cuda_check(cudaGetLastError(), "setup: full-line kernel");
}

// GS table of eq. (sin_1_x) for the plan's (eps, delta): tau_s = tau_lo + s h_tau for
// s = 0..terms-1 (reading of the paper's sinc quadrature, see k_gs_table).
static void gs_range(const sp_plan p, double* tau_lo, int* terms)
{
    *tau_lo = log(p->eta * sqrt(kPi) / (2.0 * p->delta));
    const double tau_hi = log(sqrt(log(1.0 / p->eta)) / p->eps) + 0.5;
    *terms = (int)ceil((tau_hi - *tau_lo) / p->h_tau) + 1;
}

int sp_gs_terms(const sp_plan p)
{
    double tau_lo;
    int terms;
    gs_range(p, &tau_lo, &terms);
    return terms;
}

void sp_gs_exponents(const sp_plan p, double* a)
{
    double tau_lo;
    int terms;
    gs_range(p, &tau_lo, &terms);
    for (int s = 0; s < terms; ++s) a[s] = exp(2.0 * (tau_lo + s * p->h_tau));
}

// Multiplier of the solve passes' lengths F from the 2n one (both FP64, rounded to the pass
// type last): one contraction per axis whose length changes, up to 64 output columns at a time
// so that the scratch stays at two slabs of (F0/2 + 1)(F1/2 + 1) x 64, fewer where it is short.
static sp_status setup_period(sp_plan p, cudaStream_t st)
{
    const int n0p = p->n[0] + 1, n1p = p->n[1] + 1, n2p = p->n[2] + 1;
    const int q0 = p->F[0] / 2 + 1, q1 = p->F[1] / 2 + 1, q2 = p->F[2] / 2 + 1;
    Scratch scratch(p, st);
    double* T[3] = {};
    for (int ax = 0; ax < 3; ++ax) {
        if (p->F[ax] == p->N[ax]) continue;
        const long long cnt = (long long)(p->n[ax] + 1) * (p->F[ax] / 2 + 1);
        if (!(T[ax] = scratch.take(cnt))) return sp_fail(SP_ERR_OOM, "setup: period scratch allocation failed");
        k_period_rows<<<nblk(cnt, 256), 256, 0, st>>>(p->n[ax], p->F[ax], T[ax]);
    }
    const long long column = (long long)(q0 > n0p ? q0 : n0p) * (q1 > n1p ? q1 : n1p);
    int CW = q2 < 64 ? q2 : 64;
    double* X;
    while (!(X = scratch.take(2 * CW * column))) {
        if (CW == 1) return sp_fail(SP_ERR_OOM, "setup: period scratch allocation failed");
        CW = CW >= 32 ? CW / 2 / 16 * 16 : CW / 2;  // whole tiles while there are any
    }
    double* Y = X + CW * column;
    for (int c0 = 0; c0 < q2; c0 += CW) {
        const int cols = q2 - c0 < CW ? q2 - c0 : CW;
        const double* cur = p->d_M64 + c0;  // [n1p][n0p][cols], row stride ld
        long long ld = p->ldz;
        double* next = X;
        if (T[2]) {
            dim3 grid(nblk((long long)n0p * n1p, TM), nblk(cols, TN));
            k_dgemm_nt<<<grid, kGemmThreads, 0, st>>>(n0p * n1p, cols, n2p, p->d_M64, (long long)p->ldz,
                                             T[2] + (long long)c0 * n2p, (long long)n2p, EpiStore{next, CW});
            cur = next;
            ld = CW;
            next = Y;
        }
        if (T[0]) {
            dim3 grid(nblk(cols, kNnT), nblk(q0, kNnT), n1p);
            k_dgemm_nn<<<grid, 64, 0, st>>>(q0, cols, n0p, T[0], cur, ld, ld * n0p, next, CW, (long long)CW * q0);
            cur = next;
            ld = CW;
            next = cur == X ? Y : X;
        }
        if (T[1]) {  // rows (k0', column) of one k1 are contiguous, or ld apart without an earlier step
            const long long w = (long long)q0 * ld;
            if (ld == CW) {
                dim3 grid(nblk(w, kNnT), nblk(q1, kNnT));
                k_dgemm_nn<<<grid, 64, 0, st>>>(q1, (int)w, n1p, T[1], cur, w, 0, next, w, 0);
            } else {
                dim3 grid(nblk(cols, kNnT), nblk(q1, kNnT), q0);  // one k0 at a time: batch stride ld
                k_dgemm_nn<<<grid, 64, 0, st>>>(q1, cols, n1p, T[1], cur, w, ld, next, (long long)CW * q0, CW);
                ld = CW;
            }
            cur = next;
        }
        const long long rows = (long long)q0 * q1;
        const unsigned nb = nblk(rows * cols, 256);
        if (p->prec == SP_FP64) k_put_columns<<<nb, 256, 0, st>>>(rows, cols, cur, ld, (double*)p->d_Ms, c0, p->ldf);
        else if (p->prec == SP_DF32) k_put_columns<<<nb, 256, 0, st>>>(rows, cols, cur, ld, (df32*)p->d_Ms, c0, p->ldf);
        else k_put_columns<<<nb, 256, 0, st>>>(rows, cols, cur, ld, (float*)p->d_Ms, c0, p->ldf);
    }
    return sp_cuda_check(cudaGetLastError(), "setup: change of period");
}

sp_status sp_setup_run(sp_plan p, cudaStream_t st)
{
    sp_status rc;
    // K4: GS table (unless the caller supplied one at plan creation)
    if (!p->gs_user) {
        double tau_lo;
        int terms;
        gs_range(p, &tau_lo, &terms);
        if (terms != p->gs_terms) return sp_fail(SP_ERR_INVALID, "internal: GS table length changed");
        k_gs_table<<<nblk(terms, 128), 128, 0, st>>>(tau_lo, p->h_tau, terms, p->d_gs_w, p->d_gs_a);
        if ((rc = sp_cuda_check(cudaGetLastError(), "GS table kernel"))) return rc;
    }
    // per-axis tables (allocated with the plan; axes with the same (n, L) share one)
    for (int ax = 0; ax < 3; ++ax) {
        bool shared = false;
        for (int q = 0; q < ax; ++q)
            if (p->d_G[q] == p->d_G[ax]) shared = true;
        if (shared) continue;
        if ((rc = setup_axis(p, ax, st))) return rc;
    }
    const int S = p->gs_terms;
    // K6: multiplier, GEMM over the 2S GS columns, in row chunks
    {
        const int n0p = p->n[0] + 1, n1p = p->n[1] + 1, n2p = p->n[2] + 1;
        // axes that share n and L make V symmetric in their wavenumbers: half of the rows where
        // axes 0 and 1 do, and of those about a third of the columns where all three do (the
        // rest is copied).  128^3: 2.2e6 of 16641 x 129 values are contracted three times less.
        const bool sym = p->n[0] == p->n[1] && p->L[0] == p->L[1];
        const bool cube = sym && p->n[1] == p->n[2] && p->L[1] == p->L[2];
        const long long rows_total = sym ? (long long)n0p * (n0p + 1) / 2 : (long long)n0p * n1p;
        // rows at a time: the left-hand operand of a chunk (up to 140 MB) is made just before it
        // is read; fewer, larger chunks leave fewer partly filled last waves
        const bool plain = p->kernel == SP_KERNEL_GS_PLAIN;
        const int K = plain ? S : 2 * S;  // contraction length (GS columns)
        long long most = (140LL << 20) / (8LL * K);
        most = most < 256 ? 256 : (most > 16384 ? 16384 : most);
        Scratch scratch(p, st);
        double* bt[3];
        for (int ax = 0; ax < 3; ++ax) {
            int same = ax;
            for (int q = ax - 1; q >= 0; --q)
                if (p->d_G[q] == p->d_G[ax]) same = q;
            if (same < ax) {
                bt[ax] = bt[same];
                continue;
            }
            const int nk = p->n[ax] + 1;
            if (!(bt[ax] = scratch.take((long long)nk * 2 * S))) return sp_fail(SP_ERR_OOM, "setup: multiplier scratch allocation failed");
            k_mult_rhs<<<dim3(nblk(2 * S, 256), nk), 256, 0, st>>>(S, nk, p->d_G[ax], p->d_H[ax], bt[ax]);
        }
        int chunk;
        double* Ap;
        for (;; most /= 2) {  // halved while it does not fit
            const int chunks = (int)((rows_total + most - 1) / most);
            chunk = (int)((rows_total + chunks - 1) / chunks);
            if ((Ap = scratch.take((long long)chunk * K))) break;
            if (most <= 16) return sp_fail(SP_ERR_OOM, "setup: multiplier scratch allocation failed");
        }
        EpiMultiplier epi;
        epi.M = p->d_M64;
        epi.ldz = p->ldz;
        epi.n0p = n0p;
        epi.c0 = (kPi / p->L[0]) * (kPi / p->L[0]);
        epi.c1 = (kPi / p->L[1]) * (kPi / p->L[1]);
        epi.c2 = (kPi / p->L[2]) * (kPi / p->L[2]);
        epi.invN = 1.0 / (8.0 * (double)p->n[0] * (double)p->n[1] * (double)p->n[2]);
        epi.laplacian = plain ? 0 : 1;
        epi.sym = sym;
        epi.cube = cube;
        for (long long r0 = 0; r0 < rows_total; r0 += chunk) {
            int rows = (int)((rows_total - r0) < chunk ? (rows_total - r0) : chunk);
            if (plain)
                k_plain_lhs<<<dim3(nblk(S, 256), rows), 256, 0, st>>>((int)r0, S, n0p, sym, p->d_gs_w, bt[0], bt[1], Ap);
            else
                k_mult_lhs<<<dim3(nblk(2 * S, 256), rows), 256, 0, st>>>((int)r0, S, n0p, sym, p->d_gs_w, bt[0], bt[1], Ap);
            epi.row0 = (int)r0;
            dim3 grid(nblk(rows, TM), nblk(n2p, TN));
            k_dgemm_nt<<<grid, kGemmThreads, 0, st>>>(rows, n2p, K, Ap, K, bt[2], 2 * S, epi);
        }
        if (cube) k_cube_fill<<<nblk((long long)n0p * n0p * n0p, 256), 256, 0, st>>>(n0p, p->ldz, p->d_M64);
        const long long mcount = (long long)n0p * n1p * p->ldz;
        if (p->d_M32) k_to_f32<<<nblk(mcount, 256), 256, 0, st>>>(mcount, p->d_M64, p->d_M32);
        if (p->d_Mdf) k_to_df<<<nblk(mcount, 256), 256, 0, st>>>(mcount, p->d_M64, p->d_Mdf);
        if ((rc = sp_cuda_check(cudaGetLastError(), "multiplier kernels"))) return rc;
    }
    // K7: twiddles
    for (int ax = 0; ax < 3; ++ax) {
        k_twiddles<<<nblk(p->N[ax], 256), 256, 0, st>>>(p->N[ax], p->d_tw64[ax], p->d_tw32[ax], p->d_twdf[ax]);
    }
    if (p->emb) {
        for (int ax = 0; ax < 3; ++ax) {
            if (!p->d_twF[ax]) continue;
            k_twiddles<<<nblk(p->F[ax], 256), 256, 0, st>>>(
                p->F[ax], p->prec == SP_FP64 ? (cpx<double>*)p->d_twF[ax] : nullptr,
                p->prec == SP_FP32 || p->prec == SP_MIXED ? (cpx<float>*)p->d_twF[ax] : nullptr,
                p->prec == SP_DF32 ? (cpx<df32>*)p->d_twF[ax] : nullptr);
        }
        if ((rc = setup_period(p, st))) return rc;
        rc = p->prec == SP_FP64 ? sp_embed_twiddles_f64(p, st)
             : p->prec == SP_DF32 ? sp_embed_twiddles_df(p, st) : sp_embed_twiddles_f32(p, st);
        if (rc) return rc;
    }
    if ((rc = sp_cuda_check(cudaGetLastError(), "twiddle kernel"))) return rc;
    if (p->prec == SP_DF32) return sp_v2_stage_twiddles_df(p, st);
    if (p->prec == SP_FP32 || p->prec == SP_MIXED) return sp_v2_stage_twiddles_f32(p, st);
    return SP_OK;
}
