// Low-memory ARPC (Appendix A, closing paragraph; Remark of Section 4.2), FP64:
// rpchol_factor_lowmem, bistoch_normalize_lowmem and the lift of
// eig_topk_lowmem.
//
// Only the accepted pivots S and W = F(S,:) (rank x rank, lower triangular:
// the Cholesky factor of K(S,S)) are kept.  Every row of F is
// F(i,:) = K(i,S) W^-T, so no N x r array exists: the N-long passes work on a
// row panel of P rows (P x r doubles, at most 128 MiB) of kernel values
// K(panel, S) = exp(-(|x_i|^2 + |x_s|^2 - 2 x_i.x_s) / eps), formed by a DGEMM
// of the panel's rows of X against X(S,:) and an exp kernel.
//
// rpchol_factor_lowmem, one round of Algorithm 2 with k pivots so far:
//   a2  proposals from rho (the FP64 path's kernel);
//   a3  F(S',:) = K(S',S) W^-T (b x k kernel block, then a triangular solve),
//       H = K(S',S') - F(S',:) F(S',:)^T (the FP64 path's kernel);
//   a4  Algorithm 3 (the FP64 path's kernel): accepted T, L = chol(H(T,T));
//   W   gains the rows [F(T,:) | L]; Z = W^-T F(T,:)^T (k x m);
//   a5  per panel R = K(p,T) - K(p,S) Z (= K(p,T) - F(p,:) F(T,:)^T),
//       G = R L^-T, rho -= rownorms(G)^2 clamped at 0, tile statistics.
// The host reads (k, m) once per round to size the library calls.
//
// bistoch_normalize_lowmem, three passes over the panels:
//   1  s_K = K(S,:) 1                       y = W^-T W^-1 s_K  (so F s = K(:,S) y)
//   2  d~ = K(:,S) y,  t_K = K(S,:) d~^-1   z = W^-T W^-1 t_K
//   3  q~ = K(:,S) z;  F_p = K(p,S) W^-T;  A += F_p^T D~^-2 F_p,
//      C += F_p^T Q~^-1 F_p (the normalisation's Gram kernels, accumulated: tensor cores,
//      or the FP64 pipe in a workspace without room for the digit planes).
// The vectors come from K(:,S) times a solved vector, which agrees with the
// rebuilt-F definition to ~1e-14 even at cond(W) ~ 3e5.  The Grams use the
// rebuilt F_p: W^-1 (K^T D K) W^-T loses accuracy with cond(W)^2 (2e-10 at
// cond(W) = 6e3).
//
// The lift of eig_topk_lowmem: U = D~^-1 K(:,S) (W^-T Y), per panel.
//
// The panels' dot products, the products with L^-1 and the solve with W run on the tensor
// cores from seven digit planes (ozmm.cu); K(p,S) Z, DGEMV and the small triangular solves are
// cuBLAS calls, and so are all products below the rules' lines (lm_round, carve_lm_norm)
// and under KEVD_ENGINE=fp64.  Set-up, exp, residual update, statistics and Grams are kernels
// of this library.
#include <cublas_v2.h>

#include <algorithm>
#include <climits>
#include <cstdlib>

#include "common.cuh"
#include "factor.cuh"
#include "gram_tc.cuh"
#include "lowmem.cuh"
#include "oz_digits.cuh"
#include "ozgemm.cuh"
#include "trace.cuh"

cudaError_t kevd_gram_weighted(const double* F, int64_t ldf, int64_t N, int rank, const double* wa, const double* wc,
                               double* gpart, double* A, double* C, int acc, cudaStream_t s);
size_t kevd_gram_partial_doubles(int64_t N, int k);

#define LM_BLAS(expr)                                               \
    do {                                                            \
        if ((expr) != CUBLAS_STATUS_SUCCESS) return KEVD_ECUDA;     \
    } while (0)

namespace kevd {

// cuBLAS handle per device and host thread, bound to stream s.
static cublasHandle_t lm_blas(cudaStream_t s) {
    thread_local cublasHandle_t handles[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!handles[dev] && cublasCreate(&handles[dev]) != CUBLAS_STATUS_SUCCESS) handles[dev] = nullptr;
    if (!handles[dev] || cublasSetStream(handles[dev], s) != CUBLAS_STATUS_SUCCESS) return nullptr;
    return handles[dev];
}

constexpr size_t kLmPanelDoubles = size_t(1) << 24;   // 128 MiB of kernel values per panel

// Rows per panel: a multiple of the 64-row rho tile, at most 2^24 / r (at
// least 64), and no more than N rounded up to the tile.  KEVD_LOWMEM_PANEL=rows
// in the environment lowers the 2^24 / r rule (rounded down to a multiple of
// 64, at least 64; a larger value is capped by the rule, so P r stays within
// 2^24 doubles and every panel index fits an int); workspace sizing and the
// calls must see the same setting.
static int64_t lm_panel_rows(int64_t N, int r) {
    int64_t p = (int64_t)(kLmPanelDoubles / (size_t)std::max(r, 1));
    if (const char* e = getenv("KEVD_LOWMEM_PANEL")) {
        const long long v = atoll(e);
        if (v > 0 && v < p) p = v;
    }
    p = std::max<int64_t>(p / kBM * kBM, kBM);
    return std::min<int64_t>(p, (N + kBM - 1) / kBM * kBM);
}

// A panel of kernel values and the pivot rows it is formed from.
struct LmPanel {
    double* xn;    // N: |x_i|^2
    double* XS;    // r x d row-major: X(S,:)
    double* xnS;   // r: |x_s|^2
    double* Kp;    // P x r column-major (ld P)
    int64_t P;
};

// own_xn = false: |x_i|^2 lives elsewhere (the caller sets p.xn).
static LmPanel carve_panel(Carver& c, int64_t N, int d, int r, bool own_xn = true) {
    LmPanel p;
    p.P = lm_panel_rows(N, r);
    p.xn = own_xn ? c.take<double>(N) : nullptr;
    p.XS = c.take<double>((size_t)r * d);
    p.xnS = c.take<double>(r);
    p.Kp = c.take<double>((size_t)p.P * r);
    return p;
}

// Scratch of the products on the tensor cores (seven digit planes, ozmm.cu) for `rows`
// rows of a panel at a time.  One buffer holds the left operand of each product in turn.
struct LmOz {
    uint16_t *Ap, *Bp;    // the rows' operand; columns of Z, or rows of W
    uint16_t* XSp;        // X(S,:)
    int *ae, *be, *xse;
    double* rmax;         // row maxima
    double *C, *C2;       // products
    int* flags;           // bit 2: a bounded wait gave up
    int nqx;
    int64_t rows;
};
constexpr int kLmBlock = 128;                          // columns of F solved at a time in the normalisation
constexpr int64_t kLmOzRows = 1024;                    // fewest rows worth a launch
constexpr size_t kLmScratch = (size_t)64 << 20;        // of the normalisation

// The parts that depend on the rows: aq quarters of the left operand, bn x bq quarters of the
// right one, cn columns of the product.
static void carve_lm_oz(Carver& c, LmOz& o, int64_t rows, int aq, int bn, int bq, int cn) {
    o.rows = rows;
    o.Ap = c.take<uint16_t>(oz_tile_elems(rows, aq, kDigits));
    o.Bp = c.take<uint16_t>(oz_tile_elems(bn, bq, kDigits));
    o.ae = c.take<int>(rows);
    o.be = c.take<int>(bn);
    o.rmax = c.take<double>(std::max<int64_t>(rows, bn));
    o.C = c.take<double>((size_t)rows * cn);
    o.C2 = c.take<double>((size_t)rows * cn);
}

// |x_i|^2, summed in the order of the FP64 path's set-up kernel.
__global__ void k_lm_norms(const double* __restrict__ X, int64_t N, int d, double* __restrict__ xn) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double* x = X + i * d;
    double s = 0.0;
    for (int c = 0; c < d; ++c) s = fma(x[c], x[c], s);
    xn[i] = s;
}

// XS(a,:) = X(S_a,:) and xnS(a) = |x_{S_a}|^2 for a < n.  A pivot outside
// [0, N) sets flags bit 2 and is not read.
__global__ void k_lm_gather(const double* __restrict__ X, int64_t N, int d, const int64_t* __restrict__ piv, int n,
                            const double* __restrict__ xn, double* __restrict__ XS, double* __restrict__ xnS,
                            int* __restrict__ flags) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)n * d) return;
    const int a = (int)(e / d), c = (int)(e % d);
    const int64_t p = piv[a];
    if (p < 0 || p >= N) {
        if (c == 0) atomicOr(flags, 4);
        XS[e] = 0.0;
        if (c == 0) xnS[a] = 0.0;
        return;
    }
    XS[e] = X[p * d + c];
    if (c == 0) xnS[a] = xn[p];
}

// Kernel values over the DGEMM's dot products, in place:
// Kp(i,a) = exp(-max(|x_i|^2 + |x_s|^2 - 2 Kp(i,a), 0) / eps) with i the row
// i0 + i and s = S_a (exactly 1 where the row is the pivot itself), divided by
// rowdiv(i0 + i) when rowdiv is given.
__global__ void k_lm_kexp(double* __restrict__ Kp, int64_t P, int64_t Pc, int n, int64_t i0,
                          const double* __restrict__ xn, const double* __restrict__ xnS,
                          const int64_t* __restrict__ piv, double inv_eps, const double* __restrict__ rowdiv) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= Pc * n) return;
    const int64_t i = e % Pc;
    const int a = (int)(e / Pc);
    const int64_t row = i0 + i;
    double* kp = Kp + (int64_t)a * P + i;
    double v;
    if (piv[a] == row) v = 1.0;
    else v = exp(-fmax(xn[row] + xnS[a] - 2.0 * *kp, 0.0) * inv_eps);
    if (rowdiv) v /= rowdiv[row];
    *kp = v;
}

// A -= C, a column per grid row, `rows` of the rows of both.
__global__ void k_lm_sub(double* __restrict__ A, int64_t lda, const double* __restrict__ C, int64_t ldc, int64_t rows) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < rows) A[blockIdx.y * lda + i] -= C[blockIdx.y * ldc + i];
}

// A = C + D, likewise.
__global__ void k_lm_sum(double* __restrict__ A, int64_t lda, const double* __restrict__ C,
                         const double* __restrict__ D, int64_t ldc, int64_t rows) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < rows) A[blockIdx.y * lda + i] = C[blockIdx.y * ldc + i] + D[blockIdx.y * ldc + i];
}

// The diagonal blocks of W (lower triangles), kLmBlock columns, zero elsewhere.
__global__ void k_lm_diag(const double* __restrict__ W, int64_t ldw, double* __restrict__ E, int r) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= r) return;
    const int j0 = a / kLmBlock * kLmBlock, c = blockIdx.y;
    E[(size_t)c * r + a] = j0 + c <= a ? W[(int64_t)(j0 + c) * ldw + a] : 0.0;
}

// What the seven digits of the rows of E (r x kLmBlock, exponents ex) leave out, in place: exact.
__global__ void k_lm_rest(double* __restrict__ E, int r, const int* __restrict__ ex) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= r) return;
    const double x = E[(size_t)blockIdx.y * r + a];
    const int e = ex[a];                                        // -900: no digits
    E[(size_t)blockIdx.y * r + a] = e <= -900 ? 0.0 : x - ldexp((double)oz_T_f64<kDigits>(x, e), e - 54);
}

// The unit blocks of the diagonal, kLmBlock columns: E(a, a mod kLmBlock) = 1.
__global__ void k_lm_unit(double* __restrict__ E, int r) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a < r) E[(size_t)(a % kLmBlock) * r + a] = 1.0;
}

// C(i, j) = sum_c A(i, c) B(j, c) from seven digit planes, level 7 included: without it rho's error
// against long double was 5 to 18 % above that of the FP64 library's products, and the rebuilt F's
// 1.6 to 1.8 times as large; with it 10 to 16 % below and 0.4 to 0.5 times (N = 6,000, r = 256).
static cudaError_t lm_product(const OzOperand& A, const OzOperand& B, int64_t M, int n, int K, double* C, int64_t ldc,
                              int* flags, cudaStream_t s) {
    return launch_ozmm(A, B, M, n, K, nullptr, C, ldc, 0, nullptr, 0, flags, s, kDigits, nullptr, false, true);
}

// Kp(0:Pc, 0:n) = K(i0:i0+Pc, S_0:S_n) [/ rowdiv]: one DGEMM of the panel's
// rows of X against X(S,:), then the exp kernel.
static int kernel_panel(cublasHandle_t h, const double* X, int d, int64_t i0, int64_t Pc, int n, const LmPanel& p,
                        const int64_t* piv, double inv_eps, const double* rowdiv, cudaStream_t s,
                        const LmOz* o = nullptr) {
    const double one = 1.0, zero = 0.0;
    if (o) {   // the planes of X(S,:) are the caller's
        for (int64_t r0 = 0; r0 < Pc; r0 += o->rows) {
            const int64_t rows = std::min(o->rows, Pc - r0);
            KEVD_CUDA_TRY(oz_cut_rowmajor(X + (i0 + r0) * d, rows, d, o->Ap, o->ae, s));
            KEVD_CUDA_TRY(lm_product(OzOperand{o->Ap, o->nqx, o->ae, 0}, OzOperand{o->XSp, o->nqx, o->xse, 0}, rows, n,
                                     16 * o->nqx, p.Kp + r0, p.P, o->flags, s));
        }
    } else {
        LM_BLAS(cublasDgemm(h, CUBLAS_OP_T, CUBLAS_OP_N, (int)Pc, n, d, &one, X + i0 * d, d, p.XS, d, &zero, p.Kp,
                            (int)p.P));
    }
    const int64_t tot = Pc * n;
    k_lm_kexp<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(p.Kp, p.P, Pc, n, i0, p.xn, p.xnS, piv, inv_eps, rowdiv);
    KEVD_LAUNCH_CHECK();
    return KEVD_OK;
}

// G = R M^-T for nb <= 128 columns of `rows` rows of the panel, in place, from the planes of M
// and of its explicit inverse: the product with the inverse, corrected once by its residual,
// without which the error against 64 bits was up to three times that of a triangular solve.
// The residual takes M whole, `mat` and what its digits leave out (`rest`, 2^-55 of a row's
// largest entry): that error is the same in every row of F, so the Grams' sums over the rows
// don't average it out (A's error from the solve alone, emulated for N = 2,000 and ranks 150 and
// 190: 1.35 and 1.16 times a triangular solve's without the rest, 0.77 and 0.96 times with it).
static int solve_block(const LmOz& o, double* R, int64_t P, int rows, int nb, const OzOperand& mat,
                       const OzOperand& rest, const OzOperand& inv, cudaStream_t s) {
    const int nq = (nb + 15) / 16;
    const dim3 grid((rows + 255) / 256, nb);
    const OzOperand A{o.Ap, nq, o.ae, 0};
    KEVD_CUDA_TRY(oz_cut_rows(R, P, rows, nb, nq, o.Ap, o.ae, o.rmax, s));
    KEVD_CUDA_TRY(lm_product(A, inv, rows, nb, 16 * nq, o.C, o.rows, o.flags, s));
    KEVD_CUDA_TRY(oz_cut_rows(o.C, o.rows, rows, nb, nq, o.Ap, o.ae, o.rmax, s));
    for (const OzOperand& m : {mat, rest}) {
        KEVD_CUDA_TRY(lm_product(A, m, rows, nb, 16 * nq, o.C2, o.rows, o.flags, s));
        k_lm_sub<<<grid, 256, 0, s>>>(R, P, o.C2, o.rows, rows);
    }
    KEVD_CUDA_TRY(oz_cut_rows(R, P, rows, nb, nq, o.Ap, o.ae, o.rmax, s));
    KEVD_CUDA_TRY(lm_product(A, inv, rows, nb, 16 * nq, o.C2, o.rows, o.flags, s));
    k_lm_sum<<<grid, 256, 0, s>>>(R, P, o.C, o.C2, o.rows, rows);
    KEVD_LAUNCH_CHECK();
    return KEVD_OK;
}

// ---------------------------------------------------------------------------
// Factor kernels
// ---------------------------------------------------------------------------

// X(S',:) of the proposals as a d x b panel (XSP) and their |x|^2 (xnS): the
// FP64 path's gather without the rows of F.
__global__ void k_lm_gather_prop(FactorWs w, const double* __restrict__ X, int d, int b) {
    if (w.st->done) return;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= d * b) return;
    const int j = e % b, c = e / b;
    const int64_t p = w.prop[j];
    w.XSP[(size_t)c * b + j] = X[p * d + c];
    if (c == 0) w.xnS[j] = w.xn[p];
}

// K(S', S) of the b proposals against the k pivots, column-major b x k (ld b),
// into FSP (a triangular solve with W then turns it into F(S',:)).
__global__ void k_lm_kq(FactorWs w, const double* __restrict__ XS, const double* __restrict__ xnS,
                        const int64_t* __restrict__ piv, int k, int d, int b, double inv_eps) {
    if (w.st->done) return;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= b * k) return;
    const int j = e % b, a = e / b;
    double dot = 0.0;
    for (int c = 0; c < d; ++c) dot = fma(w.XSP[(size_t)c * b + j], XS[(size_t)a * d + c], dot);
    double v;
    if (w.prop[j] == piv[a]) v = 1.0;
    else v = exp(-fmax(w.xnS[j] + xnS[a] - 2.0 * dot, 0.0) * inv_eps);
    w.FSP[(size_t)a * b + j] = v;
}

// Rows k..k+m-1 of W = [F(T,:k) | L], Zt = F(T,:k)^T (k x m, ld k), and the
// new pivots' rows of XS and entries of xnS.  One thread per (a, column).
__global__ void k_lm_extend(FactorWs w, const double* __restrict__ X, int d, int k, int m, int b,
                            const int64_t* __restrict__ piv, double* __restrict__ W, int64_t ldw,
                            double* __restrict__ XS, double* __restrict__ xnS, double* __restrict__ Zt) {
    const int width = k + m + d;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)m * width) return;
    const int a = (int)(e / width), c = (int)(e % width);
    if (c < k) {
        const double v = w.FSP[(size_t)c * b + w.acc_pos[a]];
        W[(int64_t)c * ldw + k + a] = v;
        Zt[(size_t)a * k + c] = v;
    } else if (c < k + m) {
        const int a2 = c - k;
        W[(int64_t)(k + a2) * ldw + k + a] = a2 <= a ? w.Lc[(size_t)a * b + a2] : 0.0;
    } else {
        const int cc = c - k - m;
        const int64_t p = piv[k + a];
        XS[(size_t)(k + a) * d + cc] = X[p * d + cc];
        if (cc == 0) xnS[k + a] = w.xn[p];
    }
}

// rho -= rownorms(G)^2 (G = R L^-T, P-strided columns), clamped at 0, and the
// per-64-row-tile sum and (max, lowest index) of rho that the proposal kernel
// reads, summed in the FP64 engine's order.  256 threads = 4 tiles; i0 is a
// multiple of 64.
__global__ void __launch_bounds__(256) k_lm_rho(FactorWs w, const double* __restrict__ G, int64_t P, int64_t Pc,
                                                int m, int64_t i0, double* __restrict__ rho) {
    __shared__ double ssum[8], smax[8];
    __shared__ int64_t sidx[8];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t li = (int64_t)blockIdx.x * 256 + tid;
    double rnew = 0.0, rmax = -1.0;
    int64_t ridx = LLONG_MAX;
    if (li < Pc) {
        const int64_t row = i0 + li;
        double nrm = 0.0;
        for (int j = 0; j < m; ++j) {
            const double g = G[(int64_t)j * P + li];
            nrm = fma(g, g, nrm);
        }
        rnew = fmax(rho[row] - nrm, 0.0);
        rho[row] = rnew;
        rmax = rnew;
        ridx = row;
    }
    const double sw = warp_sum(rnew);
    warp_argmax(rmax, ridx);
    if (lane == 0) {
        ssum[wid] = sw;
        smax[wid] = rmax;
        sidx[wid] = ridx;
    }
    __syncthreads();
    if (tid < 4) {
        const int64_t lt = (int64_t)blockIdx.x * 256 + 64 * tid;   // first local row of the tile
        if (lt < Pc) {
            double ts = 0.0, tm = -1.0;
            int64_t ti = LLONG_MAX;
            for (int q = 2 * tid; q < 2 * tid + 2; ++q) {
                ts += ssum[q];
                argmax_merge(tm, ti, smax[q], sidx[q]);
            }
            const int64_t t = (i0 + lt) / kBM;
            w.tile_sum[t] = ts;
            w.tile_max[t] = tm;
            w.tile_idx[t] = ti;
        }
    }
}

// ---------------------------------------------------------------------------
// Normalisation kernels
// ---------------------------------------------------------------------------
__global__ void k_lm_fill(double* __restrict__ x, int64_t n, double v) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = v;
}

// 1/d~ of a panel's rows; flags bit 0 where d~ <= 0 (Algorithm 1, first assert).
__global__ void k_lm_recip(const double* __restrict__ d, int64_t n, double* __restrict__ out, int* __restrict__ flags) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (!(d[i] > 0.0)) atomicOr(flags, 1);
    out[i] = 1.0 / d[i];
}

// Gram weights of a panel's rows, 1/d~^2 and 1/q~ (with root the row scales 1/d~ and
// 1/sqrt(q~) that the tensor-core Grams take); flags bit 1 where q~ <= 0.
__global__ void k_lm_weights(const double* __restrict__ d, const double* __restrict__ q, int64_t n, int root,
                             double* __restrict__ wa, double* __restrict__ wc, int* __restrict__ flags) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (!(q[i] > 0.0)) atomicOr(flags, 2);
    wa[i] = 1.0 / (root ? d[i] : d[i] * d[i]);
    wc[i] = 1.0 / (root ? sqrt(q[i]) : q[i]);
}

constexpr int kLmSMs = 152;   // wave sizing of the Gram grids (a performance choice only)

static int grid1(int64_t n) { return (int)((n + 255) / 256); }

// ---------------------------------------------------------------------------
// Workspaces
// ---------------------------------------------------------------------------
struct LmFactorWs {
    FactorWs w;
    LmPanel p;
    double* Zt;    // r x b: F(T,:)^T, then W^-T F(T,:)^T
};

static LmFactorWs carve_lm_factor(void* base, int64_t N, int d, int r, int b, size_t* bytes) {
    LmFactorWs L{};
    size_t fb = 0;
    L.w = carve_factor_fp64(base, N, d, r, b, &fb);
    Carver c(base);
    c.off = fb;
    L.p = carve_panel(c, N, d, r, false);
    L.p.xn = L.w.xn;   // |x_i|^2 of the FP64 path's workspace
    L.Zt = c.take<double>((size_t)r * b);
    *bytes = c.off;
    return L;
}

// The factor's dot products X X(S,:)^T and its products with L^-1 run on the tensor cores, with
// their scratch taken out of the panel's own memory, so that the workspace stays as it is:
// `rows` of the P rows are formed at a time, and the rest of the buffer holds the operands (14
// max(d, 128) bytes a row beside the panel's 8 r).  K(p,S) Z stays with the library's FP64
// GEMM: Z's entries reach far above 1, and digits cut by the largest entry of a row left rho
// with 1.4 times the GEMM's error against 64 bits.  For blocks from 32 on (the FP64 path's line:
// below, a block leaves most of a 128-row tile of the right operand empty), from 1,024
// rows on and for N r >= 7 2^18, where the factor costs more than the launches that a round adds
// (whole factor, d = 64, b = 32, these products / the library's, ms: N r = 1.0 2^20: N = 16,000
// 1.05 / 0.83, 8,000 1.84 / 1.65, 4,000 4.42 / 4.04; 1.95 2^20: 30,000 1.18 / 1.30, 16,000 2.01 / 2.21,
// 8,000 4.61 / 5.27, b = 64 at 4,000 8.12 / 8.23); otherwise the library's FP64 products and
// solves serve.
constexpr int64_t kLmOzWork = (int64_t)7 << 18;
struct LmRound {
    LmPanel p;     // Kp and P of the rows formed at a time
    LmOz o;
    OzWs li;       // L(T,T)^-1
};
static size_t carve_lm_round(Carver& c, LmRound& q, int64_t rows, int d, int r, int b) {
    q.o.nqx = (d + 15) / 16;
    q.p.P = rows;
    q.p.Kp = c.take<double>((size_t)rows * r);
    carve_lm_oz(c, q.o, rows, std::max(q.o.nqx, kLmBlock / 16), 0, 0, 0);
    q.o.XSp = c.take<uint16_t>(oz_tile_elems(r, q.o.nqx, kDigits));
    q.o.xse = c.take<int>(r);
    q.o.flags = c.take<int>(4);
    q.li.ldR = (b + 15) / 16 * 16;
    q.li.ldLi = (b + 1) / 2 * 2;
    q.li.Lp = c.take<uint16_t>(oz_tile_elems(b, q.li.ldR / 16, kDigits));
    q.li.le = c.take<int>(b);
    q.li.Linv = c.take<double>((size_t)b * q.li.ldLi);
    return c.off;
}
static bool lm_round(const LmPanel& p, int64_t N, int d, int r, int b, LmRound* q) {
    if (b < 32 || N * r < kLmOzWork || !oz_engine_enabled()) return false;
    const size_t bytes = (size_t)p.P * r * sizeof(double);
    q->p = p;
    int64_t lo = 0, hi = std::min<int64_t>(p.P, (N + 127) / 128 * 128) / 128;   // in tiles of 128 rows
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) / 2;
        Carver c(nullptr);
        LmRound t{};
        if (carve_lm_round(c, t, 128 * mid, d, r, b) <= bytes) lo = mid; else hi = mid - 1;
    }
    if (128 * lo < kLmOzRows) return false;
    Carver c(p.Kp);
    carve_lm_round(c, *q, 128 * lo, d, r, b);
    return true;
}

struct LmNormWs {
    LmPanel p;
    double* ones;   // P
    double* vec;    // rank: K(S,:) 1, then K(S,:) d~^-1
    double* y;      // rank: the solved vectors
    double* pv;     // P: 1/d~ of the panel's rows
    double* wa;     // P: 1/d~^2 (tensor-core Grams: 1/d~)
    double* wc;     // P: 1/q~ (tensor-core Grams: 1/sqrt(q~))
    double* gpart;  // Gram split partials of one panel
    int* flags;     // [0] bit 0: d~ <= 0, bit 1: q~ <= 0, bit 2: pivot out of range; [1], [2]: a bounded wait of
                    // the Grams, of the products gave up (bit 2)
    // tensor-core Grams of one panel
    uint32_t *sa_hi, *sc_hi, *cmax;
    int* ecol;
    uint16_t* planes;
    // tensor-core products and solve, o.rows rows of the panel at a time, in the memory of
    // the Grams' planes; o.rows = 0: the library's FP64 products
    LmOz o;
    double* Winv;     // rank x kLmBlock: W's diagonal blocks, then their inverses
    uint16_t *Wd, *Wr, *Wp;   // the planes of the blocks, of what those leave out, of the inverses
    int *wde, *wre, *we;
};

// The products' scratch for `rows` rows, in base (a size with base = NULL).
static size_t carve_lm_solve(void* base, LmOz& o, int64_t rows, int rank) {
    Carver c(base);
    carve_lm_oz(c, o, rows, std::max(o.nqx, kLmBlock / 16), rank, kLmBlock / 16, kLmBlock);
    return c.off;
}

// tc: with the buffers of the tensor-core Grams (without them a smaller workspace still
// serves, by the FP64-pipe Grams).
static LmNormWs carve_lm_norm(void* base, int64_t N, int d, int rank, bool tc, size_t* bytes) {
    Carver c(base);
    LmNormWs L{};
    L.p = carve_panel(c, N, d, rank);
    const int64_t P = L.p.P;
    L.ones = c.take<double>(P);
    L.vec = c.take<double>(rank);
    L.y = c.take<double>(rank);
    L.pv = c.take<double>(P);
    L.wa = c.take<double>(P);
    L.wc = c.take<double>(P);
    L.gpart = c.take<double>(std::max(kevd_gram_partial_doubles(P, rank),
                                      tc ? gram_oz_panel_partial_doubles(P, rank, kLmSMs) : (size_t)0));
    L.flags = c.take<int>(4);
    if (tc) {
        L.sa_hi = c.take<uint32_t>(P);
        L.sc_hi = c.take<uint32_t>(P);
        L.cmax = c.take<uint32_t>(2 * (size_t)rank);
        L.ecol = c.take<int>(2 * (size_t)rank);
        // products and solve from rank 32 on, with as many rows as 64 MiB hold (of X's planes, or
        // of 128 columns of F and of a product), at least 1,024
        L.o.nqx = (d + 15) / 16;
        int64_t rows = (std::min<int64_t>(P, N) + 127) / 128 * 128;
        LmOz t = L.o;
        while (rows >= kLmOzRows && carve_lm_solve(nullptr, t, rows, rank) > kLmScratch) rows = rows / 256 * 128;
        if (rank < 32 || rows < kLmOzRows) rows = 0;
        const size_t solve = rows ? carve_lm_solve(nullptr, t, rows, rank) : 0;
        char* scratch = c.take<char>(std::max(solve, gram_oz_panel_plane_bytes(P, rank)));
        L.planes = reinterpret_cast<uint16_t*>(scratch);
        if (rows) {
            if (base) carve_lm_solve(scratch, L.o, rows, rank);
            L.o.rows = rows;
            L.o.XSp = c.take<uint16_t>(oz_tile_elems(rank, L.o.nqx, kDigits));
            L.o.xse = c.take<int>(rank);
            L.Winv = rows >= rank ? L.o.C : c.take<double>((size_t)rank * kLmBlock);   // (read before the first product)
            L.Wd = c.take<uint16_t>(oz_tile_elems(rank, kLmBlock / 16, kDigits));
            L.Wr = c.take<uint16_t>(oz_tile_elems(rank, kLmBlock / 16, kDigits));
            L.Wp = c.take<uint16_t>(oz_tile_elems(rank, kLmBlock / 16, kDigits));
            L.wde = c.take<int>(rank);
            L.wre = c.take<int>(rank);
            L.we = c.take<int>(rank);
        }
        L.o.flags = L.flags + 2;
    }
    *bytes = c.off;
    return L;
}

static int lm_rounds(const kevd_opts* o, int r, int b, int greedy) {
    if (o->until_rank) return o->max_rounds > 0 ? o->max_rounds : 4 * ((r + b - 1) / b) + 16;
    return greedy ? r : r / b;
}

static bool aligned(const void* p) { return reinterpret_cast<uintptr_t>(p) % kAlign == 0; }

// y := W^-T W^-1 y (two triangular solves with the lower triangular W).
static int solve_ww(cublasHandle_t h, const double* W, int64_t ldw, int rank, double* y) {
    LM_BLAS(cublasDtrsv(h, CUBLAS_FILL_MODE_LOWER, CUBLAS_OP_N, CUBLAS_DIAG_NON_UNIT, rank, W, (int)ldw, y, 1));
    LM_BLAS(cublasDtrsv(h, CUBLAS_FILL_MODE_LOWER, CUBLAS_OP_T, CUBLAS_DIAG_NON_UNIT, rank, W, (int)ldw, y, 1));
    return KEVD_OK;
}

// The planes of W's diagonal blocks, of what those leave out and of the blocks' inverses.
static int solve_setup(cublasHandle_t h, const double* W, int64_t ldw, int rank, const LmNormWs& L, cudaStream_t s) {
    const double one = 1.0;
    k_lm_diag<<<dim3(grid1(rank), kLmBlock), 256, 0, s>>>(W, ldw, L.Winv, rank);
    KEVD_CUDA_TRY(oz_cut_rows(L.Winv, rank, rank, kLmBlock, kLmBlock / 16, L.Wd, L.wde, L.o.rmax, s));
    k_lm_rest<<<dim3(grid1(rank), kLmBlock), 256, 0, s>>>(L.Winv, rank, L.wde);
    KEVD_CUDA_TRY(oz_cut_rows(L.Winv, rank, rank, kLmBlock, kLmBlock / 16, L.Wr, L.wre, L.o.rmax, s));
    KEVD_CUDA_TRY(cudaMemsetAsync(L.Winv, 0, (size_t)rank * kLmBlock * sizeof(double), s));
    k_lm_unit<<<grid1(rank), 256, 0, s>>>(L.Winv, rank);
    KEVD_LAUNCH_CHECK();
    for (int j = 0; j < rank; j += kLmBlock) {
        const int nb = std::min(kLmBlock, rank - j);
        LM_BLAS(cublasDtrsm(h, CUBLAS_SIDE_LEFT, CUBLAS_FILL_MODE_LOWER, CUBLAS_OP_N, CUBLAS_DIAG_NON_UNIT, nb, nb, &one,
                            W + (int64_t)j * ldw + j, (int)ldw, L.Winv + j, rank));
    }
    KEVD_CUDA_TRY(oz_cut_rows(L.Winv, rank, rank, kLmBlock, kLmBlock / 16, L.Wp, L.we, L.o.rmax, s));
    return KEVD_OK;
}

// F_p = K(p,S) W^-T in place on the tensor cores, 128 columns at a time: F_J = R_J W_JJ^-T with
// the block's explicit inverse, then R(:, > J) -= F_J W(> J, J)^T.  Exponents are per row, so
// that W may be of any scale.  Measured at N = 60,000, rank 356: 7.6 ms of the Gram
// stage, 18.5 with the library's triangular solve.
static int solve_panel(const double* W, int64_t ldw, int rank, int64_t Pc, const LmNormWs& L, cudaStream_t s) {
    const LmOz& o = L.o;
    const int64_t P = L.p.P;
    constexpr int nq = kLmBlock / 16;
    const size_t tile = oz_tile_elems(kLmBlock, nq, kDigits);   // a diagonal block's planes
    for (int j = 0; j < rank; j += kLmBlock) {
        const int nb = std::min(kLmBlock, rank - j), rest = rank - j - nb;
        if (rest > 0)
            KEVD_CUDA_TRY(oz_cut_rows(W + (int64_t)j * ldw + j + nb, ldw, rest, nb, nq, o.Bp, o.be, o.rmax, s));
        for (int64_t r0 = 0; r0 < Pc; r0 += o.rows) {
            const int rows = (int)std::min(o.rows, Pc - r0);
            double* R = L.p.Kp + (int64_t)j * P + r0;
            const size_t at = (size_t)(j / kLmBlock) * tile;
            const int st = solve_block(o, R, P, rows, nb, OzOperand{L.Wd + at, nq, L.wde + j, 0},
                                       OzOperand{L.Wr + at, nq, L.wre + j, 0}, OzOperand{L.Wp + at, nq, L.we + j, 0}, s);
            if (st != KEVD_OK) return st;
            if (rest == 0) continue;
            KEVD_CUDA_TRY(oz_cut_rows(R, P, rows, nb, nq, o.Ap, o.ae, o.rmax, s));
            for (int c = 0; c < rest; c += kLmBlock) {
                const int n = std::min(kLmBlock, rest - c);
                KEVD_CUDA_TRY(lm_product(OzOperand{o.Ap, nq, o.ae, 0},
                                         OzOperand{o.Bp + (size_t)(c / kLmBlock) * tile, nq, o.be + c, 0}, rows, n,
                                         kLmBlock, o.C, o.rows, o.flags, s));
                k_lm_sub<<<dim3(grid1(rows), n), 256, 0, s>>>(R + (int64_t)(nb + c) * P, P, o.C, o.rows, rows);
            }
        }
    }
    KEVD_LAUNCH_CHECK();
    return KEVD_OK;
}

}  // namespace kevd

using namespace kevd;

size_t kevd_lowmem_factor_ws(int64_t N, int32_t d, int32_t r, const kevd_opts* o) {
    if (!o || N < 1 || d < 1 || r < 1 || r > N) return 0;
    const int b = o->mode == KEVD_GREEDY ? 1 : o->block_b;
    if (b < 1 || b > 128) return 0;
    size_t bytes = 0;
    carve_lm_factor(nullptr, N, d, r, b, &bytes);
    return bytes;
}

size_t kevd_lowmem_normalize_ws(int64_t N, int32_t d, int32_t rank) {
    if (N < 1 || d < 1 || rank < 1 || rank > N) return 0;
    size_t bytes = 0;
    carve_lm_norm(nullptr, N, d, rank, true, &bytes);
    return bytes;
}

size_t kevd_lowmem_lift_bytes(int64_t N, int d, int rank) {
    Carver c(nullptr);
    carve_panel(c, N, d, rank);
    c.take<int>(4);
    return c.off;
}

extern "C" int rpchol_factor_lowmem(const double* X, int64_t N, int32_t d, double eps, int32_t r,
                                    const kevd_opts* opts, double* W, int64_t ldw, int64_t* pivots, double* rho,
                                    int64_t* proposals, kevd_factor_info* info, void* workspace, size_t ws_bytes,
                                    void* stream) {
    if (!opts || !X || !W || !pivots || !rho || !info) return KEVD_EINVAL;
    if (N < 1 || N > INT_MAX || d < 1 || r < 1 || r > N || ldw < r || ldw > INT_MAX) return KEVD_EINVAL;
    if (!(eps > 0.0) || !isfinite(eps)) return KEVD_EINVAL;
    if (opts->mode != KEVD_GREEDY && opts->mode != KEVD_ARPC) return KEVD_EINVAL;
    if (opts->precision != KEVD_PREC_FP64) return KEVD_EINVAL;
    if (opts->reserved != 0 || opts->max_rounds < 0) return KEVD_EINVAL;
    if (!(opts->tol >= 0.0 && opts->tol < 1.0)) return KEVD_EINVAL;
    const int greedy = opts->mode == KEVD_GREEDY;
    const int b = greedy ? 1 : opts->block_b;
    if (b < 1 || b > 128) return KEVD_EINVAL;
    const int rounds = lm_rounds(opts, r, b, greedy);
    if (rounds < 1) return KEVD_EINVAL;
    size_t need = 0;
    LmFactorWs L = carve_lm_factor(workspace, N, d, r, b, &need);
    if (!workspace || ws_bytes < need || !aligned(workspace)) return KEVD_EWORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cublasHandle_t h = lm_blas(s);
    if (!h) return KEVD_ECUDA;
    const FactorWs& w = L.w;
    LmRound q{};
    const bool tc = lm_round(L.p, N, d, r, b, &q);
    const LmOz& o = q.o;
    const LmPanel& p = tc ? q.p : L.p;
    const double inv_eps = 1.0 / eps, one = 1.0, mone = -1.0;
    {
        TraceScope tr(kStOther, s);
        KEVD_CUDA_TRY(cudaMemset2DAsync(W, (size_t)ldw * sizeof(double), 0, (size_t)r * sizeof(double), r, s));
        launch_prepare_fp64(X, N, d, w, rho, s);
        if (tc) KEVD_CUDA_TRY(cudaMemsetAsync(o.flags, 0, sizeof(int), s));
    }
    KEVD_LAUNCH_CHECK();

    int k = 0;   // committed rank, as the proposal kernel will see it
    for (int rnd = 0; rnd < rounds; ++rnd) {
        {
            TraceScope tr(kStPropose, s);
            launch_propose(w, rho, N, b, r, greedy, opts->seed, rnd, proposals, opts->tol * N, s);
        }
        {
            TraceScope tr(kStGather, s);
            k_lm_gather_prop<<<grid1((int64_t)d * b), 256, 0, s>>>(w, X, d, b);
            if (k > 0) {
                k_lm_kq<<<grid1((int64_t)b * k), 256, 0, s>>>(w, p.XS, p.xnS, pivots, k, d, b, inv_eps);
                LM_BLAS(cublasDtrsm(h, CUBLAS_SIDE_RIGHT, CUBLAS_FILL_MODE_LOWER, CUBLAS_OP_T, CUBLAS_DIAG_NON_UNIT, b,
                                    k, &one, W, (int)ldw, w.FSP, b));   // F(S',:) = K(S',S) W^-T
            }
        }
        KEVD_LAUNCH_CHECK();
        {
            TraceScope tr(kStBlockH, s);
            launch_blockH(w, d, b, inv_eps, s);
        }
        {
            TraceScope tr(kStReject, s);
            KEVD_CUDA_TRY(launch_reject(w, b, r, greedy, opts->seed, rnd, pivots, s));
        }
        FactorState hs;
        KEVD_CUDA_TRY(cudaMemcpyAsync(&hs, w.st, sizeof(hs), cudaMemcpyDeviceToHost, s));
        KEVD_CUDA_TRY(cudaStreamSynchronize(s));
        if (hs.done) break;
        if (hs.k != k) return KEVD_ECUDA;
        const int m = hs.m;
        if (m == 0) continue;
        TraceScope tr(kStEngine, s);
        k_lm_extend<<<grid1((int64_t)m * (k + m + d)), 256, 0, s>>>(w, X, d, k, m, b, pivots, W, ldw, p.XS, p.xnS,
                                                                   L.Zt);
        KEVD_LAUNCH_CHECK();
        if (k > 0)   // Z = W^-T F(T,:)^T with the leading k x k block of W
            LM_BLAS(cublasDtrsm(h, CUBLAS_SIDE_LEFT, CUBLAS_FILL_MODE_LOWER, CUBLAS_OP_T, CUBLAS_DIAG_NON_UNIT, k, m,
                                &one, W, (int)ldw, L.Zt, k));
        // Measured at N = 60,000, r = 512, b = 64: 17.6 ms of engine time, 32.7 with the library's
        // products and solves only.
        const int nm = (m + 15) / 16;
        if (tc) {
            KEVD_CUDA_TRY(oz_cut_rowmajor(p.XS, k + m, d, o.XSp, o.xse, s));
            KEVD_CUDA_TRY(launch_linv(w, q.li, b, s));
        }
        for (int64_t i0 = 0; i0 < N; i0 += p.P) {
            const int64_t Pc = std::min(p.P, N - i0);
            const int st = kernel_panel(h, X, d, i0, Pc, k + m, p, pivots, inv_eps, nullptr, s, tc ? &o : nullptr);
            if (st != KEVD_OK) return st;
            double* R = p.Kp + (int64_t)k * p.P;
            if (k > 0)   // R = K(p,T) - K(p,S) Z
                LM_BLAS(cublasDgemm(h, CUBLAS_OP_N, CUBLAS_OP_N, (int)Pc, m, k, &mone, p.Kp, (int)p.P, L.Zt, k, &one,
                                    R, (int)p.P));
            if (tc) {   // G = R L^-T
                KEVD_CUDA_TRY(oz_cut_rows(R, p.P, (int)Pc, m, nm, o.Ap, o.ae, o.rmax, s));
                KEVD_CUDA_TRY(lm_product(OzOperand{o.Ap, nm, o.ae, 0}, OzOperand{q.li.Lp, q.li.ldR / 16, q.li.le, 0},
                                         Pc, m, 16 * nm, R, p.P, o.flags, s));
            } else {    // Lc is L row-major (ld b), i.e. L^T column-major
                LM_BLAS(cublasDtrsm(h, CUBLAS_SIDE_RIGHT, CUBLAS_FILL_MODE_UPPER, CUBLAS_OP_N, CUBLAS_DIAG_NON_UNIT, (int)Pc,
                                    m, &one, w.Lc, b, R, (int)p.P));
            }
            k_lm_rho<<<grid1(Pc), 256, 0, s>>>(w, R, p.P, Pc, m, i0, rho);
            KEVD_LAUNCH_CHECK();
        }
        k += m;
    }
    {
        TraceScope tr(kStOther, s);
        launch_finalize(w, rho, N, s);
    }
    KEVD_LAUNCH_CHECK();
    FactorState hs;
    int gave_up = 0;
    KEVD_CUDA_TRY(cudaMemcpyAsync(&hs, w.st, sizeof(hs), cudaMemcpyDeviceToHost, s));
    if (tc) KEVD_CUDA_TRY(cudaMemcpyAsync(&gave_up, o.flags, sizeof(int), cudaMemcpyDeviceToHost, s));
    KEVD_CUDA_TRY(cudaStreamSynchronize(s));
    trace_flush();
    if (gave_up) return KEVD_ETIMEOUT;
    info->rank = hs.k;
    info->rounds = hs.rounds;
    info->trace_err = hs.final_sum;
    info->sum_m_sq = hs.sum_m_sq;
    info->sum_k = hs.sum_k;
    info->engine_rounds = hs.eng_rounds;
    if (hs.bad) return KEVD_EINVAL;
    return KEVD_OK;
}

extern "C" int bistoch_normalize_lowmem(const double* X, int64_t N, int32_t d, double eps, const int64_t* pivots,
                                        const double* W, int64_t ldw, int32_t rank, double* dtil, double* qtil,
                                        double* A, double* C, void* workspace, size_t ws_bytes, void* stream) {
    if (!X || !pivots || !W || !dtil || !qtil || !A || !C) return KEVD_EINVAL;
    if (N < 1 || N > INT_MAX || d < 1 || rank < 1 || rank > N || ldw < rank || ldw > INT_MAX) return KEVD_EINVAL;
    if (!(eps > 0.0) || !isfinite(eps)) return KEVD_EINVAL;
    size_t need = 0;
    LmNormWs L = carve_lm_norm(workspace, N, d, rank, true, &need);
    const size_t need_tc = need;
    const bool tc = gram_oz_eligible(N, rank) && ws_bytes >= need;
    if (ws_bytes < need) L = carve_lm_norm(workspace, N, d, rank, false, &need);
    if (!workspace || ws_bytes < need || !aligned(workspace)) return KEVD_EWORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cublasHandle_t h = lm_blas(s);
    if (!h) return KEVD_ECUDA;
    const LmPanel& p = L.p;
    const double inv_eps = 1.0 / eps, one = 1.0, zero = 0.0;
    // (the products follow KEVD_ENGINE, the Grams KEVD_GRAM)
    const LmOz* po = ws_bytes >= need_tc && L.o.rows > 0 && oz_engine_enabled() ? &L.o : nullptr;
    const bool one_panel = N <= p.P;   // the panel is formed once and kept for all three passes
    int st;

    KEVD_CUDA_TRY(cudaMemsetAsync(L.flags, 0, 4 * sizeof(int), s));
    {
        TraceScope tr(kStDegree, s);
        k_lm_norms<<<grid1(N), 256, 0, s>>>(X, N, d, p.xn);
        k_lm_gather<<<grid1((int64_t)rank * d), 256, 0, s>>>(X, N, d, pivots, rank, p.xn, p.XS, p.xnS, L.flags);
        k_lm_fill<<<grid1(p.P), 256, 0, s>>>(L.ones, p.P, 1.0);
        KEVD_LAUNCH_CHECK();
        if (po) {
            KEVD_CUDA_TRY(oz_cut_rowmajor(p.XS, rank, d, po->XSp, po->xse, s));
        }
        // pass 1: K(S,:) 1, then y = W^-T W^-1 K(S,:) 1
        KEVD_CUDA_TRY(cudaMemsetAsync(L.vec, 0, (size_t)rank * sizeof(double), s));
        for (int64_t i0 = 0; i0 < N; i0 += p.P) {
            const int64_t Pc = std::min(p.P, N - i0);
            if ((st = kernel_panel(h, X, d, i0, Pc, rank, p, pivots, inv_eps, nullptr, s, po)) != KEVD_OK) return st;
            LM_BLAS(cublasDgemv(h, CUBLAS_OP_T, (int)Pc, rank, &one, p.Kp, (int)p.P, L.ones, 1, &one, L.vec, 1));
        }
        KEVD_CUDA_TRY(cudaMemcpyAsync(L.y, L.vec, (size_t)rank * sizeof(double), cudaMemcpyDeviceToDevice, s));
        if ((st = solve_ww(h, W, ldw, rank, L.y)) != KEVD_OK) return st;
        // pass 2: d~ = K(:,S) y and K(S,:) d~^-1, then y = W^-T W^-1 K(S,:) d~^-1
        KEVD_CUDA_TRY(cudaMemsetAsync(L.vec, 0, (size_t)rank * sizeof(double), s));
        for (int64_t i0 = 0; i0 < N; i0 += p.P) {
            const int64_t Pc = std::min(p.P, N - i0);
            if (!one_panel &&
                (st = kernel_panel(h, X, d, i0, Pc, rank, p, pivots, inv_eps, nullptr, s, po)) != KEVD_OK)
                return st;
            LM_BLAS(cublasDgemv(h, CUBLAS_OP_N, (int)Pc, rank, &one, p.Kp, (int)p.P, L.y, 1, &zero, dtil + i0, 1));
            k_lm_recip<<<grid1(Pc), 256, 0, s>>>(dtil + i0, Pc, L.pv, L.flags);
            KEVD_LAUNCH_CHECK();
            LM_BLAS(cublasDgemv(h, CUBLAS_OP_T, (int)Pc, rank, &one, p.Kp, (int)p.P, L.pv, 1, &one, L.vec, 1));
        }
        KEVD_CUDA_TRY(cudaMemcpyAsync(L.y, L.vec, (size_t)rank * sizeof(double), cudaMemcpyDeviceToDevice, s));
        if ((st = solve_ww(h, W, ldw, rank, L.y)) != KEVD_OK) return st;
    }
    {
        // pass 3: q~ = K(:,S) y; F_p = K(p,S) W^-T; A += F_p^T D~^-2 F_p, C += F_p^T Q~^-1 F_p
        TraceScope tr(kStGram, s);
        for (int64_t i0 = 0; i0 < N; i0 += p.P) {
            const int64_t Pc = std::min(p.P, N - i0);
            if (!one_panel &&
                (st = kernel_panel(h, X, d, i0, Pc, rank, p, pivots, inv_eps, nullptr, s, po)) != KEVD_OK)
                return st;
            LM_BLAS(cublasDgemv(h, CUBLAS_OP_N, (int)Pc, rank, &one, p.Kp, (int)p.P, L.y, 1, &zero, qtil + i0, 1));
            k_lm_weights<<<grid1(Pc), 256, 0, s>>>(dtil + i0, qtil + i0, Pc, tc, L.wa, L.wc, L.flags);
            KEVD_LAUNCH_CHECK();
            if (po) {
                if (i0 == 0 && (st = solve_setup(h, W, ldw, rank, L, s)) != KEVD_OK) return st;
                if ((st = solve_panel(W, ldw, rank, Pc, L, s)) != KEVD_OK) return st;
            } else {
                LM_BLAS(cublasDtrsm(h, CUBLAS_SIDE_RIGHT, CUBLAS_FILL_MODE_LOWER, CUBLAS_OP_T, CUBLAS_DIAG_NON_UNIT,
                                    (int)Pc, rank, &one, W, (int)ldw, p.Kp, (int)p.P));
            }
            if (tc)
                KEVD_CUDA_TRY(launch_gram_oz_panel(p.Kp, p.P, p.P, Pc, rank, L.wa, L.wc, L.sa_hi, L.sc_hi, L.cmax,
                                                   L.ecol, L.gpart, L.planes, L.flags + 1, A, C, i0 > 0, kLmSMs, s));
            else
                KEVD_CUDA_TRY(kevd_gram_weighted(p.Kp, p.P, Pc, rank, L.wa, L.wc, L.gpart, A, C, i0 > 0, s));
        }
    }
    int flags[3] = {0, 0, 0};
    KEVD_CUDA_TRY(cudaMemcpyAsync(flags, L.flags, sizeof(flags), cudaMemcpyDeviceToHost, s));
    KEVD_CUDA_TRY(cudaStreamSynchronize(s));
    trace_flush();
    if (flags[0] & 4) return KEVD_EINVAL;
    if (flags[0] & 1) return KEVD_ED_NONPOS;
    if (flags[0] & 2) return KEVD_EQ_NONPOS;
    if (flags[1] | flags[2]) return KEVD_ETIMEOUT;
    return KEVD_OK;
}

int kevd_lowmem_lift(const KevdLowmemLift& Lf, int64_t N, int rank, int k, double* Y, const double* dtil, double* U,
                     cudaStream_t s) {
    Carver c(Lf.ws);
    const LmPanel p = carve_panel(c, N, Lf.d, rank);
    int* flags = c.take<int>(4);
    cublasHandle_t h = lm_blas(s);
    if (!h) return KEVD_ECUDA;
    const double one = 1.0, zero = 0.0;
    int st;
    {
        TraceScope tr(kStLift, s);
        KEVD_CUDA_TRY(cudaMemsetAsync(flags, 0, 4 * sizeof(int), s));
        LM_BLAS(cublasDtrsm(h, CUBLAS_SIDE_LEFT, CUBLAS_FILL_MODE_LOWER, CUBLAS_OP_T, CUBLAS_DIAG_NON_UNIT, rank, k, &one,
                            Lf.W, (int)Lf.ldw, Y, rank));   // Y := W^-T Y
        k_lm_norms<<<grid1(N), 256, 0, s>>>(Lf.X, N, Lf.d, p.xn);
        k_lm_gather<<<grid1((int64_t)rank * Lf.d), 256, 0, s>>>(Lf.X, N, Lf.d, Lf.piv, rank, p.xn, p.XS, p.xnS, flags);
        KEVD_LAUNCH_CHECK();
        for (int64_t i0 = 0; i0 < N; i0 += p.P) {   // U(p,:) = D~^-1 K(p,S) (W^-T Y)
            const int64_t Pc = std::min(p.P, N - i0);
            if ((st = kernel_panel(h, Lf.X, Lf.d, i0, Pc, rank, p, Lf.piv, Lf.inv_eps, dtil, s)) != KEVD_OK) return st;
            LM_BLAS(cublasDgemm(h, CUBLAS_OP_N, CUBLAS_OP_N, (int)Pc, k, rank, &one, p.Kp, (int)p.P, Y, rank, &zero,
                                U + i0, (int)N));
        }
    }
    int hf = 0;
    KEVD_CUDA_TRY(cudaMemcpyAsync(&hf, flags, sizeof(int), cudaMemcpyDeviceToHost, s));
    KEVD_CUDA_TRY(cudaStreamSynchronize(s));
    return (hf & 4) ? KEVD_EINVAL : KEVD_OK;
}
