// FP64 offline stage of Algorithm 1 ("compute KKT inverse, W and b for each
// rho", Sec. III-B).
//
// For a bank entry with row penalties rho_r s (s_i = 1, or eq_scale on equality
// rows, Sec. II-B):
//   C   = A^T diag(s) A                          (once for all entries)
//   K   = P + sigma I + rho_r C                  (the matrix of Eq. Xbar_update)
//   K   = L L^T                                  (blocked right-looking Cholesky)
//   D   = K^{-1} = L^{-T} L^{-1}                 (L^{-1} by recursive doubling)
//   T   = L^{-1} A^T,  V = [D A^T; A D A^T] = [L^{-T} T; T^T T]
//   X   = sigma [D; AD] - rho_r V diag(s) A      (= [D; AD] (sigma I - rho_r C))
// (A row with a large penalty has a small column of T, and V and X keep their relative
// accuracy there.  With A D A^T formed from D, and X as [D; AD] (sigma I - rho_r C), the
// multipliers of rows with 1000 rho came out 1e-8 off after 75 layers in 64 bits; formed so,
// 1e-11, as from solving K X = [sigma I - rho_r C, A^T, -I].)
// X, V and -[D; AD] hold the layer in the factored form used on the hot path:
//   [x+; (Ax)+] = [X V] [x; 2 rho z - lam'] - [D; AD] q,
// which is Eq. gpu_update with its z and lam columns merged
// (2 D A^T rho z - D A^T lam = D A^T (2 rho z - lam)) and its z row written
// as A x+ + (A x - z + lam'/rho): the paper's z row is
// [A D(sI - A^T rho A) + A, 2 A D A^T rho - I, -A D A^T + rho^{-1}], i.e. A times
// the x row plus [A, -I, rho^{-1}], and [A, -I, rho^{-1}] v = A x - z + lam'/rho.
//
// What bounds it: GB300 runs FP64 at 1.25 TFLOP/s, two FMAs per SM and clock, so a
// 64 x 64 x 64 product alone takes one SM 64 us.  Three things follow.  The flops are
// kept down: D once and symmetric products by halves, 8 n^3 per entry at n = m, where
// solving K X = [sigma I - C, A^T, -I] for all columns and then A X took 14 n^3.  The
// serial chain (diagonal blocks, panels, doubling levels) runs for every entry at
// once, one grid slice per entry, so that it is paid once and not n_rho times.  And
// every product takes the tile that spreads it over the SMs (dgemm_batch).
#include "common.h"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

namespace rq {

namespace {

constexpr int NB = kCholNB;   // Cholesky / triangular-solve block size

// C = alpha op(A) op(B) + beta D, row-major, for a two-level batch: grid slice z is
// problem (z / nb2, z % nb2), each pointer advanced by its level-1 and level-2 strides.
// T x T tiles, 256 threads with (T/16)^2 outputs each, k in order (one fma per step, so
// an output's bits do not depend on T); the next k step's values are loaded into
// registers while the current one is multiplied.  Bound by the FP64 pipe at every T
// (16 clocks per warp instruction): T = 64 runs at 1.0 TFLOP/s on 800 x 2400 x 800.
enum : int {
    G_LOWER = 1,     // only the tiles on and below the diagonal
    G_MIRROR = 2,    // with G_LOWER: also write the transposed element (symmetric result)
    G_KBEG_M = 4,    // op(A) is zero for k < row: k starts at the tile's first row
    G_KBEG_N = 8,    // op(B) is zero for k < column
    G_KEND_M = 16,   // op(A) is zero for k > row: k ends at the tile's last row
    G_KRAG = 32,     // K is the (ragged) row count
};

struct Gemm {
    int M = 0, N = 0, K = 0, lda = 0, ldb = 0, ldc = 0, ldd = 0, nb2 = 1, flags = 0;
    bool ta = false, tb = false;
    int mtot = 0, mstep = 0;   // mstep > 0: problem z2 has min(M, mtot - z2 mstep) rows (a ragged last one)
    const double *A = nullptr, *B = nullptr, *D = nullptr;
    double* C = nullptr;
    long long sA = 0, sB = 0, sC = 0, sD = 0;       // level-1 strides
    long long tA = 0, tB = 0, tC = 0, tD = 0;       // level-2 strides
    double beta = 0.0, alpha[RQ_MAX_RHO];           // alpha by level-1 index
};

template <int T>
__global__ void __launch_bounds__(256) dgemm_kernel(const Gemm g) {
    constexpr int E = T / 16;
    __shared__ double As[16][T + 1];
    __shared__ double Bs[16][T + 1];
    const int z1 = blockIdx.z / g.nb2, z2 = blockIdx.z % g.nb2;
    const int M = g.mstep > 0 ? min(g.M, g.mtot - z2 * g.mstep) : g.M, N = g.N;
    const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
    if (m0 >= M || ((g.flags & G_LOWER) && n0 > m0)) return;
    const double* A = g.A + z1 * g.sA + z2 * g.tA;
    const double* B = g.B + z1 * g.sB + z2 * g.tB;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    int kbeg = 0, kend = (g.flags & G_KRAG) ? min(g.K, M) : g.K;
    if (g.flags & G_KBEG_M) kbeg = m0;
    if (g.flags & G_KBEG_N) kbeg = max(kbeg, n0);
    if (g.flags & G_KEND_M) kend = min(kend, m0 + T);
    double ra[E], rb[E];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int t = 0; t < E; ++t) {
            const int e = threadIdx.x + 256 * t;
            int i, k;
            if (!g.ta) { i = e >> 4; k = e & 15; } else { k = e / T; i = e % T; }
            const int gi = m0 + i, gk = k0 + k;
            ra[t] = (gi < M && gk < kend) ? (g.ta ? A[(size_t)gk * g.lda + gi] : A[(size_t)gi * g.lda + gk]) : 0.0;
        }
#pragma unroll
        for (int t = 0; t < E; ++t) {
            const int e = threadIdx.x + 256 * t;
            int j, k;
            if (!g.tb) { k = e / T; j = e % T; } else { j = e >> 4; k = e & 15; }
            const int gj = n0 + j, gk = k0 + k;
            rb[t] = (gj < N && gk < kend) ? (g.tb ? B[(size_t)gj * g.ldb + gk] : B[(size_t)gk * g.ldb + gj]) : 0.0;
        }
    };
    double acc[E][E];
#pragma unroll
    for (int i = 0; i < E; ++i)
#pragma unroll
        for (int j = 0; j < E; ++j) acc[i][j] = 0.0;
    if (kbeg < kend) fetch(kbeg);
    for (int k0 = kbeg; k0 < kend; k0 += 16) {
#pragma unroll
        for (int t = 0; t < E; ++t) {
            const int e = threadIdx.x + 256 * t;
            if (!g.ta) As[e & 15][e >> 4] = ra[t];
            else As[e / T][e % T] = ra[t];
            if (!g.tb) Bs[e / T][e % T] = rb[t];
            else Bs[e & 15][e >> 4] = rb[t];
        }
        __syncthreads();
        if (k0 + 16 < kend) fetch(k0 + 16);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            double a[E], b[E];
#pragma unroll
            for (int i = 0; i < E; ++i) a[i] = As[k][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < E; ++j) b[j] = Bs[k][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < E; ++i)
#pragma unroll
                for (int j = 0; j < E; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
    const double alpha = g.alpha[z1];
    double* C = g.C + z1 * g.sC + z2 * g.tC;
    const double* D = g.D + z1 * g.sD + z2 * g.tD;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const int gi = m0 + ty + 16 * i;
        if (gi >= M) continue;
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const int gj = n0 + tx + 16 * j;
            if (gj >= N || ((g.flags & G_LOWER) && gj > gi)) continue;
            const double v = g.beta == 0.0 ? alpha * acc[i][j] : fma(alpha, acc[i][j], g.beta * D[(size_t)gi * g.ldd + gj]);
            C[(size_t)gi * g.ldc + gj] = v;
            if (g.flags & G_MIRROR) C[(size_t)gj * g.ldc + gi] = v;
        }
    }
}

// Cholesky of the jb x jb diagonal block at (j0, j0) of every entry's K (grid = entries)
// and the inverse of its factor, which turns the panel and block solves into products.
// Thread (ty, tx) keeps the elements (ty + 16 r, tx + 16 c) of the block and of the
// inverse Y in registers; step k publishes column k of the block and row k of Y, and
// both updates subtract (a_ik / a_kk) times them: one barrier per step, no element of
// the upper triangle touched.  Bound by the FP64 pipe of its one SM and the 32 steps'
// latency.  (Replaces one thread per column of the inverse and three barriers per step
// on 64-wide blocks, 219 us each.)  A pivot <= 0 (or NaN) sets flag[entry] and is
// replaced by 1 so that the rest stays finite; the host then reports NOT_PD.
__global__ void __launch_bounds__(256) potrf_diag_kernel(const double* __restrict__ Km, long long sK, int ld, int j0,
                                                         int jb, double* __restrict__ Lm, long long sL,
                                                         double* __restrict__ Linv, long long sI, int* flag) {
    constexpr int E = NB / 16;
    __shared__ double col[2][NB], row[2][NB], rdiag[2], diag[NB], rsq[NB];
    const double* K = Km + blockIdx.x * sK;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double a[E][E], y[E][E];
#pragma unroll
    for (int r = 0; r < E; ++r)
#pragma unroll
        for (int c = 0; c < E; ++c) {
            const int i = ty + 16 * r, j = tx + 16 * c;
            a[r][c] = (i < jb && j <= i) ? K[(size_t)(j0 + i) * ld + j0 + j] : (i == j ? 1.0 : 0.0);
            y[r][c] = i == j ? 1.0 : 0.0;
        }
#pragma unroll
    for (int kb = 0; kb < E; ++kb)
        for (int kk = 0; kk < 16; ++kk) {
            const int k = 16 * kb + kk, b = k & 1;
            if (tx == kk)
#pragma unroll
                for (int r = kb; r < E; ++r) col[b][ty + 16 * r] = a[r][kb];
            if (ty == kk) {
#pragma unroll
                for (int c = 0; c <= kb; ++c) row[b][tx + 16 * c] = y[kb][c];
                if (tx == kk) {
                    double d = a[kb][kb];
                    if (!(d > 0.0)) {
                        atomicExch(flag + blockIdx.x, 1);
                        d = 1.0;
                    }
                    diag[k] = d;
                    rdiag[b] = 1.0 / d;
                }
            }
            __syncthreads();
            const double rd = rdiag[b];
#pragma unroll
            for (int r = kb; r < E; ++r) {
                const int i = ty + 16 * r;
                if (i <= k) continue;
                const double f = -col[b][i] * rd;
#pragma unroll
                for (int c = kb; c <= r; ++c)
                    if (tx + 16 * c > k) a[r][c] = fma(f, col[b][tx + 16 * c], a[r][c]);
#pragma unroll
                for (int c = 0; c <= kb; ++c) y[r][c] = fma(f, row[b][tx + 16 * c], y[r][c]);
            }
        }
    __syncthreads();
    if (threadIdx.x < NB) rsq[threadIdx.x] = 1.0 / sqrt(diag[threadIdx.x]);
    __syncthreads();
    // column j of L is a's column j over sqrt(diag_j), row i of L^{-1} is y's row i over sqrt(diag_i)
    double* L = Lm + blockIdx.x * sL;
    double* Li = Linv + blockIdx.x * sI;
#pragma unroll
    for (int r = 0; r < E; ++r)
#pragma unroll
        for (int c = 0; c < E; ++c) {
            const int i = ty + 16 * r, j = tx + 16 * c;
            if (i >= jb || j >= jb) continue;
            if (i >= j) L[(size_t)(j0 + i) * ld + j0 + j] = (i > j ? a[r][c] : diag[j]) * rsq[j];
            Li[(size_t)(j0 + i) * ld + j0 + j] = i >= j ? y[r][c] * rsq[i] : 0.0;
        }
}

__global__ void scale_rows_kernel(const double* __restrict__ A, const double* __restrict__ f,
                                  double* __restrict__ out, int m, int n) {
    const size_t total = (size_t)m * n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x)
        out[e] = f[e / n] * A[e];
}

struct RhoList {
    double v[RQ_MAX_RHO];
};

// K_z = P + sigma I + rho_z C for every entry z = blockIdx.y (C = nullptr: zero).
__global__ void kkt_kernel(const double* __restrict__ P, const double* __restrict__ C, double sigma, RhoList rho, int n,
                           double* __restrict__ Km, long long sK) {
    const size_t total = (size_t)n * n;
    const double r = rho.v[blockIdx.y];
    double* K = Km + blockIdx.y * sK;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const double d = (e / n == e % n) ? sigma : 0.0;
        K[e] = P[e] + d + (C ? r * C[e] : 0.0);
    }
}

// out_z (cols x rows) = in_z^T with in_z (rows x cols), entries z = blockIdx.z.
__global__ void transpose_f64_kernel(const double* __restrict__ in, long long s_in, double* __restrict__ out,
                                     long long s_out, int rows, int cols) {
    __shared__ double tile[32][33];
    in += blockIdx.z * s_in;
    out += blockIdx.z * s_out;
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        if (r < rows && c < cols) tile[i][threadIdx.x] = in[(size_t)r * cols + c];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        if (r < rows && c < cols) out[(size_t)c * rows + r] = tile[threadIdx.x][i];
    }
}

// Layer matrices from X (R x n), V (R x m) and DS = [D; AD] (R x n): Wt = [X V]
// (R x ldw, zero padded) and Bop = -DS (R x n), FP32 and optionally FP64.
__global__ void pack_layer_kernel(const double* __restrict__ X, const double* __restrict__ V,
                                  const double* __restrict__ DS, int n, int m, int ldw, float* __restrict__ Wt,
                                  float* __restrict__ Bop, double* __restrict__ Wt64,
                                  double* __restrict__ Bop64) {
    const int R = n + m;
    const size_t total = (size_t)R * (ldw + n);
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / (ldw + n)), c = (int)(e % (ldw + n));
        if (c < ldw) {
            const double v = c < n ? X[(size_t)r * n + c] : c < R ? V[(size_t)r * m + c - n] : 0.0;
            Wt[(size_t)r * ldw + c] = (float)v;
            if (Wt64 && c < R) Wt64[(size_t)r * R + c] = v;
        } else {
            const int k = c - ldw;
            const double v = -DS[(size_t)r * n + k];
            Bop[(size_t)r * n + k] = (float)v;
            if (Bop64) Bop64[(size_t)r * n + k] = v;
        }
    }
}

// out (rows x ldo, FP32) <- in (rows x cols, FP64); the padding stays zero.
__global__ void to_f32_pad_kernel(const double* __restrict__ in, float* __restrict__ out, int rows,
                                  int cols, int ldo) {
    const size_t count = (size_t)rows * cols;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count;
         e += (size_t)gridDim.x * blockDim.x)
        out[(e / cols) * ldo + e % cols] = (float)in[e];
}

// out (cols x ldo, FP32) <- in^T with in (rows x cols, FP64).
__global__ void transpose_f32_kernel(const double* __restrict__ in, float* __restrict__ out,
                                     int rows, int cols, int ldo) {
    __shared__ float tile[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        if (r < rows && c < cols) tile[i][threadIdx.x] = (float)in[(size_t)r * cols + c];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        if (r < rows && c < cols) out[(size_t)c * ldo + r] = tile[threadIdx.x][i];
    }
}

// v = a + b + c with each part the BF16 rounding of what is left (FP64 arithmetic).
__device__ __forceinline__ void split3_f64(double v, __nv_bfloat16& a, __nv_bfloat16& b, __nv_bfloat16& c) {
    a = __double2bfloat16(v);
    const double r1 = v - (double)__bfloat162float(a);
    b = __double2bfloat16(r1);
    c = __double2bfloat16(r1 - (double)__bfloat162float(b));
}

// The three BF16 parts of the factored layer [X V] (rows [x; Ax], K-major rows of ldk);
// rows and columns of A x start at nP.
__global__ void pack_bf16_layer_kernel(const double* __restrict__ X, const double* __restrict__ V, int n, int m, int nP,
                                       int ldk, size_t part, __nv_bfloat16* __restrict__ out) {
    const int R = n + m;
    const size_t total = (size_t)R * ldk;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / ldk), k = (int)(e % ldk);
        const double v = k < n ? X[(size_t)r * n + k] : k >= nP && k < nP + m ? V[(size_t)r * m + k - nP] : 0.0;
        __nv_bfloat16 a, b, c;
        split3_f64(v, a, b, c);
        const size_t o = (size_t)(r < n ? r : r - n + nP) * ldk + k;
        out[o] = a;
        out[o + part] = b;
        out[o + 2 * part] = c;
    }
}

// The three BF16 parts of the check matrix [[P, A^T], [A, 0]] (x columns
// [0, n64), multiplier columns [n64, n64 + m); rows [0, n) and [nP, nP + m)).
__global__ void pack_bf16_check_kernel(const double* __restrict__ P, const double* __restrict__ A, int n, int m, int nP,
                                       int n64, int ldkc, size_t part, __nv_bfloat16* __restrict__ out) {
    const size_t total = (size_t)(n + m) * ldkc;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(e / ldkc), k = (int)(e % ldkc);
        double v = 0.0;
        if (j < n) {
            if (k < n) v = P[(size_t)j * n + k];
            else if (k >= n64 && k < n64 + m) v = A[(size_t)(k - n64) * n + j];
        } else if (k < n) {
            v = A[(size_t)(j - n) * n + k];
        }
        __nv_bfloat16 a, b, c;
        split3_f64(v, a, b, c);
        const size_t o = (size_t)(j < n ? j : j - n + nP) * ldkc + k;
        out[o] = a;
        out[o + part] = b;
        out[o + 2 * part] = c;
    }
}

int grid1d(size_t total) {
    size_t g = (total + 255) / 256;
    if (g > 16384) g = 16384;
    if (g < 1) g = 1;
    return (int)g;
}

// The tile: per-SM time is the number of tiles an SM gets times T^2 (the FP64 pipe),
// smaller tiles pay more for their loads (measured: 64 x 64 at 1.0 TFLOP/s, 32 about 0.9
// of it, 16 about 0.7).  A 60 x 60 x 60 product takes 5 us in 16 x 16 tiles and 64 us in one.
int dgemm_batch(relu_qp_t h, const Gemm& g, int n1) {
    if (g.M <= 0 || g.N <= 0 || n1 <= 0 || g.nb2 <= 0) return RELU_QP_OK;
    const int sms = h->num_sms > 0 ? h->num_sms : 148;
    auto cost = [&](int T, double w) {
        double tiles = (double)ceil_div(g.M, T) * ceil_div(g.N, T);
        if (g.flags & G_LOWER) tiles = 0.5 * (tiles + ceil_div(g.M, T));
        return std::ceil(tiles * n1 * g.nb2 / sms) * T * T * w;
    };
    const double c64 = cost(64, 1.0), c32 = cost(32, 1.1), c16 = cost(16, 1.4);
    const int T = c64 <= c32 && c64 <= c16 ? 64 : c32 <= c16 ? 32 : 16;
    const dim3 grid(ceil_div(g.N, T), ceil_div(g.M, T), n1 * g.nb2);
    if (T == 64) dgemm_kernel<64><<<grid, 256, 0, h->stream>>>(g);
    else if (T == 32) dgemm_kernel<32><<<grid, 256, 0, h->stream>>>(g);
    else dgemm_kernel<16><<<grid, 256, 0, h->stream>>>(g);
    RQ_CUDA(h, cudaGetLastError());
    return RELU_QP_OK;
}

Gemm gemm(bool ta, bool tb, int M, int N, int K, double alpha, const double* A, int lda, const double* B, int ldb,
          double beta, double* C, int ldc) {
    Gemm g;
    g.ta = ta;
    g.tb = tb;
    g.M = M;
    g.N = N;
    g.K = K;
    g.A = A;
    g.lda = lda;
    g.B = B;
    g.ldb = ldb;
    g.C = C;
    g.D = C;
    g.ldc = g.ldd = ldc;
    g.beta = beta;
    for (double& a : g.alpha) a = alpha;
    return g;
}

}  // namespace

int dgemm(relu_qp_t h, bool ta, bool tb, int M, int N, int K, double alpha, const double* A,
          int lda, const double* B, int ldb, double beta, double* C, int ldc) {
    return dgemm_batch(h, gemm(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc), 1);
}

int dgemm_strided(relu_qp_t h, bool ta, bool tb, int M, int N, int K, double alpha, const double* A, int lda,
                  long long tA, const double* B, int ldb, long long tB, double* C, int ldc, long long tC, int nb) {
    Gemm g = gemm(ta, tb, M, N, K, alpha, A, lda, B, ldb, 0.0, C, ldc);
    g.nb2 = nb;
    g.tA = tA;
    g.tB = tB;
    g.tC = g.tD = tC;
    return dgemm_batch(h, g, 1);
}

int spd_inverse(relu_qp_t h, int nb, int n, double* Km, double* Lm, double* Li, long long s, double* D, int ldd,
                long long sD, int* flag) {
    for (int b = 0; b < nb; ++b) RQ_CUDA(h, cudaMemsetAsync(Li + b * s, 0, sizeof(double) * n * n, h->stream));
    auto strided = [&](Gemm g) {
        g.sA = g.sB = g.sC = g.sD = s;
        return g;
    };
    for (int j = 0; j < n; j += NB) {   // K = L L^T, and the inverses of L's diagonal blocks in Li
        const int jb = (n - j < NB) ? n - j : NB, rest = n - j - jb;
        potrf_diag_kernel<<<nb, 256, 0, h->stream>>>(Km, s, n, j, jb, Lm, s, Li, s, flag);
        RQ_CUDA(h, cudaGetLastError());
        if (rest <= 0) break;
        const size_t d = (size_t)j * n + j, p = (size_t)(j + jb) * n + j;
        RQ_TRY(dgemm_batch(h, strided(gemm(false, true, rest, jb, jb, 1.0, Km + p, n, Li + d, n, 0.0, Lm + p, n)), nb));
        Gemm u = strided(gemm(false, true, rest, rest, jb, -1.0, Lm + p, n, Lm + p, n, 1.0, Km + p + jb, n));
        u.flags = G_LOWER;
        RQ_TRY(dgemm_batch(h, u, nb));
    }
    // L^{-1}: blocks of b rows doubled pair by pair, Li21 = -Li22 (L21 Li11); K's storage is scratch
    for (int b = NB; b < n; b *= 2) {
        const int pairs = ceil_div(n - b, 2 * b);
        const long long t = 2ll * b * (n + 1);
        const size_t o = (size_t)b * n;
        Gemm g = strided(gemm(false, false, b, b, b, 1.0, Lm + o, n, Li, n, 0.0, Km + o, n));
        g.nb2 = pairs;
        g.tA = g.tB = g.tC = g.tD = t;
        g.mtot = n - b;
        g.mstep = 2 * b;
        g.flags = G_KBEG_N;
        RQ_TRY(dgemm_batch(h, g, nb));
        Gemm q = strided(gemm(false, false, b, b, b, -1.0, Li + o + b, n, Km + o, n, 0.0, Li + o, n));
        q.nb2 = pairs;
        q.tA = q.tB = q.tC = q.tD = t;
        q.mtot = n - b;
        q.mstep = 2 * b;
        q.flags = G_KEND_M | G_KRAG;
        RQ_TRY(dgemm_batch(h, q, nb));
    }
    // D = L^{-T} L^{-1}
    Gemm g = strided(gemm(true, false, n, n, n, 1.0, Li, n, Li, n, 0.0, D, ldd));
    g.sC = g.sD = sD;
    g.flags = G_LOWER | G_MIRROR | G_KBEG_M;
    return dgemm_batch(h, g, nb);
}

namespace {

struct Scratch {
    relu_qp_t h;
    std::vector<void*> ptrs;
    ~Scratch() {
        for (void* p : ptrs) cudaFree(p);
    }
    template <typename T>
    int get(T** p, size_t count) {
        void* q = nullptr;
        cudaError_t e = cudaMalloc(&q, count * sizeof(T) + 16);
        if (e != cudaSuccess)
            return fail(h, RELU_QP_ERR_OOM, std::string("setup scratch: ") + cudaGetErrorString(e));
        ptrs.push_back(q);
        *p = static_cast<T*>(q);
        return RELU_QP_OK;
    }
};

}  // namespace

int make_check_matrices(relu_qp_t h, const double* dP, const double* dA) {
    const int n = h->n, m = h->m;
    const int ldp = (int)round_up(n, 4), ldt = (int)round_up(m > 0 ? m : 1, 4);
    to_f32_pad_kernel<<<grid1d((size_t)n * n), 256, 0, h->stream>>>(dP, h->P32, n, n, ldp);
    RQ_CUDA(h, cudaGetLastError());
    if (m > 0) {
        to_f32_pad_kernel<<<grid1d((size_t)m * n), 256, 0, h->stream>>>(dA, h->A32, m, n, ldp);
        RQ_CUDA(h, cudaGetLastError());
        dim3 g(ceil_div(n, 32), ceil_div(m, 32));
        transpose_f32_kernel<<<g, dim3(32, 8), 0, h->stream>>>(dA, h->At32, m, n, ldt);
        RQ_CUDA(h, cudaGetLastError());
    }
    return RELU_QP_OK;
}

int pack_bf16_layer(relu_qp_t h, int r, const double* X, const double* V) {
    BatchWork& w = h->bw;
    const size_t part = (size_t)w.Rpad * w.ldk;
    __nv_bfloat16* out = static_cast<__nv_bfloat16*>(w.WB) + (size_t)r * 3 * part;
    pack_bf16_layer_kernel<<<grid1d((size_t)h->R * w.ldk), 256, 0, h->stream>>>(X, V, h->n, h->m, w.nP,
                                                                                       w.ldk, part, out);
    RQ_CUDA(h, cudaGetLastError());
    return RELU_QP_OK;
}

int pack_bf16_check(relu_qp_t h, const double* dP, const double* dA) {
    BatchWork& w = h->bw;
    const size_t part = (size_t)w.npad * w.ldkc;
    pack_bf16_check_kernel<<<grid1d((size_t)(h->n + h->m) * w.ldkc), 256, 0, h->stream>>>(
        dP, dA, h->n, h->m, w.nP, w.n64, w.ldkc, part, static_cast<__nv_bfloat16*>(w.WCB));
    RQ_CUDA(h, cudaGetLastError());
    return RELU_QP_OK;
}

int build_bank(relu_qp_t h, const double* dP, const double* dA, const std::vector<double>& row_scale) {
    const int n = h->n, m = h->m, R = h->R, nr = h->nr;
    const size_t nn = (size_t)n * n;
    Scratch s{h, {}};
    // scratch of one entry: K, L, L^{-1} (reused for T and X where they fit), [D; AD], V
    const bool alias = m <= 2 * n;
    const size_t per = 3 * nn + (size_t)R * n + (size_t)R * m + (alias ? 0 : (size_t)R * n);
    // as many entries together as fit 4 GiB of scratch (at least one)
    const int ge = (int)std::max<size_t>(1, std::min<size_t>(nr, ((size_t)4 << 30) / (8 * per)));
    double *C = nullptr, *sA = nullptr, *f = nullptr, *W;
    int* flag;
    RQ_TRY(s.get(&W, per * ge));
    RQ_TRY(s.get(&flag, nr));
    RQ_CUDA(h, cudaMemsetAsync(flag, 0, sizeof(int) * nr, h->stream));
    if (m > 0) {
        // C = A^T diag(s) A
        RQ_TRY(s.get(&C, nn));
        RQ_TRY(s.get(&sA, (size_t)m * n));
        RQ_TRY(s.get(&f, (size_t)m));
        RQ_CUDA(h, cudaMemcpyAsync(f, row_scale.data(), sizeof(double) * m, cudaMemcpyHostToDevice, h->stream));
        scale_rows_kernel<<<grid1d((size_t)m * n), 256, 0, h->stream>>>(dA, f, sA, m, n);
        RQ_CUDA(h, cudaGetLastError());
        Gemm g = gemm(true, false, n, n, m, 1.0, dA, n, sA, n, 0.0, C, n);
        g.flags = G_LOWER | G_MIRROR;
        RQ_TRY(dgemm_batch(h, g, 1));
    }
    for (int r0 = 0; r0 < nr; r0 += ge) {
        const int nb = std::min(ge, nr - r0);
        const long long st = (long long)per;
        double *Km = W, *Lm = W + nn, *Li = W + 2 * nn, *DS = W + 3 * nn, *V = DS + (size_t)R * n,
               *X = alias ? W : V + (size_t)R * m;
        RhoList rho{};
        for (int z = 0; z < nb; ++z) rho.v[z] = h->bank[r0 + z];
        kkt_kernel<<<dim3(grid1d(nn), nb), 256, 0, h->stream>>>(dP, C, h->sigma, rho, n, Km, st);
        RQ_CUDA(h, cudaGetLastError());
        RQ_TRY(spd_inverse(h, nb, n, Km, Lm, Li, st, DS, n, st, flag + r0));
        if (m > 0) {
            double *AD = DS + nn, *T = alias ? W : X;   // (K and L, or X, are free now or still)
            Gemm g = gemm(false, true, n, m, n, 1.0, Li, n, dA, n, 0.0, T, m);
            g.sA = g.sC = g.sD = st;
            g.flags = G_KEND_M;
            RQ_TRY(dgemm_batch(h, g, nb));
            g = gemm(true, false, m, m, n, 1.0, T, m, T, m, 0.0, V + (size_t)n * m, m);
            g.sA = g.sB = g.sC = g.sD = st;
            g.flags = G_LOWER | G_MIRROR;
            RQ_TRY(dgemm_batch(h, g, nb));
            g = gemm(true, false, n, m, n, 1.0, Li, n, T, m, 0.0, V, m);
            g.sA = g.sB = g.sC = g.sD = st;
            g.flags = G_KBEG_M;
            RQ_TRY(dgemm_batch(h, g, nb));
            transpose_f64_kernel<<<dim3(ceil_div(m, 32), ceil_div(n, 32), nb), dim3(32, 8), 0, h->stream>>>(V, st, AD,
                                                                                                        st, n, m);
            RQ_CUDA(h, cudaGetLastError());
        }
        Gemm g = gemm(false, false, R, n, m, 0.0, V, m, sA, n, h->sigma, X, n);
        for (int z = 0; z < nb; ++z) g.alpha[z] = -rho.v[z];
        g.D = DS;
        g.sA = g.sC = g.sD = st;
        RQ_TRY(dgemm_batch(h, g, nb));
        for (int z = 0; z < nb; ++z) {
            rq::BankEntry& be = h->be[r0 + z];
            be.rho = rho.v[z];
            pack_layer_kernel<<<grid1d((size_t)R * (h->ldw + n)), 256, 0, h->stream>>>(
                X + z * st, V + z * st, DS + z * st, n, m, h->ldw, be.Wt, be.Bop, be.Wt64, be.Bop64);
            RQ_CUDA(h, cudaGetLastError());
            if (h->bw.cap > 0 && h->bw.prec == RELU_QP_PREC_BF16X3)
                RQ_TRY(pack_bf16_layer(h, r0 + z, X + z * st, V + z * st));
        }
    }
    std::vector<int> hflag(nr, 0);
    RQ_CUDA(h, cudaMemcpyAsync(hflag.data(), flag, sizeof(int) * nr, cudaMemcpyDeviceToHost, h->stream));
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    for (int r = 0; r < nr; ++r)
        if (hflag[r])
            return fail(h, RELU_QP_ERR_NOT_PD,
                        "Cholesky pivot <= 0 for rho = " + std::to_string(h->bank[r]) +
                            ": P + sigma I + A^T rho A is not positive definite");
    return RELU_QP_OK;
}

}  // namespace rq
