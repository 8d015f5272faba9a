// Dense, LQR-preconditioned condensing of a linear MPC problem (Sec. IV,
// "Dense Model-Predictive Control") in FP64 on the GPU.
//
// Plant x_{k+1} = A x_k + B u_k, controls u_k = -K x_k + du_k with the
// infinite-horizon LQR gain K as preconditioner, Abar = A - B K.  The
// decision vector is ytilde = [du_0; ...; du_{N-1}] (n = N nu) and the
// trajectory y = [u_0; x_1; u_1; x_2; ...; u_{N-1}; x_N] = S ytilde + M x0 with
//   u_k rows of S:     -K Abar^{k-1-j} B (j < k),  I (j = k),  0 (j > k)
//   x_{k+1} rows of S:  Abar^{k-j} B (j <= k),  0 (j > k)
//   u_k rows of M:     -K Abar^k,     x_{k+1} rows of M:  Abar^{k+1}.
// With H = blkdiag(R, Q, ..., R, Q_N) the QP is Hbar = S^T H S, gbar = S^T H M x0
// (so q = F x0 with F = S^T H M), and limits on u_k (and optionally x_{k+1})
// become rows of S with bounds shifted by the matching rows of M x0
// (l = l0 - E x0, u = u0 - E x0 with E = the rows of M).
//
// GPU formulation.  Powers: Z_j = [Abar^{j+1} | Abar^j B], doubled (Z_{j+s} = Abar^s Z_j
// for all j < s in one launch), and -K Z_j.  Hbar: S is block Toeplitz, so with T_a and
// U_a the x and u blocks at distance a (U_0 = I, U_a = -K T_{a-1})
//   Hbar(i, j) = sum_{a = 0}^{N-1-i} T_a^T Q T_{a+i-j} + U_a^T R U_{a+i-j}   (i >= j; Q_N in
// the last term), i.e. running sums along the block diagonals of one Gram matrix with
// nx + nu rows: 2 n^2 (nx + nu) flops where S^T H S takes 2 n^2 N (nx + nu), 4 ms at
// n = 800.  The gradient map the same way: its blocks are
//   F_j = (sum_{a = 0}^{N-1-j} V_a Abar^a) Abar^j,  V_a = T_a^T Q Abar - U_a^T R K.
//
// K: the Riccati iteration X <- Q + A^T X (A - B K(X)), K(X) = (R + B^T X B)^{-1} B^T X A,
// run until max|X+ - X| <= 1e-13 max(1, max|X+|).  Where Q >= 0 and R > 0 its iterates are
// first doubled (structure-preserving doubling, Chu, Fan, Lin and Wang 2004): H_k is the
// iterate after 2^k steps, so that 128 steps take 7 doublings; one plain step from the
// result, corrected by one Newton step, then has to meet the same test.  Everything else, and a doubling that does not
// get there, takes the plain iteration from X = Q, with its results and errors.
#include "common.h"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace rq {
namespace {

constexpr int kRiccatiMaxIter = 100000;
constexpr int kRiccatiCheckEvery = 16;
constexpr double kRiccatiTol = 1e-13;

int grid_for(size_t total) { return (int)std::max<size_t>(1, std::min<size_t>((total + 255) / 256, 16384)); }

// One element of the prediction matrices' blocks: right(k, i, t) = (Abar^k B)(i, t).
struct Blocks {
    const double *Z, *W, *K;   // Z: N blocks nx x nc, W = -K Z: N blocks nu x nc, nc = nx + nu
    int nx, nu, N;
    __device__ __forceinline__ double T(int a, int i, int t) const {
        return Z[((size_t)a * nx + i) * (nx + nu) + nx + t];
    }
    __device__ __forceinline__ double U(int a, int i, int t) const {
        return a == 0 ? (i == t ? 1.0 : 0.0) : W[((size_t)(a - 1) * nu + i) * (nx + nu) + nx + t];
    }
    __device__ __forceinline__ double Mx(int k, int i, int t) const { return Z[((size_t)k * nx + i) * (nx + nu) + t]; }
    __device__ __forceinline__ double Mu(int k, int i, int t) const {
        return k == 0 ? -K[(size_t)i * nx + t] : W[((size_t)(k - 1) * nu + i) * (nx + nu) + t];
    }
};

// Rows of S and M that are constraint rows: u rows (N nu), then x rows (N nx, with
// state limits).  A_con: rows x n, E: rows x nx.
__global__ void constraint_fill_kernel(Blocks b, int rows, double* __restrict__ Acon, double* __restrict__ E) {
    const int n = b.N * b.nu, w = n + b.nx;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)rows * w; e += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / w), c = (int)(e % w);
        const bool x = r >= n;
        const int q = x ? r - n : r, rb = x ? b.nx : b.nu, k = q / rb, i = q % rb;
        if (c >= n) {
            E[(size_t)r * b.nx + c - n] = x ? b.Mx(k, i, c - n) : b.Mu(k, i, c - n);
        } else {
            const int j = c / b.nu, t = c % b.nu;
            Acon[(size_t)r * n + c] = j > k ? 0.0 : x ? b.T(k - j, i, t) : b.U(k - j, i, t);
        }
    }
}

// TU (nc x n): column block a is [T_a; U_a].
__global__ void tu_fill_kernel(Blocks b, double* __restrict__ TU) {
    const int n = b.N * b.nu, nc = b.nx + b.nu;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)nc * n; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / n), c = (int)(e % n), a = c / b.nu, t = c % b.nu;
        TU[e] = i < b.nx ? b.T(a, i, t) : b.U(a, i - b.nx, t);
    }
}

// Hbar from the Gram matrices G (Q) and GN (Q_N; may be G): thread (d, r, c) runs down
// block diagonal d.  Term a of block (i, i - d), a = N - 1 - i the last one, is
// (G(a, a + d)(r, c) + G(a + d, a)(c, r)) / 2, which makes the result symmetric bit for bit.
__global__ void hbar_kernel(const double* __restrict__ G, const double* __restrict__ GN, int N, int nu,
                            double* __restrict__ P) {
    const int n = N * nu;
    const size_t total = (size_t)N * nu * nu;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(e % nu), r = (int)(e / nu % nu), d = (int)(e / ((size_t)nu * nu));
        double sum = 0.0;
#pragma unroll 4
        for (int a = 0; a < N - d; ++a) {
            const size_t o = ((size_t)a * nu + r) * n + (size_t)(a + d) * nu + c;
            const size_t t = ((size_t)(a + d) * nu + c) * n + (size_t)a * nu + r;
            const double last = sum + 0.5 * (GN[o] + GN[t]);
            sum += 0.5 * (G[o] + G[t]);
            const int i = N - 1 - a, j = i - d;
            P[((size_t)i * nu + r) * n + (size_t)j * nu + c] = last;
            P[((size_t)j * nu + c) * n + (size_t)i * nu + r] = last;
        }
    }
}

// S_j = sum_{a < N-1-j} Y_a + YN_{N-1-j} (N blocks nu x nx).
__global__ void prefix_kernel(const double* __restrict__ Y, const double* __restrict__ YN, int N, size_t blk,
                              double* __restrict__ S) {
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < blk; e += (size_t)gridDim.x * blockDim.x) {
        double sum = 0.0;
#pragma unroll 4
        for (int a = 0; a < N; ++a) {
            const double y = Y[(size_t)a * blk + e];
            S[(size_t)(N - 1 - a) * blk + e] = sum + YN[(size_t)a * blk + e];
            sum += y;
        }
    }
}

// Winv = (I + W)^{-1} (n x n, n <= kGaussMax) in one CTA: in-place Gauss-Jordan
// elimination with row pivoting in shared memory.  A thread keeps its column (j = lane +
// 32 c) while it walks down the rows, so an element costs two shared reads, an FMA and a
// store; rows are exchanged by name (piv) and moved once at the end.  Bound by the FP64
// pipe of one SM (n^3 FMAs at two a clock, 52 us at n = 60) and three barriers a step.
// (226 us a call at n = 60; 279 with a division per element for its row and column.)  A singular matrix
// leaves infinities or NaN, which the caller's convergence test sees.
constexpr int kGaussMax = 160;
constexpr int kGaussThreads = 512;

__global__ void __launch_bounds__(kGaussThreads) gauss_inverse_kernel(const double* __restrict__ W, int n,
                                                                      double* __restrict__ Winv) {
    extern __shared__ double gsm[];
    __shared__ double col[kGaussMax], row[kGaussMax];
    __shared__ int piv[kGaussMax], used[kGaussMax];   // step k's row; whether a row has been one
    __shared__ double s_inv;
    const int ld = n | 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kW = kGaussThreads / 32;
    for (int i = warp; i < n; i += kW)
        for (int j = lane; j < n; j += 32) gsm[i * ld + j] = W[(size_t)i * n + j] + (i == j ? 1.0 : 0.0);
    for (int i = tid; i < n; i += kGaussThreads) used[i] = 0;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (warp == 0) {
            // the largest element of column k among the rows not used yet (the first of equals)
            double best = -1.0;
            int at = n;
            for (int i = lane; i < n; i += 32) {
                const double v = used[i] ? -1.0 : fabs(gsm[i * ld + k]);
                if (v > best) {
                    best = v;
                    at = i;
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const double v = __shfl_xor_sync(0xffffffffu, best, o);
                const int a = __shfl_xor_sync(0xffffffffu, at, o);
                if (v > best || (v == best && a < at)) {
                    best = v;
                    at = a;
                }
            }
            if (at >= n) {   // only NaN left: any unused row
                at = 0;
                while (at < n - 1 && used[at]) ++at;
            }
            if (lane == 0) {
                piv[k] = at;
                used[at] = 1;
                s_inv = 1.0 / gsm[at * ld + k];
            }
        }
        __syncthreads();
        const int p = piv[k];
        const double inv = s_inv;
        // minus column k, and row p times the inverse pivot
        if (tid < kGaussThreads / 2) {
            for (int i = tid; i < n; i += kGaussThreads / 2) col[i] = -gsm[i * ld + k];
        } else {
            for (int j = tid - kGaussThreads / 2; j < n; j += kGaussThreads / 2) row[j] = j == k ? inv : gsm[p * ld + j] * inv;
        }
        __syncthreads();
        for (int j = lane; j < n; j += 32) {
            const double r = row[j];
            for (int i = warp; i < n; i += kW) {
                double* w = gsm + i * ld + j;
                *w = i == p ? r : j == k ? col[i] * inv : fma(col[i], r, *w);
            }
        }
        __syncthreads();
    }
    // step k worked on row piv[k] and column k: element (piv[i], j) is the inverse's (i, piv[j])
    for (int i = warp; i < n; i += kW)
        for (int j = lane; j < n; j += 32) Winv[(size_t)i * n + piv[j]] = gsm[piv[i] * ld + j];
}

// X <- (X + X^T) / 2 (n x n, rows of ld) and, with red, the convergence measures of a
// Riccati step: red[0] = max |X_new - X_old|, red[1] = max |X_new| (bits of non-negative doubles).
__global__ void sym_diff_kernel(double* __restrict__ Xn, const double* __restrict__ X, int n, int ld,
                                unsigned long long* red) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
        const int i = e / n, j = e % n;
        if (j < i) continue;
        const double v = 0.5 * (Xn[(size_t)i * ld + j] + Xn[(size_t)j * ld + i]);
        Xn[(size_t)i * ld + j] = v;
        Xn[(size_t)j * ld + i] = v;
        if (!red) continue;
        const double d = fmax(fabs(v - X[(size_t)i * ld + j]), fabs(v - X[(size_t)j * ld + i]));
        atomicMax(red, (unsigned long long)__double_as_longlong(d));
        atomicMax(red + 1, (unsigned long long)__double_as_longlong(fabs(v)));
    }
}

// out = a X + b Y
__global__ void combine_kernel(double a, const double* __restrict__ X, double b, const double* __restrict__ Y, size_t count,
                               double* __restrict__ out) {
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
        out[e] = a * X[e] + b * Y[e];
}

struct Ctx {
    relu_qp_s h;     // carries the stream, the error message and the allocations
    ~Ctx() {
        cudaStreamSynchronize(h.stream);
        for (void* p : h.allocs) cudaFree(p);
    }
    // uninitialised: everything below writes a buffer before reading it
    int raw(double** p, size_t count) {
        void* q = nullptr;
        RQ_CUDA(&h, cudaMalloc(&q, sizeof(double) * count));
        h.allocs.push_back(q);
        *p = static_cast<double*>(q);
        return RELU_QP_OK;
    }
};

// Buffers of the Riccati iteration, carved from the call's one allocation.
struct Riccati {
    int nx, nu;
    const double *A, *B, *Q, *R;
    double *X, *Xn, *BtX, *G, *K0, *S, *XA;
    double *W, *Wi, *AG, *AG2, *Z, *HZ;     // doubling (nx <= kGaussMax)
    unsigned long long* red;                // (max|X+ - X|, max|X+|) of up to kRiccatiCheckEvery steps
    int* flag;
};

// K (nu x nx) = (R + B^T X B)^{-1} B^T X A for the current X.
int gain(Ctx& c, const Riccati& r, double* K) {
    relu_qp_t h = &c.h;
    const int nx = r.nx, nu = r.nu;
    const size_t uu = (size_t)nu * nu;
    RQ_TRY(dgemm(h, true, false, nu, nx, nx, 1.0, r.B, nu, r.X, nx, 0.0, r.BtX, nx));        // B^T X
    RQ_CUDA(h, cudaMemcpyAsync(r.G, r.R, sizeof(double) * uu, cudaMemcpyDeviceToDevice, h->stream));
    RQ_TRY(dgemm(h, false, false, nu, nu, nx, 1.0, r.BtX, nx, r.B, nu, 1.0, r.G, nu));        // R + B^T X B
    RQ_TRY(dgemm(h, false, false, nu, nx, nx, 1.0, r.BtX, nx, r.A, nx, 0.0, r.K0, nx));       // B^T X A
    RQ_TRY(spd_inverse(h, 1, nu, r.G, r.S, r.S + uu, (long long)uu, r.S + 2 * uu, nu, (long long)uu, r.flag));
    return dgemm(h, false, false, nu, nx, nu, 1.0, r.S + 2 * uu, nu, r.K0, nx, 0.0, K, nx);
}

// X <- Q + A^T X (A - B K(X)); its change goes to red + 2 slot.
int riccati_step(Ctx& c, Riccati& r, double* K, int slot) {
    relu_qp_t h = &c.h;
    const int nx = r.nx, nu = r.nu;
    RQ_TRY(gain(c, r, K));
    RQ_CUDA(h, cudaMemcpyAsync(r.Xn, r.A, sizeof(double) * nx * nx, cudaMemcpyDeviceToDevice, h->stream));
    RQ_TRY(dgemm(h, false, false, nx, nx, nu, -1.0, r.B, nu, K, nx, 1.0, r.Xn, nx));           // A - B K
    RQ_TRY(dgemm(h, false, false, nx, nx, nx, 1.0, r.X, nx, r.Xn, nx, 0.0, r.XA, nx));          // X (A - B K)
    RQ_CUDA(h, cudaMemcpyAsync(r.Xn, r.Q, sizeof(double) * nx * nx, cudaMemcpyDeviceToDevice, h->stream));
    RQ_TRY(dgemm(h, true, false, nx, nx, nx, 1.0, r.A, nx, r.XA, nx, 1.0, r.Xn, nx));           // Q + A^T X (A - B K)
    sym_diff_kernel<<<grid_for((size_t)nx * nx), 256, 0, h->stream>>>(r.Xn, r.X, nx, nx, r.red + 2 * slot);
    RQ_CUDA(h, cudaGetLastError());
    std::swap(r.X, r.Xn);
    return RELU_QP_OK;
}

struct Change {
    double d, mx;
    bool finite() const { return std::isfinite(d) && std::isfinite(mx); }
    bool met() const { return finite() && d <= kRiccatiTol * std::max(1.0, mx); }
};

// The changes of `steps` steps and the Cholesky flag (one synchronisation).
int read_changes(Ctx& c, const Riccati& r, int steps, Change* out, int* flag) {
    relu_qp_t h = &c.h;
    unsigned long long w[2 * kRiccatiCheckEvery];
    RQ_CUDA(h, cudaMemcpyAsync(w, r.red, sizeof(w[0]) * 2 * steps, cudaMemcpyDeviceToHost, h->stream));
    RQ_CUDA(h, cudaMemcpyAsync(flag, r.flag, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    for (int s = 0; s < steps; ++s) {
        std::memcpy(&out[s].d, &w[2 * s], sizeof(double));
        std::memcpy(&out[s].mx, &w[2 * s + 1], sizeof(double));
    }
    return RELU_QP_OK;
}

int clear_changes(Ctx& c, const Riccati& r) {
    RQ_CUDA(&c.h, cudaMemsetAsync(r.red, 0, sizeof(unsigned long long) * 2 * kRiccatiCheckEvery, c.h.stream));
    return RELU_QP_OK;
}

// The iterate after 2^k steps for k = 1, 2, .. until it no longer changes; *ok = 0 when
// it does not settle within the plain iteration's 2^17 > kRiccatiMaxIter steps.  A_k and
// G_k sit side by side (AG, nx x 2 nx): with Z = (I + G_k H_k)^{-1} [A_k G_k],
//   A+ = A_k Z_A,  G+ = G_k + (A_k Z_G) A_k^T,  H+ = H_k + A_k^T H_k Z_A;
// A_0 = A, G_0 = B R^{-1} B^T, H_0 = Q.
int riccati_doubling(Ctx& c, Riccati& r, bool* ok, int* doublings) {
    relu_qp_t h = &c.h;
    const int nx = r.nx, nu = r.nu, w = 2 * nx;
    const size_t uu = (size_t)nu * nu, row = sizeof(double) * nx;
    *ok = false;
    RQ_TRY(clear_changes(c, r));
    RQ_CUDA(h, cudaMemsetAsync(r.flag, 0, sizeof(int), h->stream));
    RQ_CUDA(h, cudaMemcpyAsync(r.X, r.Q, sizeof(double) * nx * nx, cudaMemcpyDeviceToDevice, h->stream));
    RQ_CUDA(h, cudaMemcpy2DAsync(r.AG, 2 * row, r.A, row, row, nx, cudaMemcpyDeviceToDevice, h->stream));
    RQ_CUDA(h, cudaMemcpyAsync(r.G, r.R, sizeof(double) * uu, cudaMemcpyDeviceToDevice, h->stream));
    RQ_TRY(spd_inverse(h, 1, nu, r.G, r.S, r.S + uu, (long long)uu, r.S + 2 * uu, nu, (long long)uu, r.flag));
    RQ_TRY(dgemm(h, false, true, nu, nx, nu, 1.0, r.S + 2 * uu, nu, r.B, nu, 0.0, r.BtX, nx));   // R^{-1} B^T
    RQ_TRY(dgemm(h, false, false, nx, nx, nu, 1.0, r.B, nu, r.BtX, nx, 0.0, r.AG + nx, w));
    const size_t smem = sizeof(double) * nx * (nx | 1);
    RQ_CUDA(h, cudaFuncSetAttribute(gauss_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    constexpr int kMost = 17, kUnread = 5;   // (the first doublings are not waited for)
    static_assert(kMost <= 2 * kRiccatiCheckEvery, "one pair of words per doubling");
    for (int k = 0; k < kMost; ++k) {
        const int slot = k % kRiccatiCheckEvery;
        if (k == kRiccatiCheckEvery) RQ_TRY(clear_changes(c, r));
        RQ_TRY(dgemm(h, false, false, nx, nx, nx, 1.0, r.AG + nx, w, r.X, nx, 0.0, r.W, nx));
        gauss_inverse_kernel<<<1, kGaussThreads, smem, h->stream>>>(r.W, nx, r.Wi);
        RQ_CUDA(h, cudaGetLastError());
        RQ_TRY(dgemm(h, false, false, nx, w, nx, 1.0, r.Wi, nx, r.AG, w, 0.0, r.Z, w));
        RQ_TRY(dgemm(h, false, false, nx, w, nx, 1.0, r.AG, w, r.Z, w, 0.0, r.AG2, w));         // [A+, A_k Z_G]
        RQ_TRY(dgemm(h, false, false, nx, nx, nx, 1.0, r.X, nx, r.Z, w, 0.0, r.HZ, nx));
        RQ_CUDA(h, cudaMemcpyAsync(r.Xn, r.X, sizeof(double) * nx * nx, cudaMemcpyDeviceToDevice, h->stream));
        RQ_TRY(dgemm(h, true, false, nx, nx, nx, 1.0, r.AG, w, r.HZ, nx, 1.0, r.Xn, nx));
        // G+ over G_k, then beside A+
        RQ_TRY(dgemm(h, false, true, nx, nx, nx, 1.0, r.AG2 + nx, w, r.AG, w, 1.0, r.AG + nx, w));
        RQ_CUDA(h, cudaMemcpy2DAsync(r.AG2 + nx, 2 * row, r.AG + nx, 2 * row, row, nx, cudaMemcpyDeviceToDevice, h->stream));
        sym_diff_kernel<<<grid_for((size_t)nx * nx), 256, 0, h->stream>>>(r.AG2 + nx, r.AG2 + nx, nx, w, nullptr);
        sym_diff_kernel<<<grid_for((size_t)nx * nx), 256, 0, h->stream>>>(r.Xn, r.X, nx, nx, r.red + 2 * slot);
        RQ_CUDA(h, cudaGetLastError());
        std::swap(r.X, r.Xn);
        std::swap(r.AG, r.AG2);
        if (k + 1 < kUnread) continue;
        Change ch[kRiccatiCheckEvery];
        int fl = 0;
        RQ_TRY(read_changes(c, r, slot + 1, ch, &fl));
        if (fl || !ch[slot].finite()) return RELU_QP_OK;
        if (ch[slot].met()) {
            *ok = true;
            *doublings = k + 1;
            return RELU_QP_OK;
        }
    }
    return RELU_QP_OK;
}

// One Newton step on X = F(X) from a converged X: X + D with D = F(X) - X + P^T D P,
// P = A - B K(X), the sum over P's powers doubled.  The doubling's own rounding (the gain
// off by 1e-13, as much as the plain iteration's stop test leaves) falls to 1e-15, which
// the gradient map F needs: at the optimal gain its terms cancel to 1e-4 of their size.
int riccati_newton(Ctx& c, Riccati& r, int doublings, double* K) {
    relu_qp_t h = &c.h;
    const int nx = r.nx, nu = r.nu, g = grid_for((size_t)nx * nx);
    const size_t xx = (size_t)nx * nx;
    RQ_TRY(riccati_step(c, r, K, 0));        // r.X = F(X), r.Xn = X
    double *D = r.W, *T = r.HZ, *P = r.Z, *P2 = r.Z + xx;
    combine_kernel<<<g, 256, 0, h->stream>>>(1.0, r.X, -1.0, r.Xn, xx, D);
    RQ_CUDA(h, cudaGetLastError());
    RQ_CUDA(h, cudaMemcpyAsync(P, r.A, sizeof(double) * xx, cudaMemcpyDeviceToDevice, h->stream));
    RQ_TRY(dgemm(h, false, false, nx, nx, nu, -1.0, r.B, nu, K, nx, 1.0, P, nx));
    for (int k = 0; k < doublings; ++k) {
        RQ_TRY(dgemm(h, false, false, nx, nx, nx, 1.0, D, nx, P, nx, 0.0, T, nx));
        RQ_TRY(dgemm(h, true, false, nx, nx, nx, 1.0, P, nx, T, nx, 1.0, D, nx));
        if (k + 1 == doublings) break;
        RQ_TRY(dgemm(h, false, false, nx, nx, nx, 1.0, P, nx, P, nx, 0.0, P2, nx));
        std::swap(P, P2);
    }
    sym_diff_kernel<<<g, 256, 0, h->stream>>>(D, D, nx, nx, nullptr);
    combine_kernel<<<g, 256, 0, h->stream>>>(1.0, r.Xn, 1.0, D, xx, r.X);
    RQ_CUDA(h, cudaGetLastError());
    return RELU_QP_OK;
}

bool symmetric(const double* M, int n) {
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < i; ++j)
            if (M[(size_t)i * n + j] != M[(size_t)j * n + i]) return false;
    return true;
}

// Symmetric and positive definite (a Cholesky factorisation exists).
bool positive_definite(const double* M, int n) {
    if (!symmetric(M, n)) return false;
    std::vector<double> a(M, M + (size_t)n * n);
    for (int k = 0; k < n; ++k) {
        double d = a[(size_t)k * n + k];
        for (int t = 0; t < k; ++t) d -= a[(size_t)k * n + t] * a[(size_t)k * n + t];
        if (!(d > 0.0)) return false;
        d = std::sqrt(d);
        a[(size_t)k * n + k] = d;
        for (int i = k + 1; i < n; ++i) {
            double v = a[(size_t)i * n + k];
            for (int t = 0; t < k; ++t) v -= a[(size_t)i * n + t] * a[(size_t)k * n + t];
            a[(size_t)i * n + k] = v / d;
        }
    }
    return true;
}

// Symmetric positive semidefinite as far as that is plain: diagonal with no negative
// entry, or positive definite.
bool semidefinite(const double* M, int n) {
    bool diagonal = true;
    for (int i = 0; i < n && diagonal; ++i)
        for (int j = 0; j < n && diagonal; ++j)
            diagonal = i == j ? M[(size_t)i * n + j] >= 0.0 : M[(size_t)i * n + j] == 0.0;
    return diagonal || positive_definite(M, n);
}

int lqr_gain(Ctx& c, Riccati& r, bool doubling, double* K) {
    relu_qp_t h = &c.h;
    const int nx = r.nx;
    bool converged = false;
    if (doubling) {
        int doublings = 0;
        RQ_TRY(riccati_doubling(c, r, &converged, &doublings));
        if (converged) {   // one plain step has to meet the plain iteration's own test
            Change ch;
            int fl = 0;
            RQ_TRY(riccati_newton(c, r, doublings, K));
            RQ_TRY(clear_changes(c, r));
            RQ_TRY(riccati_step(c, r, K, 0));
            RQ_TRY(read_changes(c, r, 1, &ch, &fl));
            converged = !fl && ch.met();
        }
    }
    if (!converged) {
        RQ_CUDA(h, cudaMemsetAsync(r.flag, 0, sizeof(int), h->stream));
        RQ_CUDA(h, cudaMemcpyAsync(r.X, r.Q, sizeof(double) * nx * nx, cudaMemcpyDeviceToDevice, h->stream));
    }
    for (int it = 0; it < kRiccatiMaxIter && !converged; it += kRiccatiCheckEvery) {
        RQ_TRY(clear_changes(c, r));
        for (int s = 0; s < kRiccatiCheckEvery; ++s) RQ_TRY(riccati_step(c, r, K, s));
        Change ch[kRiccatiCheckEvery];
        int fl = 0;
        RQ_TRY(read_changes(c, r, kRiccatiCheckEvery, ch, &fl));
        // a diverging X (unstabilizable plant) also breaks the Cholesky of R + B^T X B:
        // report the divergence first
        for (const Change& v : ch) {
            if (!v.finite())
                return fail(h, RELU_QP_ERR_INVALID, "condense: the Riccati iteration diverged ((A, B) not stabilizable?)");
            if (v.met()) converged = true;
        }
        if (fl) return fail(h, RELU_QP_ERR_NOT_PD, "condense: R + B^T X B is not positive definite");
    }
    if (!converged)
        return fail(h, RELU_QP_ERR_INVALID, "condense: the Riccati iteration did not converge");
    return gain(c, r, K);
}

int condense(Ctx& c, int nx, int nu, int N, const double* hA, const double* hB, const double* hQ, const double* hR,
             const double* hQN, bool state, const double* hK, int precondition, double* oP, double* oA, double* oF,
             double* oE, double* oK) {
    relu_qp_t h = &c.h;
    const int n = N * nu, nc = nx + nu, rows = n + (state ? N * nx : 0);
    const size_t xx = (size_t)nx * nx, xu = (size_t)nx * nu, uu = (size_t)nu * nu, nn = (size_t)n * n;
    const bool lqr = !hK && precondition, ownQN = hQN && std::memcmp(hQN, hQ, sizeof(double) * xx) != 0;
    const bool doubling = lqr && nx <= kGaussMax && nu <= kGaussMax && positive_definite(hR, nu) && semidefinite(hQ, nx);
    // one allocation: inputs (as on the host), the iteration's buffers, the products
    double *in, *Z, *W, *TU, *HTU, *HTN, *G, *GN, *P, *F, *Acon, *E, *HM, *V, *VN, *Y, *YN, *S;
    Riccati r{};
    size_t total = 0;
    auto lay = [&](double* base) {
        size_t o = 0;
        auto get = [&](double*& p, size_t count) {
            p = base ? base + o : nullptr;
            o += round_up(count, 2);
        };
        get(in, 3 * xx + 2 * xu + uu);
        if (lqr) {
            double* words;
            get(r.X, xx);
            get(r.Xn, xx);
            get(r.XA, xx);
            get(r.BtX, xu);
            get(r.K0, xu);
            get(r.G, uu);
            get(r.S, 3 * uu);
            get(words, 2 * kRiccatiCheckEvery + 1);
            r.red = reinterpret_cast<unsigned long long*>(words);
            r.flag = reinterpret_cast<int*>(words ? words + 2 * kRiccatiCheckEvery : nullptr);
            if (doubling) {
                get(r.W, xx);
                get(r.Wi, xx);
                get(r.HZ, xx);
                get(r.AG, 2 * xx);
                get(r.AG2, 2 * xx);
                get(r.Z, 2 * xx);
            }
        }
        get(Z, (size_t)N * nx * nc);
        get(W, (size_t)N * nu * nc);
        get(TU, (size_t)nc * n);
        get(HTU, (size_t)nc * n);
        get(HTN, ownQN ? (size_t)nc * n : 0);
        get(G, nn);
        get(GN, ownQN ? nn : 0);
        get(P, nn);
        get(Acon, (size_t)rows * n);
        get(E, (size_t)rows * nx);
        get(HM, 2 * (size_t)nc * nx);
        for (double** p : {&V, &Y, &S, &F}) get(*p, (size_t)n * nx);
        for (double** p : {&VN, &YN}) get(*p, ownQN ? (size_t)n * nx : 0);
        return o;
    };
    total = lay(nullptr);
    double* base;
    RQ_TRY(c.raw(&base, total));
    lay(base);
    std::vector<double> host(3 * xx + 2 * xu + uu, 0.0);   // A, B, Q, Q_N, R, K (zero: no preconditioning)
    std::memcpy(host.data(), hA, sizeof(double) * xx);
    std::memcpy(host.data() + xx, hB, sizeof(double) * xu);
    std::memcpy(host.data() + xx + xu, hQ, sizeof(double) * xx);
    std::memcpy(host.data() + 2 * xx + xu, hQN ? hQN : hQ, sizeof(double) * xx);
    std::memcpy(host.data() + 3 * xx + xu, hR, sizeof(double) * uu);
    if (hK) std::memcpy(host.data() + 3 * xx + xu + uu, hK, sizeof(double) * xu);
    RQ_CUDA(h, cudaMemcpyAsync(in, host.data(), sizeof(double) * host.size(), cudaMemcpyHostToDevice, h->stream));
    double *A = in, *B = A + xx, *Q = B + xu, *QN = Q + xx, *R = QN + xx, *K = R + uu;
    if (lqr) {
        r.nx = nx;
        r.nu = nu;
        r.A = A;
        r.B = B;
        r.Q = Q;
        r.R = R;
        RQ_TRY(lqr_gain(c, r, doubling, K));
    }
    // Z_0 = [A - B K | B], doubled; W = -K Z
    const size_t zb = (size_t)nx * nc, wb = (size_t)nu * nc;
    RQ_CUDA(h, cudaMemcpy2DAsync(Z, sizeof(double) * nc, A, sizeof(double) * nx, sizeof(double) * nx, nx,
                                 cudaMemcpyDeviceToDevice, h->stream));
    RQ_CUDA(h, cudaMemcpy2DAsync(Z + nx, sizeof(double) * nc, B, sizeof(double) * nu, sizeof(double) * nu, nx,
                                 cudaMemcpyDeviceToDevice, h->stream));
    RQ_TRY(dgemm(h, false, false, nx, nx, nu, -1.0, B, nu, K, nx, 1.0, Z, nc));
    for (int s = 1; s < N; s *= 2)
        RQ_TRY(dgemm_strided(h, false, false, nx, nc, nx, 1.0, Z + (s - 1) * zb, nc, 0, Z, nc, (long long)zb, Z + s * zb,
                             nc, (long long)zb, std::min(s, N - s)));
    RQ_TRY(dgemm_strided(h, false, false, nu, nc, nx, -1.0, K, nx, 0, Z, nc, (long long)zb, W, nc, (long long)wb, N));
    const Blocks blocks{Z, W, K, nx, nu, N};
    constraint_fill_kernel<<<grid_for((size_t)rows * (n + nx)), 256, 0, h->stream>>>(blocks, rows, Acon, E);
    tu_fill_kernel<<<grid_for((size_t)nc * n), 256, 0, h->stream>>>(blocks, TU);
    RQ_CUDA(h, cudaGetLastError());
    // Gram matrices and Hbar
    const size_t ur = (size_t)nx * n;   // first u row of TU
    RQ_TRY(dgemm(h, false, false, nx, n, nx, 1.0, Q, nx, TU, n, 0.0, HTU, n));
    RQ_TRY(dgemm(h, false, false, nu, n, nu, 1.0, R, nu, TU + ur, n, 0.0, HTU + ur, n));
    RQ_TRY(dgemm(h, true, false, n, n, nc, 1.0, TU, n, HTU, n, 0.0, G, n));
    if (ownQN) {
        RQ_TRY(dgemm(h, false, false, nx, n, nx, 1.0, QN, nx, TU, n, 0.0, HTN, n));
        RQ_CUDA(h, cudaMemcpyAsync(HTN + ur, HTU + ur, sizeof(double) * nu * n, cudaMemcpyDeviceToDevice, h->stream));
        RQ_TRY(dgemm(h, true, false, n, n, nc, 1.0, TU, n, HTN, n, 0.0, GN, n));
    }
    hbar_kernel<<<grid_for((size_t)n * nu), 256, 0, h->stream>>>(G, ownQN ? GN : G, N, nu, P);
    RQ_CUDA(h, cudaGetLastError());
    // F: V = TU^T [Q Abar; -R K], Y_a = V_a Abar^a, running sums, times Abar^j
    auto gradient = [&](const double* q, double* hm, double* v, double* y) -> int {
        RQ_TRY(dgemm(h, false, false, nx, nx, nx, 1.0, q, nx, Z, nc, 0.0, hm, nx));
        RQ_TRY(dgemm(h, false, false, nu, nx, nu, -1.0, R, nu, K, nx, 0.0, hm + xx, nx));
        RQ_TRY(dgemm(h, true, false, n, nx, nc, 1.0, TU, n, hm, nx, 0.0, v, nx));
        RQ_CUDA(h, cudaMemcpyAsync(y, v, sizeof(double) * xu, cudaMemcpyDeviceToDevice, h->stream));
        return dgemm_strided(h, false, false, nu, nx, nx, 1.0, v + xu, nx, (long long)xu, Z, nc, (long long)zb, y + xu, nx,
                             (long long)xu, N - 1);
    };
    RQ_TRY(gradient(Q, HM, V, Y));
    if (ownQN) RQ_TRY(gradient(QN, HM + (size_t)nc * nx, VN, YN));
    prefix_kernel<<<grid_for(xu), 256, 0, h->stream>>>(Y, ownQN ? YN : Y, N, xu, S);
    RQ_CUDA(h, cudaGetLastError());
    RQ_CUDA(h, cudaMemcpyAsync(F, S, sizeof(double) * xu, cudaMemcpyDeviceToDevice, h->stream));
    RQ_TRY(dgemm_strided(h, false, false, nu, nx, nx, 1.0, S + xu, nx, (long long)xu, Z, nc, (long long)zb, F + xu, nx,
                         (long long)xu, N - 1));
    RQ_CUDA(h, cudaMemcpyAsync(oP, P, sizeof(double) * nn, cudaMemcpyDeviceToHost, h->stream));
    RQ_CUDA(h, cudaMemcpyAsync(oF, F, sizeof(double) * n * nx, cudaMemcpyDeviceToHost, h->stream));
    RQ_CUDA(h, cudaMemcpyAsync(oA, Acon, sizeof(double) * rows * n, cudaMemcpyDeviceToHost, h->stream));
    RQ_CUDA(h, cudaMemcpyAsync(oE, E, sizeof(double) * rows * nx, cudaMemcpyDeviceToHost, h->stream));
    if (oK) RQ_CUDA(h, cudaMemcpyAsync(oK, K, sizeof(double) * xu, cudaMemcpyDeviceToHost, h->stream));
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    return RELU_QP_OK;
}

}  // namespace

int condense_mpc(int nx, int nu, int N, const double* A, const double* B, const double* Q, const double* R,
                 const double* QN, bool state_rows, const double* K, int precondition, void* stream, double* P,
                 double* Acon, double* F, double* E, double* K_out, std::string* err) {
    Ctx c;
    c.h.stream = (cudaStream_t)stream;
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&c.h.num_sms, cudaDevAttrMultiProcessorCount, dev);
    const int rc = condense(c, nx, nu, N, A, B, Q, R, QN, state_rows, K, precondition, P, Acon, F, E, K_out);
    if (rc != RELU_QP_OK) *err = c.h.err;
    return rc;
}

}  // namespace rq
