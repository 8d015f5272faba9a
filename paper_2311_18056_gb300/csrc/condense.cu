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
// GPU formulation.  Powers: Z_j = [Abar^{j+1} | Abar^j B], one after the other, and -K Z_j.
// (Doubled, Z_{j+s} = Abar^s Z_j for all j < s, they take 0.05 ms instead of 0.3 at nx = 60,
// N = 40, but every doubling doubles the rounding that is there: 1.1e-14 of P and 1.2e-14 of F at
// spectral radius 1.2 and N = 60 without preconditioning, against 2.4e-15 and 7e-16.)  Hbar: S is block Toeplitz, so with T_a and
// U_a the x and u blocks at distance a (U_0 = I, U_a = -K T_{a-1})
//   Hbar(i, j) = sum_{a = 0}^{N-1-i} T_a^T Q T_{a+i-j} + U_a^T R U_{a+i-j}   (i >= j; Q_N in
// the last term), i.e. running sums along the block diagonals of one Gram matrix with
// nx + nu rows: 2 n^2 (nx + nu) flops where S^T H S takes 2 n^2 N (nx + nu), 4 ms at
// n = 800.  The gradient map the same way: its blocks are
//   F_j = (sum_{a = 0}^{N-1-j} V_a Abar^a) Abar^j,  V_a = T_a^T Q Abar - U_a^T R K.
//
// K: the Riccati iteration X <- Q + A^T X (A - B K(X)), K(X) = (R + B^T X B)^{-1} B^T X A,
// run until max|X+ - X| <= 1e-13 max(1, max|X+|), 16 steps between the host's looks.  Up to
// kOneMaxX states the 16 steps are one launch of one cluster (riccati_kernel).
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

// `steps` steps of the Riccati iteration (X in X[0], then X[1], ..) by one cluster of 16
// CTAs, or (steps = 0) K of X[0] alone.  The matrices stay in L2; a thread forms one entry
// of a product, with a hardware cluster barrier between products.  R + B^T X B is inverted
// by every CTA for itself (Gauss-Jordan, one barrier a step, the next pivot's reciprocal
// taken by the thread that has it); a pivot <= 0 sets *flag and counts as 1, as in the
// blocked Cholesky.  Bound by the FP64 pipes of 16 SMs (0.7 M FMAs a step at nx = 60,
// nu = 20: 11 us), the inverse's 20 dependent steps and eight barriers: 51 us a step with a
// product's entries dealt out CTA by CTA.  A launch per product took 75 us.
constexpr int kOneMaxX = 96, kOneMaxU = 48, kOneCtas = 16, kOneThreads = 256;

struct OneArgs {
    int nx, nu, steps;
    const double *A, *B, *Q, *R;
    double *X[2], *BtX, *G, *K0, *K, *T, *XA;
    unsigned long long* red;
    int* flag;
};

__device__ __forceinline__ void cluster_barrier_hw() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// sum_k a(k) b(k), loads past the L1 (other CTAs write these matrices), in k order
template <class FA, class FB>
__device__ __forceinline__ double dot_k(int n, FA a, FB b) {
    double acc = 0.0;
    int k = 0;
    constexpr int U = 12;   // loads in flight: an L2 trip is some 700 clocks
    for (; k + U <= n; k += U) {
        double u[U], v[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
            u[t] = a(k + t);
            v[t] = b(k + t);
        }
#pragma unroll
        for (int t = 0; t < U; ++t) acc = fma(u[t], v[t], acc);
    }
    for (; k < n; ++k) acc = fma(a(k), b(k), acc);
    return acc;
}

__global__ void __launch_bounds__(kOneThreads) riccati_kernel(const OneArgs g) {
    __shared__ double s_g[2][kOneMaxU][kOneMaxU + 1];
    __shared__ double s_inv[2];
    // (a product's entries go to the CTAs warp by warp, so that a small one uses every SM)
    const int nx = g.nx, nu = g.nu, tid = threadIdx.x, gt = ((tid >> 5) * kOneCtas + blockIdx.x) * 32 + (tid & 31);
    constexpr int NT = kOneCtas * kOneThreads;
    for (int s = 0; s < (g.steps > 0 ? g.steps : 1); ++s) {
        const double* X = g.X[s & 1];
        double* Xn = g.X[(s & 1) ^ 1];
        // B^T X
        for (int o = gt; o < nu * nx; o += NT) {
            const int i = o / nx, j = o % nx;
            g.BtX[o] = dot_k(nx, [&](int k) { return __ldg(g.B + (size_t)k * nu + i); },
                             [&](int k) { return __ldcg(X + (size_t)k * nx + j); });
        }
        cluster_barrier_hw();
        // B^T X A and R + B^T X B
        for (int o = gt; o < nu * (nx + nu); o += NT) {
            const int i = o / (nx + nu), j = o % (nx + nu);
            const double v = dot_k(nx, [&](int k) { return __ldcg(g.BtX + (size_t)i * nx + k); },
                                   [&](int k) { return j < nx ? __ldg(g.A + (size_t)k * nx + j) : __ldg(g.B + (size_t)k * nu + j - nx); });
            if (j < nx) g.K0[(size_t)i * nx + j] = v;
            else g.G[(size_t)i * nu + j - nx] = __ldg(g.R + (size_t)i * nu + j - nx) + v;
        }
        cluster_barrier_hw();
        // the inverse of its lower triangle's symmetric matrix, in every CTA
        auto pivot = [&](double d) {
            if (!(d > 0.0)) {
                if (blockIdx.x == 0) atomicExch(g.flag, 1);
                d = 1.0;
            }
            return 1.0 / d;
        };
        for (int o = tid; o < nu * nu; o += kOneThreads) {
            const int i = o / nu, j = o % nu;
            const double v = __ldcg(g.G + (i >= j ? (size_t)i * nu + j : (size_t)j * nu + i));
            s_g[0][i][j] = v;
            if (o == 0) s_inv[0] = pivot(v);
        }
        __syncthreads();
        for (int k = 0; k < nu; ++k) {
            const double(*a)[kOneMaxU + 1] = s_g[k & 1];
            double(*b)[kOneMaxU + 1] = s_g[(k & 1) ^ 1];
            const double inv = s_inv[k & 1];
            for (int o = tid; o < nu * nu; o += kOneThreads) {
                const int i = o / nu, j = o % nu;
                double v;
                if (i == k) v = j == k ? inv : a[k][j] * inv;
                else if (j == k) v = -a[i][k] * inv;
                else v = fma(-a[i][k] * inv, a[k][j], a[i][j]);
                b[i][j] = v;
                if (i == k + 1 && j == k + 1) s_inv[(k & 1) ^ 1] = pivot(v);
            }
            __syncthreads();
        }
        const double(*gi)[kOneMaxU + 1] = s_g[nu & 1];
        for (int o = gt; o < nu * nx; o += NT) {
            const int i = o / nx, j = o % nx;
            g.K[o] = dot_k(nu, [&](int k) { return gi[i][k]; }, [&](int k) { return __ldcg(g.K0 + (size_t)k * nx + j); });
        }
        if (g.steps == 0) break;
        cluster_barrier_hw();
        // A - B K, X (A - B K), Q + A^T X (A - B K)
        for (int o = gt; o < nx * nx; o += NT) {
            const int i = o / nx, j = o % nx;
            g.T[o] = __ldg(g.A + o) - dot_k(nu, [&](int k) { return __ldg(g.B + (size_t)i * nu + k); },
                                            [&](int k) { return __ldcg(g.K + (size_t)k * nx + j); });
        }
        cluster_barrier_hw();
        for (int o = gt; o < nx * nx; o += NT) {
            const int i = o / nx, j = o % nx;
            g.XA[o] = dot_k(nx, [&](int k) { return __ldcg(X + (size_t)i * nx + k); },
                            [&](int k) { return __ldcg(g.T + (size_t)k * nx + j); });
        }
        cluster_barrier_hw();
        for (int o = gt; o < nx * nx; o += NT) {
            const int i = o / nx, j = o % nx;
            g.T[o] = __ldg(g.Q + o) + dot_k(nx, [&](int k) { return __ldg(g.A + (size_t)k * nx + i); },
                                            [&](int k) { return __ldcg(g.XA + (size_t)k * nx + j); });
        }
        cluster_barrier_hw();
        // symmetrised, and its change (as sym_diff_kernel)
        unsigned long long d = 0, mx = 0;
        for (int o = gt; o < nx * nx; o += NT) {
            const int i = o / nx, j = o % nx;
            const double v = 0.5 * (i <= j ? __ldcg(g.T + o) + __ldcg(g.T + (size_t)j * nx + i)
                                           : __ldcg(g.T + (size_t)j * nx + i) + __ldcg(g.T + o));
            Xn[o] = v;
            d = max(d, (unsigned long long)__double_as_longlong(fabs(v - __ldcg(X + o))));
            mx = max(mx, (unsigned long long)__double_as_longlong(fabs(v)));
        }
        for (int o = 16; o > 0; o >>= 1) {
            d = max(d, __shfl_xor_sync(0xffffffffu, d, o));
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if ((tid & 31) == 0) {
            atomicMax(g.red + 2 * s, d);
            atomicMax(g.red + 2 * s + 1, mx);
        }
        cluster_barrier_hw();
    }
    cluster_barrier_hw();
}

// X <- (X + X^T) / 2 (n x n) and the convergence measures of the Riccati step:
// red[0] = max |X_new - X_old|, red[1] = max |X_new| (bits of non-negative doubles).
__global__ void sym_diff_kernel(double* __restrict__ Xn, const double* __restrict__ X, int n,
                                unsigned long long* red) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
        const int i = e / n, j = e % n;
        if (j < i) continue;
        const double v = 0.5 * (Xn[(size_t)i * n + j] + Xn[(size_t)j * n + i]);
        Xn[(size_t)i * n + j] = v;
        Xn[(size_t)j * n + i] = v;
        const double d = fmax(fabs(v - X[(size_t)i * n + j]), fabs(v - X[(size_t)j * n + i]));
        atomicMax(red, (unsigned long long)__double_as_longlong(d));
        atomicMax(red + 1, (unsigned long long)__double_as_longlong(fabs(v)));
    }
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
    sym_diff_kernel<<<grid_for((size_t)nx * nx), 256, 0, h->stream>>>(r.Xn, r.X, nx, r.red + 2 * slot);
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

// riccati_kernel: `steps` steps from r.X, or (0) K(r.X); RELU_QP_ERR_UNSUPPORTED when the
// cluster cannot be launched here.
int riccati_cluster(Ctx& c, Riccati& r, int steps, double* K) {
    relu_qp_t h = &c.h;
    if (r.nx > kOneMaxX || r.nu > kOneMaxU) return RELU_QP_ERR_UNSUPPORTED;
    OneArgs g{r.nx, r.nu, steps, r.A, r.B, r.Q, r.R, {r.X, r.Xn}, r.BtX, r.G, r.K0, K, r.S, r.XA, r.red, r.flag};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kOneCtas);
    cfg.blockDim = dim3(kOneThreads);
    cfg.stream = h->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kOneCtas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(riccati_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaLaunchKernelEx(&cfg, riccati_kernel, g) != cudaSuccess) {
        cudaGetLastError();
        return RELU_QP_ERR_UNSUPPORTED;
    }
    if (steps & 1) std::swap(r.X, r.Xn);
    return RELU_QP_OK;
}

int lqr_gain(Ctx& c, Riccati& r, double* K) {
    relu_qp_t h = &c.h;
    bool converged = false, one = true;
    RQ_CUDA(h, cudaMemsetAsync(r.flag, 0, sizeof(int), h->stream));
    RQ_CUDA(h, cudaMemcpyAsync(r.X, r.Q, sizeof(double) * r.nx * r.nx, cudaMemcpyDeviceToDevice, h->stream));
    for (int it = 0; it < kRiccatiMaxIter && !converged; it += kRiccatiCheckEvery) {
        RQ_TRY(clear_changes(c, r));
        one = one && riccati_cluster(c, r, kRiccatiCheckEvery, K) == RELU_QP_OK;
        for (int s = 0; s < kRiccatiCheckEvery && !one; ++s) RQ_TRY(riccati_step(c, r, K, s));
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
    return one && riccati_cluster(c, r, 0, K) == RELU_QP_OK ? RELU_QP_OK : gain(c, r, K);
}

int condense(Ctx& c, int nx, int nu, int N, const double* hA, const double* hB, const double* hQ, const double* hR,
             const double* hQN, bool state, const double* hK, int precondition, double* oP, double* oA, double* oF,
             double* oE, double* oK) {
    relu_qp_t h = &c.h;
    const int n = N * nu, nc = nx + nu, rows = n + (state ? N * nx : 0);
    const size_t xx = (size_t)nx * nx, xu = (size_t)nx * nu, uu = (size_t)nu * nu, nn = (size_t)n * n;
    const bool lqr = !hK && precondition, ownQN = hQN && std::memcmp(hQN, hQ, sizeof(double) * xx) != 0;
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
            get(r.S, std::max(3 * uu, xx));   // spd_inverse's scratch, or the cluster's X (A - B K)
            get(words, 2 * kRiccatiCheckEvery + 1);
            r.red = reinterpret_cast<unsigned long long*>(words);
            r.flag = reinterpret_cast<int*>(words ? words + 2 * kRiccatiCheckEvery : nullptr);
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
        RQ_TRY(lqr_gain(c, r, K));
    }
    // Z_0 = [A - B K | B], Z_j = Abar Z_{j-1}; W = -K Z
    const size_t zb = (size_t)nx * nc, wb = (size_t)nu * nc;
    RQ_CUDA(h, cudaMemcpy2DAsync(Z, sizeof(double) * nc, A, sizeof(double) * nx, sizeof(double) * nx, nx,
                                 cudaMemcpyDeviceToDevice, h->stream));
    RQ_CUDA(h, cudaMemcpy2DAsync(Z + nx, sizeof(double) * nc, B, sizeof(double) * nu, sizeof(double) * nu, nx,
                                 cudaMemcpyDeviceToDevice, h->stream));
    RQ_TRY(dgemm(h, false, false, nx, nx, nu, -1.0, B, nu, K, nx, 1.0, Z, nc));
    for (int j = 1; j < N; ++j)
        RQ_TRY(dgemm(h, false, false, nx, nc, nx, 1.0, Z, nc, Z + (j - 1) * zb, nc, 0.0, Z + j * zb, nc));
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
