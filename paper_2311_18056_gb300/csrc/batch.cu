// Batched online stage of Algorithm 1: B QPs sharing P and A (so every W_rho
// of the bank) with their own q, l, u, warm start and penalty index.
//
// One chunk = check_interval layers (25 by default, Sec. III-C).  Every layer
// is one GEMM over the active slots with the element-wise layer in its
// epilogue (batch.h).  At the end of a chunk the residuals of Eqs. primal and
// dual are formed per QP, the decision kernel applies the stop test and the
// penalty rule of Eq. rho_update (nearest bank entry, Sec. III-C), converged
// QPs leave the batch, and the rest are regrouped so that a 128-slot tile
// holds QPs of one bank entry only.  The host reads one counter per chunk.
//
// Backends: FP32 on the CUDA cores (this file) and BF16 hi+lo split operands
// on the tcgen05 tensor cores (batch_tc.cu) with FP32 accumulation.  In the
// split form the first layer of a chunk is an accurate (3-way split) product
// that stores c = Wt s_ref + b, and the other layers apply the 2-way split
// only to the increment: t = c + Wt (s - s_ref).
#include "batch.h"
#include "grid_sync.h"
#include "tile32.h"

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <thread>
#include <new>

namespace rq {

namespace {

inline int __float_as_int_host(float f) {
    int i;
    std::memcpy(&i, &f, sizeof(i));
    return i;
}

struct W32Ptrs {
    const float* w[RQ_MAX_RHO];
};

// Problem updates: up to kMaps products of one X (M x K) with different W (N x K) in one
// launch, C[i][j'] = alpha * sum_k X[i][k] W[j][k] + (off ? off[j] : 0), with a second result
// C2 of the same sums and its own offsets (l and u), and j' = j, or j + shift from
// j = split on (rows of a layer into its padded layout).  Every sum runs over k in order.
// One update is 3 + n_rho maps of a few microseconds each (at 250 QPs, nx = 70: seven
// launches, 173 us, when each was a kernel of 16 to 25 tiles): together they fill the SMs.
// Rows and columns in 64 x 64 tiles, 4 x 4 outputs a thread; the next 16 columns of k are
// loaded into registers while the current ones are multiplied.
constexpr int kMaps = RQ_MAX_RHO + 4;

struct MapTask {
    const float* W;
    const float *off, *off2;
    float *C, *C2;
    int N, ldw, ldc, split, shift, tile0;   // tile0: first column tile of the launch
    float alpha;
};

struct MapTasks {
    MapTask t[kMaps];
    int count;
};

__global__ void __launch_bounds__(256) map_kernel(int M, int K, const float* __restrict__ X, int ldx, const MapTasks ts) {
    __shared__ float Xs[16][64 + 4];
    __shared__ float Ws[16][64 + 4];
    int a = 0;
    while (a + 1 < ts.count && (int)blockIdx.x >= ts.t[a + 1].tile0) ++a;
    const MapTask& T = ts.t[a];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int i0 = blockIdx.y * 64, j0 = (blockIdx.x - T.tile0) * 64;
    const int lr = threadIdx.x >> 2, lk = (threadIdx.x & 3) * 4;   // this thread loads 4 columns of one row of each
    const int gi = i0 + lr, gj = j0 + lr;
    const bool vx = (ldx & 3) == 0 && gi < M, vw = (T.ldw & 3) == 0 && gj < T.N;
    float xr[4], wr[4];
    auto fetch4 = [&](const float* row, bool vec, bool in, int k, float (&v)[4]) {
        if (vec && k + 4 <= K) {
            const float4 q = *reinterpret_cast<const float4*>(row + k);
            v[0] = q.x;
            v[1] = q.y;
            v[2] = q.z;
            v[3] = q.w;
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = in && k + u < K ? row[k + u] : 0.f;
        }
    };
    auto fetch = [&](int k0) {
        fetch4(X + (size_t)gi * ldx, vx, gi < M, k0 + lk, xr);
        fetch4(T.W + (size_t)gj * T.ldw, vw, gj < T.N, k0 + lk, wr);
    };
    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            Xs[lk + u][lr] = xr[u];
            Ws[lk + u][lr] = wr[u];
        }
        __syncthreads();
        if (k0 + 16 < K) fetch(k0 + 16);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float4 x = *reinterpret_cast<const float4*>(&Xs[k][ty * 4]);
            const float4 w = *reinterpret_cast<const float4*>(&Ws[k][tx * 4]);
            const float xa[4] = {x.x, x.y, x.z, x.w}, wa[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(xa[u], wa[v], acc[u][v]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = i0 + ty * 4 + u;
        if (i >= M) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int j = j0 + tx * 4 + v;
            if (j >= T.N) continue;
            const size_t o = (size_t)i * T.ldc + j + (j >= T.split ? T.shift : 0);
            T.C[o] = T.alpha * acc[u][v] + (T.off ? T.off[j] : 0.f);
            if (T.C2) T.C2[o] = T.alpha * acc[u][v] + T.off2[j];
        }
    }
}

// Shared main loop of the FP32 batched kernels: a TS-slot x TR-row tile of
// sum_k X[slot, k] W[row, k] over k in [kbeg, kend) (rows of X and W have
// leading dimension ld, zero padded to a multiple of 64).  256 threads: thread
// (ty, tx) = (tid / 16, tid % 16) accumulates slots ty + 16 i (i < TS / 16) and
// rows tx + 16 j (j < TR / 16).  Every 16-wide k step is summed, in k order,
// into a fresh partial that is then added to the running sum: with
// multipliers of ~1e3 the terms of these dot products cancel heavily, and one
// long sequential FP32 sum would lose ~sqrt(K) units in the last place of its
// largest partial sum (measured: dual residuals off by 1e-3 on the humanoid
// workload).  The arithmetic of an output does not depend on TS or TR.
// k tiles of KB columns stream through a STAGES-deep cp.async pipeline into shared
// memory laid out [slot or row][k] with a padded stride, so that the copies run
// ahead of the arithmetic by STAGES - 1 tiles.  (A 32 x 32 tile's 16 columns are 32 clocks of
// FMAs per scheduler, less than the barrier and the copies' bookkeeping around them: with
// KB = 16 a layer at n + m = 420 took 15.2 us, now 9.)
template <int TS, int TR>
struct F32Tile {
    static constexpr int SA = TS / 16, RA = TR / 16;
    static constexpr int KB = 64;            // (divides every range of k)
    static constexpr int LDS = KB + 4;       // padded k stride in floats (16-byte aligned, rows 4 banks apart)
    static constexpr int STAGES = 3;
    static constexpr int XS = TS * LDS, WS = TR * LDS;
    static constexpr int BYTES = STAGES * (XS + WS) * 4;
};

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// `prep` runs once the results of the previous kernel can be read, the first copies in flight.
template <int TS, int TR, class F>
__device__ __forceinline__ void fp32_tile(const float* __restrict__ X, const float* __restrict__ W, int ld,
                                          int kbeg, int kend, int nrows, int slot0, int row0,
                                          float (&acc)[TS / 16][TR / 16], F prep) {
    using T = F32Tile<TS, TR>;
    extern __shared__ __align__(16) float fsm[];
    float* Xs = fsm;
    float* Ws = fsm + T::STAGES * T::XS;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < T::SA; ++a)
#pragma unroll
        for (int b = 0; b < T::RA; ++b) acc[a][b] = 0.f;
    // one k tile of X (TS rows) or of W (TR rows), KB / 4 chunks of 16 bytes a row
    constexpr int C = T::KB / 4;
    auto load_x = [&](int stage, int k0) {
        for (int e = threadIdx.x; e < C * TS; e += 256) {
            const int c = e % C, sl = e / C;
            cp_async16(Xs + stage * T::XS + sl * T::LDS + 4 * c, X + (size_t)(slot0 + sl) * ld + k0 + 4 * c, true);
        }
    };
    auto load_w = [&](int stage, int k0) {
        for (int e = threadIdx.x; e < C * TR; e += 256) {
            const int c = e % C, rw = e / C;
            const bool ok = row0 + rw < nrows;
            cp_async16(Ws + stage * T::WS + rw * T::LDS + 4 * c, ok ? W + (size_t)(row0 + rw) * ld + k0 + 4 * c : W, ok);
        }
    };
    // the weights of the first stages do not depend on the previous kernel of the stream
#pragma unroll
    for (int s = 0; s < T::STAGES - 1; ++s)
        if (kbeg + T::KB * s < kend) load_w(s, kbeg + T::KB * s);
    griddep_wait();
#pragma unroll
    for (int s = 0; s < T::STAGES - 1; ++s) {
        if (kbeg + T::KB * s < kend) load_x(s, kbeg + T::KB * s);
        cp_async_commit();   // (the first group also holds the weights above)
    }
    prep();
    int it = 0;
    for (int k0 = kbeg; k0 < kend; k0 += T::KB, ++it) {
        cp_async_wait<T::STAGES - 2>();
        __syncthreads();
        const int kn = k0 + T::KB * (T::STAGES - 1);
        if (kn < kend) {
            load_w((it + T::STAGES - 1) % T::STAGES, kn);
            load_x((it + T::STAGES - 1) % T::STAGES, kn);
        }
        cp_async_commit();
        const float* xs = Xs + (it % T::STAGES) * T::XS;
        const float* ws = Ws + (it % T::STAGES) * T::WS;
#pragma unroll
        for (int k1 = 0; k1 < T::KB; k1 += 16) {
            float part[T::SA][T::RA];
#pragma unroll
            for (int a = 0; a < T::SA; ++a)
#pragma unroll
                for (int b = 0; b < T::RA; ++b) part[a][b] = 0.f;
#pragma unroll
            for (int kk = k1; kk < k1 + 16; kk += 4) {
                float4 xa[T::SA], wb[T::RA];
#pragma unroll
                for (int a = 0; a < T::SA; ++a) xa[a] = *reinterpret_cast<const float4*>(xs + (ty + 16 * a) * T::LDS + kk);
#pragma unroll
                for (int b = 0; b < T::RA; ++b) wb[b] = *reinterpret_cast<const float4*>(ws + (tx + 16 * b) * T::LDS + kk);
#pragma unroll
                for (int a = 0; a < T::SA; ++a)
#pragma unroll
                    for (int b = 0; b < T::RA; ++b) {
                        part[a][b] = fmaf(xa[a].x, wb[b].x, part[a][b]);
                        part[a][b] = fmaf(xa[a].y, wb[b].y, part[a][b]);
                        part[a][b] = fmaf(xa[a].z, wb[b].z, part[a][b]);
                        part[a][b] = fmaf(xa[a].w, wb[b].w, part[a][b]);
                    }
            }
#pragma unroll
            for (int a = 0; a < T::SA; ++a)
#pragma unroll
                for (int b = 0; b < T::RA; ++b) acc[a][b] += part[a][b];
        }
    }
    cp_async_wait<0>();
    // the next kernel may set up and load its weights while this one's epilogue runs
    griddep_launch();
}

// Slot range of a CTA: TS-slot sub-tiles of the 128-slot tiles; a sub-tile
// with no active QP has nothing to do (the active QPs of a bank group fill
// its slots from the first one on, so perm of the first slot decides).
template <int TS>
__device__ __forceinline__ bool fp32_slots(const BatchParams& p, int& tile, int& slot0) {
    tile = (blockIdx.y * TS) / kSlotTile;
    slot0 = blockIdx.y * TS;
    if (tile >= p.counters[CNT_TILES]) return false;
    return p.perm[slot0] >= 0;
}

// One layer for every active slot tile (FP32 backend).  What the element-wise part reads is
// loaded for all elements of a thread before any of them is written: the compiler cannot move
// a load above a store that might alias it, and one round trip to L2 per element (some 0.5 us)
// took longer than the product.  Up to 8 elements it is loaded under the product (at most 56
// registers), beyond that a row of the tile at a time after it.
template <int TS, int TR>
__global__ void __launch_bounds__(256) batch_layer_fp32_kernel(BatchParams p, const __grid_constant__ W32Ptrs wp) {
    constexpr int SA = TS / 16, RA = TR / 16;
    constexpr bool EARLY = SA * RA <= 8;
    int tile, slot0;
    if (!fp32_slots<TS>(p, tile, slot0)) return;
    const int ri = p.tile_rho[tile];
    const int row0 = blockIdx.x * TR;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    int qp[SA];
#pragma unroll
    for (int a = 0; a < SA; ++a) qp[a] = p.perm[slot0 + ty + 16 * a];
    LayerIn in[EARLY ? SA : 1][RA];
    auto load = [&](int a, LayerIn (&v)[RA]) {
        if (qp[a] < 0) return;
#pragma unroll
        for (int b = 0; b < RA; ++b) {
            const int r = row0 + tx + 16 * b;
            if (r < p.R) layer_load(p, qp[a], ri, r, v[b]);
        }
    };
    float acc[SA][RA];
    fp32_tile<TS, TR>(p.Sin, wp.w[ri], p.ldk, 0, p.ldk, p.R, slot0, row0, acc, [&] {
        if constexpr (EARLY) {
#pragma unroll
            for (int a = 0; a < SA; ++a) load(a, in[a]);
        }
    });
#pragma unroll
    for (int a = 0; a < SA; ++a) {
        if (!EARLY) load(a, in[0]);
        if (qp[a] < 0) continue;
#pragma unroll
        for (int b = 0; b < RA; ++b) {
            const int r = row0 + tx + 16 * b;
            if (r < p.R) layer_apply(p, p.flags, slot0 + ty + 16 * a, qp[a], ri, r, acc[a][b], in[EARLY ? a : 0][b]);
        }
    }
}

// max over the 16 threads of a half warp that share ty (NaN kept)
__device__ __forceinline__ float half_warp_max(float v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v = nmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Residual products (FP32 backend).  Phase 1: [P; A] x over the x columns of
// the check operand; phase 2: A^T lam_std over its multiplier columns.
template <int TS, int TR>
__global__ void __launch_bounds__(256) batch_check_fp32_kernel(BatchParams p, const float* __restrict__ Wc, int phase) {
    int tile, slot0;
    if (!fp32_slots<TS>(p, tile, slot0)) return;
    const int ri = p.tile_rho[tile];
    const int row0 = blockIdx.x * TR;
    const int rows = phase == 1 ? p.n + p.m : p.n;
    float acc[TS / 16][TR / 16];
    if (phase == 1)
        fp32_tile<TS, TR>(p.CK32, Wc, p.ldkc, 0, p.n64, rows, slot0, row0, acc, [] {});
    else
        fp32_tile<TS, TR>(p.CK32, Wc, p.ldkc, p.n64, p.ldkc, rows, slot0, row0, acc, [] {});
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < TS / 16; ++a) {
        const int slot = slot0 + ty + 16 * a;
        const int qp = p.perm[slot];     // the same in the 16 threads of a half warp
        float r0 = 0.f, r1 = 0.f, r2 = 0.f, r3 = 0.f;
        if (qp >= 0) {
#pragma unroll
            for (int b = 0; b < TR / 16; ++b) {
                const int r = row0 + tx + 16 * b;
                if (r >= rows) continue;
                if (phase == 1) check1_elem(p, slot, qp, ri, r, acc[a][b], r0, r1, r2, r3);
                else check2_elem(p, qp, r, acc[a][b], r0, r1);
            }
        }
        r0 = half_warp_max(r0);
        r1 = half_warp_max(r1);
        r2 = half_warp_max(r2);
        r3 = half_warp_max(r3);
        if (qp < 0 || tx != 0) continue;
        if (phase == 1) {
            red_slot(p.RED, qp, RW_RP, r0);
            red_slot(p.RED, qp, RW_AX, r1);
            red_slot(p.RED, qp, RW_Z, r2);
            red_slot(p.RED, qp, RW_PX, r3);
        } else {
            red_slot(p.RED, qp, RW_RD, r0);
            red_slot(p.RED, qp, RW_ATL, r1);
        }
    }
}

// All `nl` layers of a chunk (FP32 backend, n + m <= 512), TS slots per cluster of up to 8 CTAs
// with 64 rows each.  A launch per layer is bound by what lies between two products: the launch,
// the weights and the operand from L2 again, the state in and out.  Here a CTA keeps its rows of
// Wt and the slots' operand in shared memory and its elements' state in registers, and a layer
// is the product, one cluster barrier - every CTA has read the operand - under the element-wise
// part, and the new operand sent by st.async into every CTA's copy, counted in bytes on its
// mbarrier.  The arithmetic of an output is fp32_tile's and layer_apply's.
// What bounds it is the product's shared memory reads: a 16-byte read of 32 rows is four passes
// whoever else reads them, so a warp takes 64 rows and 4 slots (12 passes to 32 FMA
// instructions; with 32 rows and 4 slots in 16 lanes each, 18).  The exchange takes 1.1 us.
// A layer at n + m = 420: 7.9 us (16 slots a cluster) and 12.3 (32), with a launch per layer 12 to
// 18; solves, ms, one launch per layer / per chunk: n + m = 420, 40 QPs 3.42 / 2.94, 333 QPs 5.13 /
// 4.22, 1000 QPs 8.06 / 7.41; 500, 200 QPs 5.46 / 4.02; 80, 600 QPs 1.91 / 1.75.
constexpr int kChunk32Rows = 64;
constexpr int kChunk32MaxK = 512;      // 8 CTAs, the portable cluster

template <int TS>
constexpr int chunk32_bytes(int ld) { return (kChunk32Rows + TS) * (ld + 4) * (int)sizeof(float); }

template <int TS>
__global__ void __launch_bounds__(8 * TS, 1) batch_chunk_fp32_kernel(BatchParams p, const __grid_constant__ W32Ptrs wp,
                                                               int nl, unsigned last_flags, int* err,
                                                               long long timeout_ns) {
    constexpr int THREADS = 8 * TS, NW = TS / 4, SA = 4, RA = kChunk32Rows / 32;   // a warp: 4 slots, 64 rows
    extern __shared__ __align__(16) float fsm[];
    __shared__ __align__(8) unsigned long long s_bar;
    int tile, slot0;
    if (!fp32_slots<TS>(p, tile, slot0)) return;       // uniform over the cluster
    const int ri = p.tile_rho[tile], ld = p.ldk, lds = ld + 4, c4 = ld / 4;
    const int row0 = blockIdx.x * kChunk32Rows, ctas = gridDim.x;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // slots ty + NW a, rows tx + 32 b
    float* Ws = fsm;                                   // [64][lds] (rows 4 banks apart)
    float* Xs = fsm + kChunk32Rows * lds;              // [TS][lds]
    const uint32_t bar = cl_smem(&s_bar);
    const uint32_t bytes = (uint32_t)(TS * ld * 4);    // a layer's operand: every CTA sends TS x 64
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        cl_expect(bar, bytes);
    }
    const float* W = wp.w[ri];
    for (int e = threadIdx.x; e < kChunk32Rows * c4; e += THREADS) {
        const int rw = e / c4, c = e - rw * c4;
        const bool ok = row0 + rw < p.R;
        cp_async16(Ws + rw * lds + 4 * c, ok ? W + (size_t)(row0 + rw) * ld + 4 * c : W, ok);
    }
    griddep_wait();
    griddep_launch();
    for (int e = threadIdx.x; e < TS * c4; e += THREADS) {
        const int sl = e / c4, c = e - sl * c4;
        cp_async16(Xs + sl * lds + 4 * c, p.Sin + (size_t)(slot0 + sl) * ld + 4 * c, true);
    }
    cp_async_commit();
    int qp[SA];
    LayerIn in[SA][RA];
#pragma unroll
    for (int a = 0; a < SA; ++a) {
        qp[a] = p.perm[slot0 + ty + NW * a];
#pragma unroll
        for (int b = 0; b < RA; ++b)
            if (const int r = row0 + tx + 32 * b; qp[a] >= 0 && r < p.R) layer_load(p, qp[a], ri, r, in[a][b]);
    }
    cp_async_wait<0>();
    __syncthreads();
    cl_sync_hw();                                      // every CTA's mbarrier is armed
    // a thread whose wait gave up goes through the layers (its warp's shuffles and the barriers name
    // it) but sends nothing, so that its partners' waits find the error word and not their bytes,
    // and nobody goes on sending to a CTA that no longer counts what arrives
    bool failed = false;
    for (int j = 0; j < nl; ++j) {
        const bool last = j == nl - 1;
        if (j > 0) {
            if (!failed && !cl_wait(bar, (uint32_t)((j - 1) & 1), err, timeout_ns)) failed = true;
            if (threadIdx.x == 0 && !failed && !last) cl_expect(bar, bytes);
        }
        float acc[SA][RA];
#pragma unroll
        for (int a = 0; a < SA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) acc[a][b] = 0.f;
        for (int k0 = 0; k0 < ld; k0 += 16) {
            float part[SA][RA];
#pragma unroll
            for (int a = 0; a < SA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b) part[a][b] = 0.f;
#pragma unroll
            for (int kk = k0; kk < k0 + 16; kk += 4) {
                float4 xa[SA], wb[RA];
#pragma unroll
                for (int a = 0; a < SA; ++a) xa[a] = *reinterpret_cast<const float4*>(Xs + (ty + NW * a) * lds + kk);
#pragma unroll
                for (int b = 0; b < RA; ++b) wb[b] = *reinterpret_cast<const float4*>(Ws + (tx + 32 * b) * lds + kk);
#pragma unroll
                for (int a = 0; a < SA; ++a)
#pragma unroll
                    for (int b = 0; b < RA; ++b) {
                        part[a][b] = fmaf(xa[a].x, wb[b].x, part[a][b]);
                        part[a][b] = fmaf(xa[a].y, wb[b].y, part[a][b]);
                        part[a][b] = fmaf(xa[a].z, wb[b].z, part[a][b]);
                        part[a][b] = fmaf(xa[a].w, wb[b].w, part[a][b]);
                    }
            }
#pragma unroll
            for (int a = 0; a < SA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b) acc[a][b] += part[a][b];
        }
        if (last) {
            if (failed) break;
#pragma unroll
            for (int a = 0; a < SA; ++a)
#pragma unroll
                for (int b = 0; b < RA; ++b)
                    if (const int r = row0 + tx + 32 * b; qp[a] >= 0 && r < p.R)
                        layer_apply(p, last_flags, slot0 + ty + NW * a, qp[a], ri, r, acc[a][b], in[a][b]);
            break;
        }
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        float sn[SA][RA];
#pragma unroll
        for (int a = 0; a < SA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) {
                const int r = row0 + tx + 32 * b;
                sn[a][b] = qp[a] >= 0 && r < p.R ? layer_carry(p, ri, r, acc[a][b], in[a][b]) : 0.f;
            }
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        __syncwarp();
        // four lanes hold rows 4 q .. 4 q + 3 of two slots, for either b: transposed, a lane has
        // four consecutive rows to send at once
        const int jl = tx & 3;
#pragma unroll
        for (int a = 0; a < SA; a += 2) {
            float o[4];
#pragma unroll
            for (int st = 0; st < 4; ++st) {
                const int c = jl ^ st;
                const float v = c == 0 ? sn[a][0] : c == 1 ? sn[a][1] : c == 2 ? sn[a + 1][0] : sn[a + 1][1];
                const float g = __shfl_xor_sync(0xffffffffu, v, st);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i == c) o[i] = g;
            }
            const uint32_t dst = cl_smem(Xs + (ty + NW * (a + (jl >> 1))) * lds + row0 + 32 * (jl & 1) + (tx & 28));
            for (int q = 0; q < (failed ? 0 : ctas); ++q) cl_send4(dst, bar, q, o[0], o[1], o[2], o[3]);
        }
    }
    cl_close(failed);
}

// pdl: the kernel may start before the previous one of the stream has ended (its griddep_wait)
template <class K, class... Args>
int launch_pdl(relu_qp_t h, K k, dim3 grid, int threads, int smem, bool pdl, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = h->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    RQ_CUDA(h, cudaLaunchKernelEx(&cfg, k, args...));
    return RELU_QP_OK;
}

template <class K, class... Args>
int launch32(relu_qp_t h, K k, dim3 grid, int smem, bool pdl, Args... args) {
    RQ_CUDA(h, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return launch_pdl(h, k, grid, 256, smem, pdl, args...);
}

template <int TS, int TR>
int launch_layer32(relu_qp_t h, const BatchParams& q, const W32Ptrs& wp, int tiles_max, bool pdl) {
    return launch32(h, batch_layer_fp32_kernel<TS, TR>, dim3(ceil_div(h->R, TR), tiles_max * (kSlotTile / TS)),
                    F32Tile<TS, TR>::BYTES, pdl, q, wp);
}

int layer32(relu_qp_t h, const BatchParams& q, const W32Ptrs& wp, int tiles_max, int active, bool pdl) {
    const Tile32 t = tile32(h->R, active, h->nr, h->num_sms);
    if (t.tr == 64) return launch_layer32<64, 64>(h, q, wp, tiles_max, pdl);
    if (t.ts == 64) return launch_layer32<64, 32>(h, q, wp, tiles_max, pdl);
    return launch_layer32<32, 32>(h, q, wp, tiles_max, pdl);
}

template <int TS, int TR>
int launch_check32(relu_qp_t h, const BatchParams& q, const float* Wc, int tiles_max, int phase) {
    const int rows = phase == 1 ? h->n + h->m : h->n;
    return launch32(h, batch_check_fp32_kernel<TS, TR>, dim3(ceil_div(rows, TR), tiles_max * (kSlotTile / TS)),
                    F32Tile<TS, TR>::BYTES, true, q, Wc, phase);
}

int check32(relu_qp_t h, const BatchParams& q, const float* Wc, int tiles_max, int active, int phase) {
    const Tile32 t = tile32(phase == 1 ? h->n + h->m : h->n, active, h->nr, h->num_sms);
    if (t.tr == 64) return launch_check32<64, 64>(h, q, Wc, tiles_max, phase);
    if (t.ts == 64) return launch_check32<64, 32>(h, q, Wc, tiles_max, phase);
    return launch_check32<32, 32>(h, q, Wc, tiles_max, phase);
}

template <int TS>
int launch_chunk32(relu_qp_t h, const BatchParams& q, const W32Ptrs& wp, int tiles_max, int nl, unsigned last_flags) {
    BatchWork& w = h->bw;
    auto k = batch_chunk_fp32_kernel<TS>;
    const int smem = chunk32_bytes<TS>(w.ldk), ctas = w.ldk / kChunk32Rows;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas, tiles_max * (kSlotTile / TS));
    cfg.blockDim = dim3(8 * TS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = h->stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    int& fit = w.chunk32_fit[TS == 32];
    if (fit < 0) {
        int room = 0;
        RQ_TRY(allow_shared(h, (const void*)k, &room));
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&fit, k, &cfg) != cudaSuccess) {
            cudaGetLastError();
            fit = 0;
        }
        cfg.numAttrs = 2;
    }
    if (nl <= 0) return RELU_QP_OK;        // (nl = 0: only w.chunk32_fit)
    RQ_CUDA(h, cudaLaunchKernelEx(&cfg, k, q, wp, nl, last_flags, w.counters + CNT_ERR, 2000000000LL));
    return RELU_QP_OK;
}

// The chunk's layers in one launch, or RELU_QP_ERR_UNSUPPORTED where a launch per layer is better:
// the clusters of all slots must fit the GPU at once, preferably of 16 slots.  (In two waves the
// tiles that fill every SM win: n + m = 420, 600 QPs 6.23 ms against 5.17, 1000 QPs 7.63 against 7.47.)
int chunk32(relu_qp_t h, const BatchParams& q, const W32Ptrs& wp, int tiles_max, int active, int nl, unsigned last_flags) {
    BatchWork& w = h->bw;
    if (w.ldk > kChunk32MaxK) return RELU_QP_ERR_UNSUPPORTED;
    auto fits = [&](int ts, int fit) { return ceil_div(active, ts) + (active > ts ? h->nr - 1 : 0) <= fit; };
    if (w.chunk32_fit[0] < 0) RQ_TRY(launch_chunk32<16>(h, q, wp, tiles_max, 0, 0u));
    if (fits(16, w.chunk32_fit[0])) return launch_chunk32<16>(h, q, wp, tiles_max, nl, last_flags);
    if (w.chunk32_fit[1] < 0) RQ_TRY(launch_chunk32<32>(h, q, wp, tiles_max, 0, 0u));
    if (fits(32, w.chunk32_fit[1])) return launch_chunk32<32>(h, q, wp, tiles_max, nl, last_flags);
    return RELU_QP_ERR_UNSUPPORTED;
}

// Stop test and penalty rule per QP (one 128-thread block per QP: thread 0
// decides, the block copies the outputs of a finished QP or rebases lam' on a
// bank switch).
constexpr int kDecideThreads = 128;

// by_slot: one block per slot of the tiles in use (QP = perm[slot], padding
// slots return), which covers every active QP; else one block per QP id.
__global__ void __launch_bounds__(kDecideThreads) batch_decide_kernel(BatchParams p, DecideArgs d, int by_slot) {
    griddep_wait();
    griddep_launch();
    const int qp = by_slot ? p.perm[blockIdx.x] : (int)blockIdx.x;
    if (qp < 0 || qp >= d.B) return;
    __shared__ int s_act, s_nri;    // s_act: -1 not active, 0 continue, 1 finished, 2 bank switch
    unsigned* red = p.RED + (size_t)qp * RW_WORDS;
    if (threadIdx.x == 0) {
        int act = -1, nri = 0;
        if (d.status[qp] == QP_ACTIVE) {
            const unsigned w[RW_WORDS] = {red[0], red[1], red[2], red[3], red[4], red[5], red[6], red[7]};
            act = decide_qp(p, d, qp, w, nri);
        }
        s_act = act;
        s_nri = nri;
    }
    __syncthreads();
    const int act = s_act;
    if (act < 0) return;
    if (act == 1) {
        for (int k = threadIdx.x; k < p.n; k += kDecideThreads) d.XO[(size_t)qp * p.n + k] = p.Y[(size_t)qp * p.ldn + k];
        for (int i = threadIdx.x; i < p.m; i += kDecideThreads) {
            d.ZO[(size_t)qp * p.m + i] = p.Z[(size_t)qp * p.ldm + i];
            d.LO[(size_t)qp * p.m + i] = p.LSTD[(size_t)qp * p.ldm + i];
        }
    } else if (act == 2) {
        // rebase lam' so that the next layer is standard ADMM with the new rho
        const int nri = s_nri;
        for (int i = threadIdx.x; i < p.m; i += kDecideThreads) {
            const size_t o = (size_t)qp * p.ldm + i;
            const float rho_i = (float)(p.rhod[nri] * (double)p.rs[i]);
            p.LAM[o] = lam_standard(p.LSTD[o], -rho_i, p.AY[o] - p.Z[o]);
        }
    }
    if (threadIdx.x < RW_WORDS) red[threadIdx.x] = 0u;
}

// (Not __restrict__: what an earlier kernel writes must not be read before griddep_wait.)
// Regroup the active QPs by bank index: slots [base_g, base_g + count_g) hold
// group g in increasing QP id, each group padded to a multiple of 128 slots.
__global__ void __launch_bounds__(1024) batch_assign_kernel(int B, int slots, int nr, const int* status,
                                                            const int* rho_idx, int* perm,
                                                            int* tile_rho, int* counters) {
    __shared__ int cnt[RQ_MAX_RHO], base[RQ_MAX_RHO], warp_cnt[32], run;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    griddep_wait();
    griddep_launch();
    for (int s = tid; s < slots; s += blockDim.x) perm[s] = -1;
    if (tid < RQ_MAX_RHO) cnt[tid] = 0;
    __syncthreads();
    for (int qp = tid; qp < B; qp += blockDim.x)
        if (status[qp] == QP_ACTIVE) atomicAdd(&cnt[rho_idx[qp]], 1);
    __syncthreads();
    if (tid == 0) {
        int off = 0, t = 0, tot = 0;
        for (int g = 0; g < nr; ++g) {
            base[g] = off;
            const int tiles = (cnt[g] + kSlotTile - 1) / kSlotTile;
            for (int k = 0; k < tiles; ++k) tile_rho[t++] = g;
            off += tiles * kSlotTile;
            tot += cnt[g];
        }
        counters[CNT_TILES] = t;
        counters[CNT_ACTIVE] = tot;
    }
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    for (int g = 0; g < nr; ++g) {
        if (cnt[g] == 0) continue;
        for (int c0 = 0; c0 < B; c0 += blockDim.x) {
            const int qp = c0 + tid;
            const bool flag = qp < B && status[qp] == QP_ACTIVE && rho_idx[qp] == g;
            const unsigned ball = __ballot_sync(0xffffffffu, flag);
            if (lane == 0) warp_cnt[warp] = __popc(ball);
            __syncthreads();
            if (tid == 0) {
                int acc = 0;
                for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
                    const int c = warp_cnt[w];
                    warp_cnt[w] = acc;
                    acc += c;
                }
                run = acc;
            }
            __syncthreads();
            if (flag) perm[base[g] + warp_cnt[warp] + __popc(ball & lt)] = qp;
            __syncthreads();
            if (tid == 0) base[g] += run;
            __syncthreads();
        }
    }
}

// Operand of the first layer of a chunk: s = [x; 2 rho z - lam'] per slot, in
// FP32 or as a 3-way BF16 split; padding slots get zeros.  One thread per 4
// consecutive columns of a slot.
__global__ void batch_fill_kernel(BatchParams p, const int* rho_idx, float* S32, __nv_bfloat16* T,
                                  size_t part) {
    griddep_wait();
    griddep_launch();
    const int q4 = p.ldk >> 2;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int slot = (int)(e / q4);
    const int k0 = (int)(e % q4) * 4;
    if (slot >= p.counters[CNT_TILES] * kSlotTile) return;
    const int qp = p.perm[slot];
    const int ri = qp >= 0 ? rho_idx[qp] : 0;
    float v[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int k = k0 + t;
        v[t] = 0.f;
        if (qp >= 0) {
            if (k < p.n) {
                v[t] = p.Y[(size_t)qp * p.ldn + k];
            } else if (k < p.R) {
                const int i = k - p.n;
                const size_t o = (size_t)qp * p.ldm + i;
                v[t] = next_operand(p.rho[ri] * p.rs[i], p.Z[o], p.LAM[o]);
            }
        }
    }
    const size_t o = (size_t)slot * p.ldk + k0;
    if (S32) {
        st4(S32 + o, v);
    } else {
        __nv_bfloat16 a[4], b[4], c[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) split3(v[t], a[t], b[t], c[t]);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            T[o + t] = a[t];
            T[o + t + part] = b[t];
            T[o + t + 2 * part] = c[t];
        }
    }
}

// Start state per QP: x given (Y) or 0, z = A x (AY holds A x for warm starts),
// lam' = lam_warm (staged in LSTD) or 0.
// One block per QP.
constexpr int kInitThreads = 128;
__global__ void __launch_bounds__(kInitThreads) batch_init_kernel(BatchParams p, int B, int warm, int lam_given,
                                                                  const int* __restrict__ rw, int rho0, int* status,
                                                                  int* rho_idx, int* iters, int* nsw) {
    const int qp = blockIdx.x, tid = threadIdx.x;
    if (tid == 0) {
        status[qp] = qp < B ? QP_ACTIVE : QP_UNUSED;
        rho_idx[qp] = (qp < B && rw) ? rw[qp] : rho0;   // (rw may be iters: read first)
        iters[qp] = 0;
        nsw[qp] = 0;
    }
    if (tid < RW_WORDS) p.RED[(size_t)qp * RW_WORDS + tid] = 0u;
    if (qp >= B) return;
    // (the padding is zeroed too: a QP of NaN data leaves NaN there)
    for (int i = tid; i < p.ldm; i += kInitThreads) {
        const size_t o = (size_t)qp * p.ldm + i;
        const float ax = warm && i < p.m ? p.AY[o] : 0.f;
        p.AY[o] = ax;
        p.Z[o] = ax;
        p.LAM[o] = lam_given && i < p.m ? p.LSTD[o] : 0.f;
    }
    for (int k = (warm ? p.n : 0) + tid; k < p.ldn; k += kInitThreads) p.Y[(size_t)qp * p.ldn + k] = 0.f;
}

// The solve's records as the caller's relu_qp_info (solve_ms is the host's).
__global__ void pack_info_kernel(int B, const int* __restrict__ status, const int* __restrict__ iters,
                                 const int* __restrict__ rho_idx, const int* __restrict__ nsw,
                                 const float* __restrict__ rp, const float* __restrict__ rd, relu_qp_info* out) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    relu_qp_info r;
    r.status = status[b];
    r.iters = iters[b];
    r.rho_index = rho_idx[b];
    r.rho_switches = nsw[b];
    r.r_prim = rp[b];
    r.r_dual = rd[b];
    r.solve_ms = 0.0;
    out[b] = r;
}

// out[r] = max_k |X[r][k] f[k]| (f = nullptr: 1).
__global__ void row_absmax_kernel(const float* __restrict__ X, int rows, int cols, int ld,
                                  const float* __restrict__ f, float* out) {
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    float v = 0.f;
    for (int k = lane; k < cols; k += 32) v = fmaxf(v, fabsf(f ? X[(size_t)r * ld + k] * f[k] : X[(size_t)r * ld + k]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) out[r] = v;
}

// X[r][k] *= f[k] for rows [0, rows): the problem scaling's maps between the
// original and the scaled problem's data and iterates.
__global__ void scale_rows_kernel(float* X, int rows, int cols, int ld, const float* __restrict__ f) {
    const size_t total = (size_t)rows * cols;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / cols), k = (int)(e % cols);
        X[(size_t)r * ld + k] *= f[k];
    }
}

// Check matrix [[P, A^T], [A, 0]] in FP32: x columns [0, n64), multiplier
// columns [n64, n64 + m64); rows [0, n) for P and A^T, [n, n + m) for A.
__global__ void build_wc32_kernel(const float* __restrict__ P32, const float* __restrict__ A32, int ldp,
                                  const float* __restrict__ At32, int ldt, int n, int m, int n64, int ldkc,
                                  float* __restrict__ Wc) {
    const size_t total = (size_t)(n + m) * ldkc;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(e / ldkc), k = (int)(e % ldkc);
        float v = 0.f;
        if (j < n) {
            if (k < n) v = P32[(size_t)j * ldp + k];
            else if (k >= n64 && k < n64 + m) v = At32[(size_t)j * ldt + (k - n64)];
        } else if (k < n) {
            v = A32[(size_t)(j - n) * ldp + k];
        }
        Wc[e] = v;
    }
}

// The maps of one X, gathered and launched together.
struct Maps {
    MapTasks ts{};
    int tiles = 0;
    void add(int N, const float* W, int ldw, float alpha, const float* off, float* C, int ldc, int split = 0, int shift = 0,
             const float* off2 = nullptr, float* C2 = nullptr) {
        if (N <= 0) return;
        ts.t[ts.count++] = MapTask{W, off, off2, C, C2, N, ldw, ldc, split, shift, tiles, alpha};
        tiles += ceil_div(N, 64);
    }
    int run(relu_qp_t h, int M, int K, const float* X, int ldx) const {
        if (M <= 0 || ts.count == 0) return RELU_QP_OK;
        map_kernel<<<dim3(tiles, ceil_div(M, 64)), 256, 0, h->stream>>>(M, K, X, ldx, ts);
        RQ_CUDA(h, cudaGetLastError());
        ++h->launches;
        return RELU_QP_OK;
    }
};

BatchParams base_params(relu_qp_t h) {
    BatchWork& w = h->bw;
    BatchParams p{};
    p.n = h->n;
    p.m = h->m;
    p.R = h->R;
    p.ldn = w.ldn;
    p.ldm = w.ldm;
    p.ldR = w.ldR;
    p.ldk = w.ldk;
    p.n64 = w.n64;
    p.ldkc = w.ldkc;
    p.cap = w.cap;
    p.slots = w.slots;
    p.nr = h->nr;
    p.bsh = w.nP - h->n;
    for (int r = 0; r < h->nr; ++r) {
        p.rho[r] = (float)h->be[r].rho;
        p.rhod[r] = h->be[r].rho;
    }
    p.rs = h->rs32;
    p.rsx = h->sc_rx;
    p.rsz = h->sc_z;
    p.Y = w.Y; p.Z = w.Z; p.LAM = w.LAM; p.AY = w.AY; p.RR = w.RR; p.LSTD = w.LSTD; p.C = w.C; p.SREF = w.SREF; p.PY = w.PY;
    p.L = w.L; p.U = w.U; p.Q = w.Q; p.BIAS = w.BIAS; p.QN = w.QN;
    p.perm = w.perm; p.tile_rho = w.tile_rho; p.counters = w.counters; p.RED = w.RED;
    return p;
}

// p in the backend's row layout (the padded one of the split form), for the kernels that
// run the layers and the residual products and fill their operand
BatchParams layer_params(relu_qp_t h, const BatchParams& p) {
    BatchParams q = p;
    q.n = h->bw.nP;
    q.m = h->bw.RP - h->bw.nP;
    q.R = h->bw.RP;
    q.bsh = 0;
    return q;
}

int scale_rows(relu_qp_t h, float* X, int rows, int cols, int ld, const float* f) {
    if (!f || rows <= 0 || cols <= 0) return RELU_QP_OK;
    const size_t total = (size_t)rows * cols;
    const int g = (int)std::min<size_t>((total + 255) / 256, 4096);
    scale_rows_kernel<<<g, 256, 0, h->stream>>>(X, rows, cols, ld, f);
    RQ_CUDA(h, cudaGetLastError());
    ++h->launches;
    return RELU_QP_OK;
}

int copy_rows_in(relu_qp_t h, float* dst, int ld, const float* src, int rows, int cols) {
    if (rows <= 0 || cols <= 0) return RELU_QP_OK;
    RQ_CUDA(h, cudaMemcpy2DAsync(dst, sizeof(float) * ld, src, sizeof(float) * cols, sizeof(float) * cols, rows,
                                 cudaMemcpyDefault, h->stream));
    return RELU_QP_OK;
}

}  // namespace

// Device bytes per QP slot of a batched handle: the arrays batch_alloc sizes by
// max_batch (per-QP state, bias rows of every bank entry, outputs, records) and
// the share of the slot-indexed operands (cap slots of the slots rows).
size_t batch_slot_bytes(relu_qp_t h) {
    const BatchWork& w = h->bw;
    const size_t mm = h->m > 0 ? h->m : 1, f = sizeof(float);
    size_t b = 3 * w.ldn * f + f;                       // Y, Q, PY, QN
    b += 7 * w.ldm * f;                                 // Z, LAM, AY, RR, LSTD, L, U
    b += (size_t)h->nr * w.ldR * f;                     // BIAS
    b += (h->n + 2 * mm) * f;                           // XO, ZO, LO
    b += RW_WORDS * sizeof(unsigned) + 6 * sizeof(int); // RED, rho_idx, status, iters, nsw, rp, rd
    b += sizeof(int);                                   // perm
    if (w.prec == RELU_QP_PREC_BF16X3) {
        b += 2 * w.ldR * f;                             // C, SREF
        b += 2 * (7 * (size_t)w.ldk + 3 * (size_t)w.ldkc);   // BF16 operand parts and check operand
    } else {
        b += 2 * w.ldk * f + w.ldkc * f;                // S32 pair, CK32
    }
    return b;
}

int batch_alloc(relu_qp_t h) {
    BatchWork& w = h->bw;
    const int n = h->n, m = h->m, R = h->R, nr = h->nr;
    const int mm = m > 0 ? m : 1;
    w.cap = h->opts.max_batch;
    w.prec = h->opts.batch_precision;
    w.slots = (int)round_up(w.cap, kSlotTile) + nr * kSlotTile;
    const bool bf16 = w.prec == RELU_QP_PREC_BF16X3;
    w.nP = bf16 ? (int)round_up(n, 16) : n;
    w.RP = bf16 ? w.nP + (int)round_up(m, 16) : R;
    w.ldn = (int)round_up(n, bf16 ? 16 : 4);
    w.ldm = (int)round_up(mm, bf16 ? 16 : 4);
    w.ldR = (int)round_up(w.RP, 4);
    w.ldk = (int)round_up(w.RP, 64);
    w.n64 = (int)round_up(n, 64);
    w.m64 = (int)round_up(mm, 64);
    w.ldkc = w.n64 + w.m64;
    w.Rpad = (int)round_up(w.RP, 256);
    w.npad = w.Rpad;
    const size_t cap = w.cap;
    RQ_TRY(alloc(h, &w.Y, cap * w.ldn));
    RQ_TRY(alloc(h, &w.Q, cap * w.ldn));
    RQ_TRY(alloc(h, &w.PY, cap * w.ldn));
    RQ_TRY(alloc(h, &w.QN, cap));
    RQ_TRY(alloc(h, &w.Z, cap * w.ldm));
    RQ_TRY(alloc(h, &w.LAM, cap * w.ldm));
    RQ_TRY(alloc(h, &w.AY, cap * w.ldm));
    RQ_TRY(alloc(h, &w.RR, cap * w.ldm));
    RQ_TRY(alloc(h, &w.LSTD, cap * w.ldm));
    RQ_TRY(alloc(h, &w.L, cap * w.ldm));
    RQ_TRY(alloc(h, &w.U, cap * w.ldm));
    RQ_TRY(alloc(h, &w.BIAS, (size_t)nr * cap * w.ldR));
    RQ_TRY(alloc(h, &w.XO, cap * n));
    RQ_TRY(alloc(h, &w.ZO, cap * mm));
    RQ_TRY(alloc(h, &w.LO, cap * mm));
    RQ_TRY(alloc(h, &w.RED, cap * RW_WORDS));
    RQ_TRY(alloc(h, &w.rho_idx, cap));
    RQ_TRY(alloc(h, &w.status, cap));
    RQ_TRY(alloc(h, &w.iters, cap));
    RQ_TRY(alloc(h, &w.nsw, cap));
    RQ_TRY(alloc(h, &w.rp, cap));
    RQ_TRY(alloc(h, &w.rd, cap));
    RQ_TRY(alloc(h, &w.perm, (size_t)w.slots));
    RQ_TRY(alloc(h, &w.tile_rho, (size_t)w.slots / kSlotTile));
    RQ_TRY(alloc(h, &w.counters, CNT_WORDS));
    RQ_CUDA(h, cudaMemset(w.counters, 0, sizeof(int) * CNT_WORDS));
    if (bf16) {
        RQ_TRY(alloc(h, &w.C, cap * w.ldR));
        RQ_TRY(alloc(h, &w.SREF, cap * w.ldR));
        RQ_TRY(alloc(h, &w.Wc32, (size_t)(n + m) * w.ldkc));
        RQ_TRY(dev_alloc(h, &w.OPND, sizeof(uint16_t) * 7 * (size_t)w.slots * w.ldk + 1024));
        RQ_TRY(dev_alloc(h, &w.CK, sizeof(uint16_t) * 3 * (size_t)w.slots * w.ldkc + 1024));
        RQ_TRY(dev_alloc(h, &w.WB, sizeof(uint16_t) * (size_t)nr * 3 * w.Rpad * w.ldk + 1024));
        RQ_TRY(dev_alloc(h, &w.WCB, sizeof(uint16_t) * 3 * (size_t)w.npad * w.ldkc + 1024));
        RQ_TRY(alloc(h, &w.chunk_sync, tc_sync_words(h)));   // layer counters, done counters
        RQ_CUDA(h, cudaMemset(w.chunk_sync, 0, sizeof(unsigned) * tc_sync_words(h)));
    } else {
        RQ_TRY(alloc(h, &w.S32, 2 * (size_t)w.slots * w.ldk));
        RQ_TRY(alloc(h, &w.CK32, (size_t)w.slots * w.ldkc));
        RQ_TRY(alloc(h, &w.Wc32, (size_t)(n + m) * w.ldkc));
    }
    RQ_TRY(batch_tail_alloc(h));
    RQ_CUDA(h, cudaMallocHost(reinterpret_cast<void**>(&w.cnt_host), sizeof(int) * CNT_WORDS));
    RQ_CUDA(h, cudaMallocHost(reinterpret_cast<void**>(&w.info_host), sizeof(relu_qp_info) * cap));
    RQ_CUDA(h, cudaEventCreateWithFlags(&w.ev_cnt, cudaEventDisableTiming));
    return RELU_QP_OK;
}

// Tuning layout: the first `active_tiles` tiles hold `per_tile` QPs each (a prefix
// of the tile, as the regrouping leaves it).
__global__ void tune_perm_kernel(int slots, int cap, int active_tiles, int per_tile, int* perm, int* tile_rho,
                                 int* counters) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < slots; s += gridDim.x * blockDim.x) {
        const bool in = s / kSlotTile < active_tiles && s % kSlotTile < per_tile && s < cap;
        perm[s] = in ? s : -1;
        if (s % kSlotTile == 0) tile_rho[s / kSlotTile] = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        counters[CNT_TILES] = active_tiles;
        counters[CNT_ACTIVE] = min(cap, active_tiles * per_tile);
    }
}

// Choose the refined layer's configuration (K split over a cluster, tile
// width) for every number of active slot tiles by timing what a chunk would
// run: the persistent chunk kernel where the tiles fit one wave, else one
// launch per layer.  Counts of one or two tiles are timed with tiles that hold
// 48 QPs each (the convergence tail); larger counts with full tiles.  State
// values do not matter here; every buffer the layers touch is re-initialised by
// the next solve.  Where a configuration fits the chunk kernel, only those are
// timed, the two narrowest of each K split: over eleven problems (n + m from 160
// to 3200, up to 11 tiles) no other was ever fastest by more than 0.1 %, and they
// were three quarters of the tuning.  RELU_QP_TUNE_LOG=1 prints the measurements to stderr.
int tc_tune(relu_qp_t h) {
    BatchWork& w = h->bw;
    BatchParams p = layer_params(h, base_params(h));
    const size_t opart = (size_t)w.slots * w.ldk;
    __nv_bfloat16* OP = static_cast<__nv_bfloat16*>(w.OPND);
    p.flags = EPI_REFINE;
    p.Dhi = OP + 2 * opart;
    p.Dlo = OP + 3 * opart;
    p.CK = static_cast<__nv_bfloat16*>(w.CK);
    const int tiles = w.slots / kSlotTile;
    const char* log_env = std::getenv("RELU_QP_TUNE_LOG");
    const bool log = log_env && log_env[0] == '1';
    std::vector<LayerCfg> cfgs;
    tc_layer_cfgs(h, cfgs);
    // measured tile counts: every count up to 12 (1024 QPs regrouped over 3 bank entries take
    // 8 to 11), then every 4th up to 32, then every 16th
    std::vector<int> counts;
    for (int t = 1; t <= tiles; ++t)
        if (t <= 12 || (t <= 32 && t % 4 == 0) || t % 16 == 0 || t == tiles) counts.push_back(t);
    std::vector<LayerCfg> table(tiles + 1, cfgs[0]);
    for (int t : counts) {
        const int per_tile = t <= 2 ? 48 : kSlotTile;
        tune_perm_kernel<<<ceil_div(w.slots, 256), 256, 0, h->stream>>>(w.slots, w.cap, t, per_tile, w.perm,
                                                                         w.tile_rho, w.counters);
        RQ_CUDA(h, cudaGetLastError());
        float best = 1e30f;
        LayerCfg best_c = cfgs[0];
        std::vector<LayerCfg> timed;   // (cfgs lists each split's widths in increasing order)
        for (const LayerCfg& c : cfgs)
            if (tc_chunk_fits(h, c, t) &&
                std::count_if(timed.begin(), timed.end(), [&](const LayerCfg& o) { return o.ks == c.ks; }) < 2)
                timed.push_back(c);
        for (const LayerCfg& c : timed.empty() ? cfgs : timed) {
            RQ_TRY(tc_set_layer_cfg(h, c));
            float ms = 0.f;
            int layers = 0;
            bool chunked = false;
            if (w.chunk_sync) {
                RQ_CUDA(h, cudaMemsetAsync(w.chunk_sync, 0, sizeof(unsigned) * tc_sync_words(h), h->stream));
                const int rc = tc_chunk(h, p, 2, 0u, t);    // warm-up (and eligibility)
                if (rc == RELU_QP_OK) {
                    RQ_CUDA(h, cudaMemsetAsync(w.chunk_sync, 0, sizeof(unsigned) * tc_sync_words(h), h->stream));
                    RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
                    RQ_TRY(tc_chunk(h, p, 8, 0u, t));
                    RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
                    layers = 8;
                    chunked = true;
                } else if (rc != RELU_QP_ERR_UNSUPPORTED) {
                    return rc;
                }
            }
            if (!chunked) {
                RQ_TRY(tc_layer(h, p, 0, tiles, t));
                RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
                RQ_TRY(tc_layer(h, p, 0, tiles, t));
                for (int rep = 1; rep < 4; ++rep) RQ_TRY(tc_layer(h, p, 0, tiles, t, true));
                RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
                layers = 4;
            }
            RQ_CUDA(h, cudaEventSynchronize(h->ev1));
            int site = 0;
            if (tc_error(h, &site))
                return fail(h, RELU_QP_ERR_TIMEOUT,
                            "tensor-core wait " + std::to_string(site) + " passed its deadline while tuning (tiles " +
                                std::to_string(t) + ", ks " + std::to_string(c.ks) + ", bn " + std::to_string(c.bn) +
                                (chunked ? ", chunk kernel)" : ", one launch per layer)"));
            RQ_CUDA(h, cudaEventElapsedTime(&ms, h->ev0, h->ev1));
            ms /= layers;
            if (log)
                std::fprintf(stderr, "relu_qp tune: n=%d m=%d tiles=%d qps/tile=%d ks=%d bn=%d %s us=%.2f\n", h->n,
                             h->m, t, per_tile, c.ks, c.bn, chunked ? "chunk" : "layer", 1e3f * ms);
            if (ms < best) {
                best = ms;
                best_c = c;
            }
        }
        for (int u = t; u <= tiles; ++u) table[u] = best_c;   // until the next measured count
        if (t == 1 && tc_small_eligible(h, per_tile, 1)) {
            // the resident-weight kernel for one tile of few QPs against the best tiled one
            RQ_CUDA(h, cudaMemsetAsync(w.chunk_sync, 0, sizeof(unsigned) * tc_sync_words(h), h->stream));
            int rc = tc_small(h, p, 2, 0u, per_tile, 1);
            if (rc == RELU_QP_OK) {
                RQ_CUDA(h, cudaMemsetAsync(w.chunk_sync, 0, sizeof(unsigned) * tc_sync_words(h), h->stream));
                RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
                RQ_TRY(tc_small(h, p, 8, 0u, per_tile, 1));
                RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
                RQ_CUDA(h, cudaEventSynchronize(h->ev1));
                int site = 0;
                if (tc_error(h, &site))
                    return fail(h, RELU_QP_ERR_TIMEOUT, "tensor-core wait " + std::to_string(site) +
                                                            " passed its deadline while tuning (resident-weight kernel)");
                float ms = 0.f;
                RQ_CUDA(h, cudaEventElapsedTime(&ms, h->ev0, h->ev1));
                ms /= 8;
                if (log)
                    std::fprintf(stderr, "relu_qp tune: n=%d m=%d tiles=1 qps/tile=%d resident-weight us=%.2f\n", h->n,
                                 h->m, per_tile, 1e3f * ms);
                tc_small_set(h, ms < best);
            } else if (rc != RELU_QP_ERR_UNSUPPORTED) {
                return rc;
            }
        }
    }
    tune_perm_kernel<<<ceil_div(w.slots, 256), 256, 0, h->stream>>>(w.slots, w.cap, tiles, kSlotTile, w.perm,
                                                                     w.tile_rho, w.counters);
    RQ_CUDA(h, cudaGetLastError());
    RQ_TRY(tc_set_layer_table(h, table));
    if (log) {
        std::fprintf(stderr, "relu_qp tune: chose (ks, bn) by active tiles:");
        for (int t = 1; t <= tiles; ++t) std::fprintf(stderr, " (%d,%d)", table[t].ks, table[t].bn);
        std::fprintf(stderr, "\n");
    }
    if (tc_error(h)) return fail(h, RELU_QP_ERR_TIMEOUT, "tensor-core kernel wait passed its deadline while tuning");
    RQ_CUDA(h, cudaMemsetAsync(w.RED, 0, sizeof(unsigned) * (size_t)w.cap * RW_WORDS, h->stream));
    RQ_CUDA(h, cudaMemsetAsync(w.counters, 0, sizeof(int) * CNT_WORDS, h->stream));
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    return RELU_QP_OK;
}

void batch_release(relu_qp_t h) {
    if (h->bw.tc) tc_release(h);
    if (h->bw.cnt_host) cudaFreeHost(h->bw.cnt_host);
    if (h->bw.ev_cnt) cudaEventDestroy(h->bw.ev_cnt);
    if (h->bw.info_host) cudaFreeHost(h->bw.info_host);
    h->bw.cnt_host = nullptr;
    h->bw.info_host = nullptr;
    h->bw.ev_cnt = nullptr;
}

// After the FP64 stage: FP32 check matrix (FP32 backend) or tensor maps and
// tile tuning (BF16 backend).
int batch_finish_setup(relu_qp_t h) {
    BatchWork& w = h->bw;
    if (w.prec == RELU_QP_PREC_BF16X3) {
        RQ_TRY(tc_prepare(h));
        RQ_TRY(tc_tune(h));
    }
    const int ldp = (int)round_up(h->n, 4), ldt = (int)round_up(h->m > 0 ? h->m : 1, 4);
    const size_t total = (size_t)(h->n + h->m) * w.ldkc;
    int g = (int)std::min<size_t>((total + 255) / 256, 8192);
    build_wc32_kernel<<<g, 256, 0, h->stream>>>(h->P32, h->A32, ldp, h->At32, ldt, h->n, h->m, w.n64, w.ldkc,
                                                w.Wc32);
    RQ_CUDA(h, cudaGetLastError());
    return RELU_QP_OK;
}

int batch_update(relu_qp_t h, int B, const float* Q, const float* L, const float* U) {
    BatchWork& w = h->bw;
    const int n = h->n, m = h->m, R = h->R;
    if (Q) RQ_TRY(copy_rows_in(h, w.Q, w.ldn, Q, B, n));
    if (L && m > 0) RQ_TRY(copy_rows_in(h, w.L, w.ldm, L, B, m));
    if (U && m > 0) RQ_TRY(copy_rows_in(h, w.U, w.ldm, U, B, m));
    // scaled handles: q -> c D q, l -> E l, u -> E u
    if (Q) RQ_TRY(scale_rows(h, w.Q, B, n, w.ldn, h->sc_q));
    if (L && m > 0) RQ_TRY(scale_rows(h, w.L, B, m, w.ldm, h->sc_e));
    if (U && m > 0) RQ_TRY(scale_rows(h, w.U, B, m, w.ldm, h->sc_e));
    if (Q) {
        Maps maps;
        for (int r = 0; r < h->nr; ++r)
            maps.add(R, h->be[r].Bop, n, 1.f, nullptr, w.BIAS + (size_t)r * w.cap * w.ldR, w.ldR, n, w.nP - n);
        RQ_TRY(maps.run(h, B, n, w.Q, w.ldn));
        row_absmax_kernel<<<ceil_div(B * 32, 256), 256, 0, h->stream>>>(w.Q, B, n, w.ldn, h->sc_rx, w.QN);
        RQ_CUDA(h, cudaGetLastError());
        ++h->launches;
    }
    w.B = B;
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    return RELU_QP_OK;
}

int batch_set_parametric(relu_qp_t h, int nx, const double* F, const double* E, const double* l0,
                         const double* u0) {
    BatchWork& w = h->bw;
    const int n = h->n, m = h->m, R = h->R;
    if (w.nx != nx) {
        w.nx = nx;
        w.ldx = (int)round_up(nx, 4);
        RQ_TRY(alloc(h, &w.F32, (size_t)n * w.ldx));
        RQ_TRY(alloc(h, &w.Ft32, (size_t)nx * w.ldn));
        RQ_TRY(alloc(h, &w.E32, (size_t)(m > 0 ? m : 1) * w.ldx));
        RQ_TRY(alloc(h, &w.l0, (size_t)(m > 0 ? m : 1)));
        RQ_TRY(alloc(h, &w.u0, (size_t)(m > 0 ? m : 1)));
        RQ_TRY(alloc(h, &w.X0, (size_t)w.cap * w.ldx));
        for (int r = 0; r < h->nr; ++r) RQ_TRY(alloc(h, &w.G[r], (size_t)R * w.ldx));
    }
    // scaled handles: F -> c D F, E -> E E, l0 -> E l0, u0 -> E u0 (in FP64)
    const bool sc = h->scaled != 0;
    std::vector<float> f((size_t)n * w.ldx, 0.f), ft((size_t)nx * w.ldn, 0.f);
    for (int i = 0; i < n; ++i) {
        const double fi = sc ? h->sC * h->sD[i] : 1.0;
        for (int k = 0; k < nx; ++k) {
            f[(size_t)i * w.ldx + k] = (float)(fi * F[(size_t)i * nx + k]);
            ft[(size_t)k * w.ldn + i] = (float)(fi * F[(size_t)i * nx + k]);
        }
    }
    RQ_CUDA(h, cudaMemcpy(w.F32, f.data(), sizeof(float) * f.size(), cudaMemcpyHostToDevice));
    RQ_CUDA(h, cudaMemcpy(w.Ft32, ft.data(), sizeof(float) * ft.size(), cudaMemcpyHostToDevice));
    if (m > 0) {
        std::vector<float> e((size_t)m * w.ldx, 0.f), lo(m), up(m);
        for (int i = 0; i < m; ++i) {
            const double ei = sc ? h->sE[i] : 1.0;
            for (int k = 0; k < nx; ++k) e[(size_t)i * w.ldx + k] = (float)(ei * E[(size_t)i * nx + k]);
            lo[i] = (float)(ei * l0[i]);
            up[i] = (float)(ei * u0[i]);
        }
        RQ_CUDA(h, cudaMemcpy(w.E32, e.data(), sizeof(float) * e.size(), cudaMemcpyHostToDevice));
        RQ_CUDA(h, cudaMemcpy(w.l0, lo.data(), sizeof(float) * m, cudaMemcpyHostToDevice));
        RQ_CUDA(h, cudaMemcpy(w.u0, up.data(), sizeof(float) * m, cudaMemcpyHostToDevice));
    }
    for (int r = 0; r < h->nr; ++r) {   // G_r = Bop_r F
        Maps maps;
        maps.add(nx, w.Ft32, w.ldn, 1.f, nullptr, w.G[r], w.ldx);
        RQ_TRY(maps.run(h, R, n, h->be[r].Bop, n));
    }
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    return RELU_QP_OK;
}

int batch_update_x0(relu_qp_t h, int B, const float* X0) {
    BatchWork& w = h->bw;
    const int n = h->n, m = h->m, R = h->R, nx = w.nx;
    RQ_TRY(copy_rows_in(h, w.X0, w.ldx, X0, B, nx));
    Maps maps;
    maps.add(n, w.F32, w.ldx, 1.f, nullptr, w.Q, w.ldn);
    maps.add(m, w.E32, w.ldx, -1.f, w.l0, w.L, w.ldm, 0, 0, w.u0, w.U);
    for (int r = 0; r < h->nr; ++r)
        maps.add(R, w.G[r], w.ldx, 1.f, nullptr, w.BIAS + (size_t)r * w.cap * w.ldR, w.ldR, n, w.nP - n);
    RQ_TRY(maps.run(h, B, nx, w.X0, w.ldx));
    row_absmax_kernel<<<ceil_div(B * 32, 256), 256, 0, h->stream>>>(w.Q, B, n, w.ldn, h->sc_rx, w.QN);
    RQ_CUDA(h, cudaGetLastError());
    ++h->launches;
    w.B = B;
    return RELU_QP_OK;
}

// Between two chunks one kernel follows another on the same few hundred QPs, each of a few us: all
// of them, the layers included, are programmatic dependent launches, so that a kernel is resident
// and set up when the one before it ends.  Each waits (griddep_wait) before it reads what an
// earlier kernel of the chain wrote and lets its successor start only after that, or reads before
// only what a kernel wrote that the chain has already waited for (counters, perm and tile_rho, by
// the chunk's layers and checks).  Batch of 64, n = 800:
// 3.90 -> 3.65 ms.

// Regroup the active QPs among the first nqp QP indices into slots.
int assign_slots(relu_qp_t h, int nqp, bool pdl) {
    BatchWork& w = h->bw;
    RQ_TRY(launch_pdl(h, batch_assign_kernel, dim3(1), 1024, 0, pdl, nqp, w.slots, h->nr, (const int*)w.status,
                      (const int*)w.rho_idx, w.perm, w.tile_rho, w.counters));
    ++h->launches;
    return RELU_QP_OK;
}

// Write the operand of the next chunk's first layer.
int fill_slots(relu_qp_t h, const BatchParams& p, bool pdl) {
    BatchWork& w = h->bw;
    const bool bf16 = w.prec == RELU_QP_PREC_BF16X3;
    const size_t opart = (size_t)w.slots * w.ldk;
    __nv_bfloat16* OP = static_cast<__nv_bfloat16*>(w.OPND);
    RQ_TRY(launch_pdl(h, batch_fill_kernel, dim3((int)((size_t)w.slots * (w.ldk / 4) / 256 + 1)), 256, 0, pdl,
                      layer_params(h, p), (const int*)w.rho_idx, bf16 ? nullptr : w.S32,
                      bf16 ? OP + 4 * opart : nullptr, opart));
    ++h->launches;
    return RELU_QP_OK;
}

// The layer counters of the chunk kernels, at zero before a solve (a chunk leaves them so; one
// that gave up does not).
int zero_chunk_sync(relu_qp_t h) {
    BatchWork& w = h->bw;
    if (w.chunk_sync) RQ_CUDA(h, cudaMemsetAsync(w.chunk_sync, 0, sizeof(unsigned) * tc_sync_words(h), h->stream));
    return RELU_QP_OK;
}

// `len` layers of one chunk over the slots of the last regroup; with `check`
// the last layer also writes x into the check operand.  `active` is the
// number of QPs in the batch (for the tile-width choice and the FLOP count).
int run_layers(relu_qp_t h, const BatchParams& p, int len, bool check, int active, int tiles_now,
               size_t& prof_used, int j_begin = 0, int j_end = 1 << 30) {
    BatchWork& w = h->bw;
    const int R = h->R;
    const bool bf16 = w.prec == RELU_QP_PREC_BF16X3;
    const int tiles_max = w.slots / kSlotTile;
    const size_t opart = (size_t)w.slots * w.ldk;
    __nv_bfloat16* OP = static_cast<__nv_bfloat16*>(w.OPND);
    W32Ptrs wp{};
    for (int r = 0; r < h->nr; ++r) wp.w[r] = h->be[r].Wt;
    // profiling: one event pair around the refined layers of the chunk (events
    // between them would break the programmatic overlap of consecutive layers)
    const bool timed = h->prof_on && bf16 && len > 1 && prof_used + 2 <= h->prof_ev.size();
    if (!bf16 && j_begin == 0 && j_end >= len) {
        BatchParams q = layer_params(h, p);
        q.flags = 0;
        q.Sin = w.S32;
        q.CK32 = w.CK32;
        const bool timed32 = h->prof_on && prof_used + 2 <= h->prof_ev.size();
        if (timed32) RQ_CUDA(h, cudaEventRecord(h->prof_ev[prof_used], h->stream));
        const int rc = chunk32(h, q, wp, tiles_max, active, len, EPI_LAST | (check ? EPI_CHECK : 0u));
        if (rc != RELU_QP_ERR_UNSUPPORTED) {
            RQ_TRY(rc);
            ++h->launches;
            h->layer_launches += len;
            h->layer_flops += len * 2.0 * (double)R * (double)R * (double)active;
            if (timed32) {
                RQ_CUDA(h, cudaEventRecord(h->prof_ev[prof_used + 1], h->stream));
                h->prof_span_launches.push_back(len);
                prof_used += 2;
            }
            return RELU_QP_OK;
        }
    }
    for (int j = j_begin; j < std::min(len, j_end); ++j) {
        BatchParams q = layer_params(h, p);
        q.flags = 0;
        if (j == len - 1) q.flags |= EPI_LAST | (check ? EPI_CHECK : 0u);
        if (bf16) {
            q.flags |= EPI_REFINE | (j == 0 ? EPI_REBASE : 0u);
            q.Dhi = OP + (size_t)(2 * (j & 1)) * opart;
            q.Dlo = q.Dhi + opart;
            q.CK = static_cast<__nv_bfloat16*>(w.CK);
            if (j == 1 && w.chunk_sync) {
                // layers 1 .. len-1 in one persistent launch when the tile's CTAs fit in one wave:
                // the resident-weight kernel for one tile of few QPs (when the tuner chose it),
                // else the tiled chunk kernel
                BatchParams qc = q;
                qc.flags = 0;
                if (timed) RQ_CUDA(h, cudaEventRecord(h->prof_ev[prof_used], h->stream));
                int rc = RELU_QP_ERR_UNSUPPORTED;
                if (tc_small_chosen(h) && tc_small_eligible(h, active, tiles_now)) {
                    rc = tc_small(h, qc, len - 1, EPI_LAST | (check ? EPI_CHECK : 0u), active, tiles_now);
                    if (rc != RELU_QP_OK && rc != RELU_QP_ERR_UNSUPPORTED) return rc;
                    if (rc == RELU_QP_OK) ++h->resident_launches;
                }
                if (rc != RELU_QP_OK) rc = tc_chunk(h, qc, len - 1, EPI_LAST | (check ? EPI_CHECK : 0u), tiles_now);
                if (rc == RELU_QP_OK) {
                    h->launches += 1;
                    h->layer_launches += len - 1;
                    h->layer_flops += (len - 1) * 2.0 * 3.0 * (double)R * (double)R * (double)active;
                    if (timed) {
                        RQ_CUDA(h, cudaEventRecord(h->prof_ev[prof_used + 1], h->stream));
                        h->prof_span_launches.push_back(len - 1);
                        prof_used += 2;
                    }
                    break;
                }
                if (rc != RELU_QP_ERR_UNSUPPORTED) return rc;
                // refused: one launch per layer below (which records the span's start again)
            }
            // operand set read by this layer: 4..6 = s (3-way), else pair ((j-1)&1)
            if (timed && j == 1) RQ_CUDA(h, cudaEventRecord(h->prof_ev[prof_used], h->stream));
            RQ_TRY(tc_layer(h, q, j == 0 ? -1 : ((j - 1) & 1), tiles_max,
                            tiles_now > 0 ? tiles_now : w.tiles_hint > 0 ? w.tiles_hint : ceil_div(active, kSlotTile) + h->nr - 1,
                            j > 0));
            ++h->launches;
            if (j > 0) {
                ++h->layer_launches;
                // three BF16 products of the (n+m) x (n+m) factored layer per active QP
                h->layer_flops += 2.0 * 3.0 * (double)R * (double)R * (double)active;
            }
            if (timed && j == len - 1) {
                RQ_CUDA(h, cudaEventRecord(h->prof_ev[prof_used + 1], h->stream));
                h->prof_span_launches.push_back(len - 1);
                prof_used += 2;
            }
        } else {
            q.Sin = w.S32 + (size_t)(j & 1) * opart;
            q.Sout = w.S32 + (size_t)((j + 1) & 1) * opart;
            q.CK32 = w.CK32;
            const bool timed32 = h->prof_on && prof_used + 2 <= h->prof_ev.size();
            if (timed32) RQ_CUDA(h, cudaEventRecord(h->prof_ev[prof_used], h->stream));
            RQ_TRY(layer32(h, q, wp, tiles_max, active, true));
            ++h->launches;
            ++h->layer_launches;
            h->layer_flops += 2.0 * (double)R * (double)R * (double)active;   // one FP32 product per QP
            if (timed32) {
                RQ_CUDA(h, cudaEventRecord(h->prof_ev[prof_used + 1], h->stream));
                h->prof_span_launches.push_back(1);
                prof_used += 2;
            }
        }
    }
    return RELU_QP_OK;
}

// Residual products of a check: [P; A] x, then A^T lam_std (Eqs. primal, dual).
// tiles_now: slot tiles in use when the host knows them (> 0), else a bound
// from the active QP count is used.
int run_check(relu_qp_t h, const BatchParams& p, int active, int tiles_now) {
    BatchWork& w = h->bw;
    const int tiles_max = w.slots / kSlotTile;
    BatchParams q = layer_params(h, p);
    if (w.prec == RELU_QP_PREC_BF16X3) {
        q.CK = static_cast<__nv_bfloat16*>(w.CK);
        const int active_tiles =
            tiles_now > 0 ? tiles_now
                          : w.tiles_hint > 0 ? w.tiles_hint : std::min(tiles_max, ceil_div(active, kSlotTile) + h->nr - 1);
        RQ_TRY(tc_check(h, q, 1, tiles_max, active_tiles));
        RQ_TRY(tc_check(h, q, 2, tiles_max, active_tiles));
    } else {
        q.CK32 = w.CK32;
        RQ_TRY(check32(h, q, w.Wc32, tiles_max, active, 1));
        RQ_TRY(check32(h, q, w.Wc32, tiles_max, active, 2));
    }
    h->launches += 2;
    return RELU_QP_OK;
}

int nearest_rho(relu_qp_t h, double rho) {
    int best = 0;
    double bd = 1e300;
    for (int k = 0; k < h->nr; ++k) {
        const double d = std::fabs(std::log(rho) - std::log(h->bank[k]));
        if (d < bd) { bd = d; best = k; }
    }
    return best;
}

int batch_solve(relu_qp_t h, int B, const float* Xw, const float* Lw, const int* rw, double eps_abs,
                double eps_rel, int max_iter, float* Xo, float* Zo, float* Lo, relu_qp_info* infos) {
    BatchWork& w = h->bw;
    const int n = h->n, m = h->m;
    const bool bf16 = w.prec == RELU_QP_PREC_BF16X3;
    BatchParams p = base_params(h);
    const int tiles_max = w.slots / kSlotTile;
    // ---- start state ----
    const int rho0 = nearest_rho(h, h->opts.rho0);
    h->prof_span_launches.clear();
    int* rw_dev = nullptr;
    if (rw) {
        RQ_CUDA(h, cudaMemcpyAsync(w.iters, rw, sizeof(int) * B, cudaMemcpyDefault, h->stream));
        rw_dev = w.iters;   // staged; batch_init copies it into rho_idx before resetting iters
    }
    // scaled handles: warm starts xb = x / D, lamb = c lam / E
    if (Xw) {
        RQ_TRY(copy_rows_in(h, w.Y, w.ldn, Xw, B, n));
        RQ_TRY(scale_rows(h, w.Y, B, n, w.ldn, h->sc_xi));
        Maps maps;
        maps.add(m, h->A32, (int)round_up(n, 4), 1.f, nullptr, w.AY, w.ldm);
        RQ_TRY(maps.run(h, B, n, w.Y, w.ldn));
    }
    if (Lw && m > 0) {
        RQ_TRY(copy_rows_in(h, w.LSTD, w.ldm, Lw, B, m));
        RQ_TRY(scale_rows(h, w.LSTD, B, m, w.ldm, h->sc_li));
    }
    RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
    RQ_CUDA(h, cudaMemsetAsync(w.counters + CNT_ERR, 0, 2 * sizeof(int), h->stream));
    RQ_TRY(zero_chunk_sync(h));
    batch_init_kernel<<<w.cap, kInitThreads, 0, h->stream>>>(p, B, Xw != nullptr, Lw != nullptr && m > 0,
                                                                        rw_dev, rho0, w.status, w.rho_idx, w.iters,
                                                                        w.nsw);
    RQ_CUDA(h, cudaGetLastError());
    ++h->launches;
    RQ_TRY(assign_slots(h, B, false));
    RQ_TRY(fill_slots(h, p, true));
    const int ci = h->opts.check_interval;
    const int chunk = ci > 0 ? ci : 25;
    int it = 0;
    int active = B;              // QPs in the batch (known to the host after each check)
    // slot tiles in use: exact at a cold start (every QP in the starting bank entry's
    // group) and after each check, an upper bound after a warm start
    int tiles_now = rw ? std::min(tiles_max, ceil_div(B, kSlotTile) + h->nr - 1) : ceil_div(B, kSlotTile);
    size_t prof_used = 0, gap_used = 0;
    bool tail_used = false;
    bool first_done = false;     // the chunk's first layer was enqueued before the host's read-back
    while (it < max_iter) {
        const int len = std::min(chunk, max_iter - it);
        const bool last_chunk = it + len == max_iter;
        const bool check = (ci > 0 && (it + len) % ci == 0) || last_chunk;
        RQ_TRY(run_layers(h, p, len, check, active, tiles_now, prof_used, first_done ? 1 : 0));
        first_done = false;
        it += len;
        if (check) {
            RQ_TRY(run_check(h, p, active, tiles_now));
            DecideArgs d{B, it, last_chunk ? 1 : 0, h->opts.adaptive_rho, eps_abs, eps_rel, w.XO, w.ZO, w.LO,
                         w.status, w.iters, w.rho_idx, w.nsw, w.rp, w.rd, 0, max_iter, nullptr, nullptr};
            // the active QPs are the ones in the slots of the last regroup: one block per slot
            const bool by_slot = tiles_now > 0 && tiles_now * kSlotTile < B;
            RQ_TRY(launch_pdl(h, batch_decide_kernel, dim3(by_slot ? tiles_now * kSlotTile : B), kDecideThreads, 0, true, p,
                              d, by_slot ? 1 : 0));
            ++h->launches;
        }
        if (last_chunk) break;
        if (check) {
            RQ_TRY(assign_slots(h, B, true));
            // the host needs the active QP and slot-tile counts of the regroup (they choose
            // the next chunk's kernel); the copy is waited for through an event, and in the
            // split form the next chunk's first (accurate) layer is enqueued before the
            // wait, so that the GPU works during the round trip.  That layer stores only
            // chunk-local data (c, s_ref, r, the operand), never x, Ax, z or lam', so nothing
            // depends on it if the host then stops or hands the last QPs to the tail kernel.
            RQ_CUDA(h, cudaMemcpyAsync(w.cnt_host, w.counters, sizeof(int) * CNT_WORDS, cudaMemcpyDeviceToHost,
                                       h->stream));
            RQ_CUDA(h, cudaEventRecord(w.ev_cnt, h->stream));
            RQ_TRY(fill_slots(h, p, false));
            const int nlen = std::min(chunk, max_iter - it);
            if (bf16 && nlen > 1) {
                const bool ncheck = (ci > 0 && (it + nlen) % ci == 0) || it + nlen == max_iter;
                RQ_TRY(run_layers(h, p, nlen, ncheck, active, tiles_now, prof_used, 0, 1));
                first_done = true;
            }
            // profiling: how long the GPU then waits for the host
            const bool gap = h->prof_on && gap_used + 2 <= h->gap_ev.size();
            if (gap) RQ_CUDA(h, cudaEventRecord(h->gap_ev[gap_used], h->stream));
            RQ_CUDA(h, cudaEventSynchronize(w.ev_cnt));
            if (gap) {
                RQ_CUDA(h, cudaEventRecord(h->gap_ev[gap_used + 1], h->stream));
                gap_used += 2;
            }
            int cnt[CNT_WORDS];
            std::memcpy(cnt, w.cnt_host, sizeof(cnt));
            if (cnt[CNT_ERR]) break;     // reported below
            if (cnt[CNT_ACTIVE] == 0) break;
            active = cnt[CNT_ACTIVE];
            tiles_now = cnt[CNT_TILES];
            if (active <= kTailMax && w.tail_grid > 0) {
                // the few QPs left finish in one cooperative launch
                DecideArgs d{B, it, 0, h->opts.adaptive_rho, eps_abs, eps_rel, w.XO, w.ZO, w.LO, w.status, w.iters,
                             w.rho_idx, w.nsw, w.rp, w.rd, 0, max_iter, nullptr, nullptr};
                RQ_TRY(batch_tail(h, p, d, active, it, max_iter));
                tail_used = true;
                break;
            }
        } else {
            RQ_TRY(fill_slots(h, p, true));
        }
    }
    if (!bf16)
        RQ_CUDA(h, cudaMemcpyAsync(w.cnt_host, w.counters, sizeof(int) * CNT_WORDS, cudaMemcpyDeviceToHost, h->stream));
    RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    if (bf16) {
        const int e = tc_error(h);
        if (e == RELU_QP_ERR_TIMEOUT) return fail(h, e, "a tensor-core kernel wait passed its deadline");
        if (e) return fail(h, RELU_QP_ERR_CUDA, "a tensor-core kernel found a launch shape it cannot run");
    } else if (w.cnt_host[CNT_ERR]) {
        return fail(h, RELU_QP_ERR_TIMEOUT, "a wait of the FP32 chunk kernel passed its deadline");
    }
    if (tail_used && batch_tail_error(h))
        return fail(h, RELU_QP_ERR_TIMEOUT, "a grid barrier of the convergence-tail kernel passed its deadline");
    for (size_t e = 0; e + 1 < prof_used; e += 2) {
        float ms = 0.f;
        RQ_CUDA(h, cudaEventElapsedTime(&ms, h->prof_ev[e], h->prof_ev[e + 1]));
        h->layer_ms += ms;
        h->layer_timed += h->prof_span_launches[e / 2];
    }
    h->prof_span_launches.clear();
    for (size_t e = 0; e + 1 < gap_used; e += 2) {
        float ms = 0.f;
        RQ_CUDA(h, cudaEventElapsedTime(&ms, h->gap_ev[e], h->gap_ev[e + 1]));
        h->host_gap_ms += ms;
        ++h->host_checks;
    }
    // ---- outputs (scaled handles: x = D xb, z = zb / E, lam = E lamb / c) ----
    RQ_TRY(scale_rows(h, w.XO, B, n, n, h->sc_x));
    if (Zo && m > 0) RQ_TRY(scale_rows(h, w.ZO, B, m, m, h->sc_z));
    if (Lo && m > 0) RQ_TRY(scale_rows(h, w.LO, B, m, m, h->sc_l));
    RQ_CUDA(h, cudaMemcpyAsync(Xo, w.XO, sizeof(float) * B * n, cudaMemcpyDefault, h->stream));
    if (Zo && m > 0) RQ_CUDA(h, cudaMemcpyAsync(Zo, w.ZO, sizeof(float) * B * m, cudaMemcpyDefault, h->stream));
    if (Lo && m > 0) RQ_CUDA(h, cudaMemcpyAsync(Lo, w.LO, sizeof(float) * B * m, cudaMemcpyDefault, h->stream));
    if (infos) {
        pack_info_kernel<<<ceil_div(B, 256), 256, 0, h->stream>>>(B, w.status, w.iters, w.rho_idx, w.nsw, w.rp, w.rd,
                                                                 w.info_host);
        RQ_CUDA(h, cudaGetLastError());
        ++h->launches;
        RQ_CUDA(h, cudaStreamSynchronize(h->stream));
        float ms = 0.f;
        cudaEventElapsedTime(&ms, h->ev0, h->ev1);
        std::memcpy(infos, w.info_host, sizeof(relu_qp_info) * B);
        for (int b = 0; b < B; ++b) infos[b].solve_ms = ms;
    }
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    return RELU_QP_OK;
}

}  // namespace rq

// ===========================================================================
// Continuous batching (serving).  A server holds several problem families,
// each a handle with its own layer bank and batch slots.  Requests (a new
// initial state x0 for one client of one family) wait in a host queue; at
// every step each family admits waiting requests into its free QP slots
// (parametric update of q, l, u, b and a warm start from the client's last
// solution, kept on the device), runs one chunk (check_interval layers, the
// residual check, the stop test and penalty rule) on its own stream, and
// retires the QPs that finished.  Families' chunks overlap on the GPU.
// ===========================================================================
namespace rq {

namespace {

struct ServeDev {
    int *idx = nullptr, *cl = nullptr, *client_of = nullptr, *done = nullptr, *cnt = nullptr;
    float *x0c = nullptr, *Qc = nullptr, *Lc = nullptr, *Uc = nullptr, *Bc = nullptr, *AYc = nullptr, *Xc = nullptr;
    float *out = nullptr;
    float *Wx = nullptr, *Wl = nullptr;
    int *Wr = nullptr, *Wv = nullptr;
};

// Admitted request j goes to QP index idx[j]: warm start from its client's
// last solution (x, lam_std, rho index) if there is one, else cold.
__global__ void serve_admit_kernel(BatchParams p, int k, const int* __restrict__ idx, const int* __restrict__ cl,
                                   const float* __restrict__ Wx, const float* __restrict__ Wl,
                                   const int* __restrict__ Wr, const int* __restrict__ Wv, int rho0, int* status,
                                   int* rho_idx, int* iters, int* nsw, int* client_of, float* Xc) {
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= k) return;
    const int qp = idx[j], c = cl[j];
    const bool warm = c >= 0 && Wv[c] != 0;
    for (int t = lane; t < p.n; t += 32) {
        const float v = warm ? Wx[(size_t)c * p.ldn + t] : 0.f;
        p.Y[(size_t)qp * p.ldn + t] = v;
        Xc[(size_t)j * p.ldn + t] = v;
    }
    for (int i = lane; i < p.ldm; i += 32)
        p.LAM[(size_t)qp * p.ldm + i] = warm && i < p.m ? Wl[(size_t)c * p.ldm + i] : 0.f;
    for (int t = p.n + lane; t < p.ldn; t += 32) p.Y[(size_t)qp * p.ldn + t] = 0.f;   // padding
    if (lane == 0) {
        status[qp] = QP_ACTIVE;
        rho_idx[qp] = warm ? Wr[c] : rho0;
        iters[qp] = 0;
        nsw[qp] = 0;
        client_of[qp] = c;
    }
    if (lane < RW_WORDS) p.RED[(size_t)qp * RW_WORDS + lane] = 0u;
}

// Compact rows of the admitted requests -> their QP rows (q, l, u, every b_r,
// and z = A x for the warm start, which also seeds the carried A x).
__global__ void serve_scatter_kernel(BatchParams p, int k, const int* __restrict__ idx, const float* __restrict__ Qc,
                                     const float* __restrict__ Lc, const float* __restrict__ Uc,
                                     const float* __restrict__ Bc, const float* __restrict__ AYc, float* Q, float* L,
                                     float* U, float* BIAS, float* QN) {
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= k) return;
    const int qp = idx[j];
    float qn = 0.f;
    for (int t = lane; t < p.n; t += 32) {
        const float v = Qc[(size_t)j * p.ldn + t];
        Q[(size_t)qp * p.ldn + t] = v;
        qn = fmaxf(qn, fabsf(p.rsx ? v * p.rsx[t] : v));   // |q|_inf of the original problem
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) qn = fmaxf(qn, __shfl_xor_sync(0xffffffffu, qn, o));
    if (lane == 0) QN[qp] = qn;
    for (int i = lane; i < p.m; i += 32) {
        const size_t o = (size_t)qp * p.ldm + i, oc = (size_t)j * p.ldm + i;
        L[o] = Lc[oc];
        U[o] = Uc[oc];
        p.AY[o] = AYc[oc];
        p.Z[o] = AYc[oc];
    }
    for (int i = p.m + lane; i < p.ldm; i += 32) {   // padding
        p.AY[(size_t)qp * p.ldm + i] = 0.f;
        p.Z[(size_t)qp * p.ldm + i] = 0.f;
    }
    for (int r = 0; r < p.nr; ++r)
        for (int t = lane; t < p.ldR; t += 32)
            BIAS[((size_t)r * p.cap + qp) * p.ldR + t] = Bc[((size_t)r * p.cap + j) * p.ldR + t];
}

// Finished QPs: pack [x | qp, status, iters, rho, switches, r_prim, r_dual] per
// result, store the client's warm start, free the QP index.
__global__ void serve_gather_kernel(BatchParams p, const int* __restrict__ done, const int* __restrict__ cnt,
                                    const int* __restrict__ client_of, int* status, const int* __restrict__ iters,
                                    const int* __restrict__ rho_idx, const int* __restrict__ nsw,
                                    const float* __restrict__ rp, const float* __restrict__ rd,
                                    const float* __restrict__ XO, const float* __restrict__ sx, float* Wx, float* Wl,
                                    int* Wr, int* Wv, float* out, int ldo) {
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= *cnt) return;
    const int qp = done[j];
    const int c = client_of[qp];
    float* o = out + (size_t)j * ldo;
    // x of the original problem (x = D xb when scaled); the client's warm start stays scaled
    for (int t = lane; t < p.n; t += 32) o[t] = sx ? XO[(size_t)qp * p.n + t] * sx[t] : XO[(size_t)qp * p.n + t];
    if (c >= 0) {
        for (int t = lane; t < p.n; t += 32) Wx[(size_t)c * p.ldn + t] = p.Y[(size_t)qp * p.ldn + t];
        for (int i = lane; i < p.m; i += 32) Wl[(size_t)c * p.ldm + i] = p.LSTD[(size_t)qp * p.ldm + i];
    }
    if (lane == 0) {
        o[p.n + 0] = __int_as_float(qp);
        o[p.n + 1] = __int_as_float(status[qp]);
        o[p.n + 2] = __int_as_float(iters[qp]);
        o[p.n + 3] = __int_as_float(rho_idx[qp]);
        o[p.n + 4] = __int_as_float(nsw[qp]);
        o[p.n + 5] = rp[qp];
        o[p.n + 6] = rd[qp];
        if (c >= 0) {
            Wr[c] = rho_idx[qp];
            Wv[c] = 1;
        }
        status[qp] = QP_UNUSED;
    }
}

}  // namespace

struct ServeRequest {
    int client;
    long long tag;
    double t_submit;
    std::vector<float> x0;
};

struct ServeFamily {
    relu_qp_t h = nullptr;
    cudaStream_t stream = nullptr, saved_stream = nullptr;
    int cap = 0, clients = 0, active = 0, ldo = 0, rho0 = 0;
    std::deque<ServeRequest> queue;
    std::vector<int> free_idx;
    std::vector<long long> tag_of;
    std::vector<double> t_submit_of;
    std::vector<int> client_of;
    ServeDev d;
    float* h_x0c = nullptr;
    int *h_idx = nullptr, *h_cl = nullptr, *h_cnt = nullptr;
    float* h_out = nullptr;
    cudaEvent_t ev = nullptr;
    bool launched = false;
    std::vector<void*> dev_allocs, host_allocs;
    size_t dev_bytes = 0;          // the server's device buffers for this family
    size_t slot_bytes = 0;         // device bytes charged per admitted request
};

struct ServeResult {
    relu_qp_result r;
    std::vector<float> x;
};

}  // namespace rq

struct relu_qp_server_s {
    std::vector<rq::ServeFamily> fam;
    std::deque<rq::ServeResult> results;
    long long budget = 0;          // device-memory budget (0: slots only)
    size_t fixed = 0;              // every family's bank and fixed buffers
    size_t in_use = 0;             // bytes charged by the requests in slots
    double eps_abs = 1e-3, eps_rel = 0.0;
    int max_iter = 4000;
    std::chrono::steady_clock::time_point t0;
    std::string err;
    double now() const {
        return std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
};

namespace rq {

namespace {

int sfail(relu_qp_server_t s, int code, const std::string& msg) {
    s->err = msg;
    return code;
}

template <typename T>
int sdev(relu_qp_server_t s, ServeFamily& f, T** p, size_t count) {
    void* q = nullptr;
    const cudaError_t e = cudaMalloc(&q, count * sizeof(T) + 16);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return sfail(s, RELU_QP_ERR_OOM, std::string("server device buffer: ") + cudaGetErrorString(e));
    }
    cudaMemset(q, 0, count * sizeof(T) + 16);
    f.dev_allocs.push_back(q);
    f.dev_bytes += count * sizeof(T) + 16;
    *p = static_cast<T*>(q);
    return RELU_QP_OK;
}

template <typename T>
int shost(relu_qp_server_t s, ServeFamily& f, T** p, size_t count) {
    void* q = nullptr;
    const cudaError_t e = cudaMallocHost(&q, count * sizeof(T) + 16);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return sfail(s, RELU_QP_ERR_OOM, std::string("server pinned buffer: ") + cudaGetErrorString(e));
    }
    f.host_allocs.push_back(q);
    *p = static_cast<T*>(q);
    return RELU_QP_OK;
}

#define RQ_SCUDA(s, call)                                                                        \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess) {                                                                 \
            cudaGetLastError();                                                                  \
            return sfail((s), RELU_QP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
        }                                                                                        \
    } while (0)

int family_launch(relu_qp_server_t s, ServeFamily& f) {
    relu_qp_t h = f.h;
    BatchWork& w = h->bw;
    const int n = h->n, m = h->m, R = h->R, nx = w.nx;
    BatchParams p = base_params(h);
    // ---- admission: a free slot, and (with a budget) room for the request's
    // slot bytes that no older waiting request of another family needs ----
    int k = (int)std::min(f.queue.size(), f.free_idx.size());
    if (s->budget > 0 && k > 0) {
        const size_t room = (size_t)s->budget - s->fixed;
        // the oldest request waiting in another family that has a free slot
        double t_old = 1e300;
        size_t b_old = 0;
        for (const auto& g : s->fam) {
            if (&g == &f || g.queue.empty() || g.free_idx.empty()) continue;
            if (g.queue.front().t_submit < t_old) {
                t_old = g.queue.front().t_submit;
                b_old = g.slot_bytes;
            }
        }
        int fit = 0;
        size_t used = s->in_use;
        while (fit < k) {
            const size_t need = used + f.slot_bytes + (f.queue[fit].t_submit > t_old ? b_old : 0);
            if (need > room) break;
            used += f.slot_bytes;
            ++fit;
        }
        k = fit;
    }
    if (k > 0) {
        s->in_use += (size_t)k * f.slot_bytes;
        for (int j = 0; j < k; ++j) {
            ServeRequest rq_ = std::move(f.queue.front());
            f.queue.pop_front();
            const int qp = f.free_idx.back();
            f.free_idx.pop_back();
            f.h_idx[j] = qp;
            f.h_cl[j] = rq_.client;
            std::memcpy(f.h_x0c + (size_t)j * w.ldx, rq_.x0.data(), sizeof(float) * nx);
            f.tag_of[qp] = rq_.tag;
            f.t_submit_of[qp] = rq_.t_submit;
            f.client_of[qp] = rq_.client;
        }
        f.active += k;
        RQ_SCUDA(s, cudaMemcpyAsync(f.d.x0c, f.h_x0c, sizeof(float) * k * w.ldx, cudaMemcpyHostToDevice, f.stream));
        RQ_SCUDA(s, cudaMemcpyAsync(f.d.idx, f.h_idx, sizeof(int) * k, cudaMemcpyHostToDevice, f.stream));
        RQ_SCUDA(s, cudaMemcpyAsync(f.d.cl, f.h_cl, sizeof(int) * k, cudaMemcpyHostToDevice, f.stream));
        serve_admit_kernel<<<ceil_div(k * 32, 256), 256, 0, f.stream>>>(p, k, f.d.idx, f.d.cl, f.d.Wx, f.d.Wl, f.d.Wr,
                                                                       f.d.Wv, f.rho0, w.status, w.rho_idx, w.iters,
                                                                       w.nsw, f.d.client_of, f.d.Xc);
        RQ_SCUDA(s, cudaGetLastError());
        ++h->launches;
        Maps maps, warm;
        maps.add(n, w.F32, w.ldx, 1.f, nullptr, f.d.Qc, w.ldn);
        maps.add(m, w.E32, w.ldx, -1.f, w.l0, f.d.Lc, w.ldm, 0, 0, w.u0, f.d.Uc);
        for (int r = 0; r < h->nr; ++r)
            maps.add(R, w.G[r], w.ldx, 1.f, nullptr, f.d.Bc + (size_t)r * w.cap * w.ldR, w.ldR, n, w.nP - n);
        RQ_TRY(maps.run(h, k, nx, f.d.x0c, w.ldx));
        warm.add(m, h->A32, (int)round_up(n, 4), 1.f, nullptr, f.d.AYc, w.ldm);
        RQ_TRY(warm.run(h, k, n, f.d.Xc, w.ldn));
        serve_scatter_kernel<<<ceil_div(k * 32, 256), 256, 0, f.stream>>>(p, k, f.d.idx, f.d.Qc, f.d.Lc, f.d.Uc,
                                                                         f.d.Bc, f.d.AYc, w.Q, w.L, w.U, w.BIAS,
                                                                         w.QN);
        RQ_SCUDA(s, cudaGetLastError());
        ++h->launches;
    }
    if (f.active == 0) return RELU_QP_OK;
    // ---- one chunk ----
    const int ci = h->opts.check_interval;
    size_t prof_used = 0;
    h->prof_span_launches.clear();    // the server does not read the layer events
    RQ_TRY(zero_chunk_sync(h));
    RQ_TRY(assign_slots(h, w.cap, false));
    RQ_TRY(fill_slots(h, p, true));
    RQ_TRY(run_layers(h, p, ci, true, f.active, 0, prof_used));
    RQ_TRY(run_check(h, p, f.active, 0));
    RQ_SCUDA(s, cudaMemsetAsync(f.d.cnt, 0, sizeof(int), f.stream));
    DecideArgs dd{w.cap, 0, 0, h->opts.adaptive_rho, s->eps_abs, s->eps_rel, w.XO, w.ZO, w.LO,
                  w.status, w.iters, w.rho_idx, w.nsw, w.rp, w.rd, ci, s->max_iter, f.d.done, f.d.cnt};
    batch_decide_kernel<<<w.cap, kDecideThreads, 0, f.stream>>>(p, dd, 0);
    RQ_SCUDA(s, cudaGetLastError());
    serve_gather_kernel<<<ceil_div(w.cap * 32, 256), 256, 0, f.stream>>>(
        p, f.d.done, f.d.cnt, f.d.client_of, w.status, w.iters, w.rho_idx, w.nsw, w.rp, w.rd, w.XO, h->sc_x, f.d.Wx,
        f.d.Wl, f.d.Wr, f.d.Wv, f.d.out, f.ldo);
    RQ_SCUDA(s, cudaGetLastError());
    h->launches += 2;
    RQ_SCUDA(s, cudaMemcpyAsync(f.h_cnt, f.d.cnt, sizeof(int), cudaMemcpyDeviceToHost, f.stream));
    RQ_SCUDA(s, cudaMemcpyAsync(f.h_cnt + 1, w.counters, sizeof(int) * CNT_WORDS, cudaMemcpyDeviceToHost, f.stream));
    RQ_SCUDA(s, cudaMemcpyAsync(f.h_out, f.d.out, sizeof(float) * (size_t)w.cap * f.ldo, cudaMemcpyDeviceToHost,
                                f.stream));
    RQ_SCUDA(s, cudaEventRecord(f.ev, f.stream));
    f.launched = true;
    return RELU_QP_OK;
}

int family_collect(relu_qp_server_t s, ServeFamily& f, int fi) {
    if (!f.launched) return RELU_QP_OK;
    f.launched = false;
    RQ_SCUDA(s, cudaEventSynchronize(f.ev));   // complete already when called from server_step
    const double t = s->now();
    if (f.h_cnt[1 + CNT_ERR]) return sfail(s, RELU_QP_ERR_TIMEOUT, "a tensor-core kernel wait passed its deadline");
    const int cnt = f.h_cnt[0];
    const int n = f.h->n;
    for (int j = 0; j < cnt; ++j) {
        const float* o = f.h_out + (size_t)j * f.ldo;
        ServeResult res;
        const int qp = __float_as_int_host(o[n + 0]);
        res.r.tag = f.tag_of[qp];
        res.r.family = fi;
        res.r.client = f.client_of[qp];
        res.r.status = __float_as_int_host(o[n + 1]);
        res.r.iters = __float_as_int_host(o[n + 2]);
        res.r.rho_index = __float_as_int_host(o[n + 3]);
        res.r.rho_switches = __float_as_int_host(o[n + 4]);
        res.r.r_prim = o[n + 5];
        res.r.r_dual = o[n + 6];
        res.r.t_submit = f.t_submit_of[qp];
        res.r.t_done = t;
        res.x.assign(o, o + n);
        s->results.push_back(std::move(res));
        f.free_idx.push_back(qp);
        --f.active;
        s->in_use -= std::min(s->in_use, f.slot_bytes);
    }
    return RELU_QP_OK;
}

}  // namespace

int server_create(relu_qp_server_t* out, relu_qp_t const* families, int nf, const int* clients, double eps_abs,
                  double eps_rel, int max_iter) {
    relu_qp_server_t s = new (std::nothrow) relu_qp_server_s;
    if (!s) return RELU_QP_ERR_OOM;
    *out = s;
    s->eps_abs = eps_abs;
    s->eps_rel = eps_rel;
    s->max_iter = max_iter;
    s->t0 = std::chrono::steady_clock::now();
    s->fam.resize(nf);
    for (int fi = 0; fi < nf; ++fi) {
        ServeFamily& f = s->fam[fi];
        relu_qp_t h = families[fi];
        BatchWork& w = h->bw;
        f.h = h;
        f.cap = w.cap;
        f.clients = clients ? clients[fi] : 0;
        f.ldo = h->n + 8;
        f.rho0 = nearest_rho(h, h->opts.rho0);
        f.tag_of.assign(f.cap, 0);
        f.t_submit_of.assign(f.cap, 0.0);
        f.client_of.assign(f.cap, -1);
        for (int q = f.cap - 1; q >= 0; --q) f.free_idx.push_back(q);
        // smaller problems get higher stream priorities, so that their short chunks
        // do not queue behind the grids of a family of large problems
        int rank = 0;
        for (int g = 0; g < nf; ++g)
            if (families[g]->R < h->R || (families[g]->R == h->R && g < fi)) ++rank;
        int prio_lo = 0, prio_hi = 0;
        RQ_SCUDA(s, cudaDeviceGetStreamPriorityRange(&prio_lo, &prio_hi));
        // (numerically lower = higher priority: the smallest family gets prio_hi)
        const int prio = std::min(prio_lo, prio_hi + rank);
        RQ_SCUDA(s, cudaStreamCreateWithPriority(&f.stream, cudaStreamNonBlocking, prio));
        RQ_SCUDA(s, cudaEventCreateWithFlags(&f.ev, cudaEventDisableTiming));
        f.saved_stream = h->stream;
        h->stream = f.stream;
        // families share the GPU: no persistent (one-wave, co-resident) chunk kernels
        if (h->bw.tc) tc_disable_chunk(h);
        // The launches take the configuration tuned for the tiles that the family's slots fill.  (Any
        // number of tiles runs under any configuration.  One tile per bank entry more, the bound on
        // them, is mostly three times the truth; the number at hand would let a request's rounding
        // depend on what shares the batch.)
        h->bw.tiles_hint = ceil_div(f.cap, kSlotTile);
        const size_t cap = f.cap, cl = f.clients > 0 ? f.clients : 1;
        RQ_TRY(sdev(s, f, &f.d.idx, cap));
        RQ_TRY(sdev(s, f, &f.d.cl, cap));
        RQ_TRY(sdev(s, f, &f.d.client_of, cap));
        RQ_TRY(sdev(s, f, &f.d.done, cap));
        RQ_TRY(sdev(s, f, &f.d.cnt, 4));
        RQ_TRY(sdev(s, f, &f.d.x0c, cap * w.ldx));
        RQ_TRY(sdev(s, f, &f.d.Qc, cap * w.ldn));
        RQ_TRY(sdev(s, f, &f.d.Xc, cap * w.ldn));
        RQ_TRY(sdev(s, f, &f.d.Lc, cap * w.ldm));
        RQ_TRY(sdev(s, f, &f.d.Uc, cap * w.ldm));
        RQ_TRY(sdev(s, f, &f.d.AYc, cap * w.ldm));
        RQ_TRY(sdev(s, f, &f.d.Bc, (size_t)h->nr * cap * w.ldR));
        RQ_TRY(sdev(s, f, &f.d.out, cap * f.ldo));
        RQ_TRY(sdev(s, f, &f.d.Wx, cl * w.ldn));
        RQ_TRY(sdev(s, f, &f.d.Wl, cl * w.ldm));
        RQ_TRY(sdev(s, f, &f.d.Wr, cl));
        RQ_TRY(sdev(s, f, &f.d.Wv, cl));
        RQ_TRY(shost(s, f, &f.h_x0c, cap * w.ldx));
        RQ_TRY(shost(s, f, &f.h_idx, cap));
        RQ_TRY(shost(s, f, &f.h_cl, cap));
        RQ_TRY(shost(s, f, &f.h_cnt, 8));
        RQ_TRY(shost(s, f, &f.h_out, cap * f.ldo));
        // every QP index starts free
        batch_init_kernel<<<w.cap, kInitThreads, 0, f.stream>>>(base_params(h), 0, 0, 0, nullptr, f.rho0,
                                                                           w.status, w.rho_idx, w.iters, w.nsw);
        RQ_SCUDA(s, cudaGetLastError());
        RQ_SCUDA(s, cudaMemsetAsync(w.counters, 0, sizeof(int) * CNT_WORDS, f.stream));
        RQ_SCUDA(s, cudaStreamSynchronize(f.stream));
        // memory accounting: a request occupies one QP slot of the handle plus its rows of the
        // server's compact buffers (x0, q, x, l, u, A x, b of every bank entry, the result row)
        const size_t fl = sizeof(float);
        const size_t serve_slot = (w.ldx + 2 * w.ldn + 3 * w.ldm + (size_t)h->nr * w.ldR + f.ldo) * fl +
                                  4 * sizeof(int);
        f.slot_bytes = batch_slot_bytes(h) + serve_slot;
        const size_t fam_fixed = h->dev_bytes + f.dev_bytes;
        const size_t fam_slots = (size_t)f.cap * f.slot_bytes;
        s->fixed += fam_fixed > fam_slots ? fam_fixed - fam_slots : 0;
    }
    return RELU_QP_OK;
}

int server_set_budget(relu_qp_server_t s, long long bytes) {
    size_t one = 0;   // room for one request of every family, so that none waits forever
    for (const auto& f : s->fam) one = std::max(one, f.slot_bytes);
    if (bytes > 0 && (size_t)bytes < s->fixed + one)
        return sfail(s, RELU_QP_ERR_OOM, "server budget of " + std::to_string(bytes) + " bytes is below the " +
                                             std::to_string(s->fixed) + " bytes of the families' banks and buffers "
                                             "plus one request of the largest family (" + std::to_string(one) + ")");
    s->budget = bytes;
    return RELU_QP_OK;
}

int server_family_bytes(relu_qp_server_t s, int family, long long* fixed_bytes, long long* slot_bytes) {
    const ServeFamily& f = s->fam[family];
    const size_t all = f.h->dev_bytes + f.dev_bytes, slots = (size_t)f.cap * f.slot_bytes;
    if (fixed_bytes) *fixed_bytes = (long long)(all > slots ? all - slots : 0);
    if (slot_bytes) *slot_bytes = (long long)f.slot_bytes;
    return RELU_QP_OK;
}

long long server_bytes_in_use(relu_qp_server_t s) { return (long long)s->in_use; }

int server_submit(relu_qp_server_t s, int family, int client, const float* x0, long long tag) {
    ServeFamily& f = s->fam[family];
    ServeRequest r;
    r.client = client;
    r.tag = tag;
    r.t_submit = s->now();
    r.x0.assign(x0, x0 + f.h->bw.nx);
    f.queue.push_back(std::move(r));
    return RELU_QP_OK;
}

// Families advance independently: a family with no chunk in flight admits and
// launches; one whose chunk has finished (its event has completed) retires,
// admits and launches again at once.  The call returns once some family has
// finished a chunk (or when no chunk is in flight), so a family of small
// problems is never held back by the chunk of a family of large ones.
int server_step(relu_qp_server_t s, int* active, int* waiting) {
    const size_t nf = s->fam.size();
    for (auto& f : s->fam)
        if (!f.launched) RQ_TRY(family_launch(s, f));
    bool any_in_flight = false;
    for (auto& f : s->fam) any_in_flight = any_in_flight || f.launched;
    bool progressed = !any_in_flight;
    while (!progressed) {
        for (size_t fi = 0; fi < nf; ++fi) {
            ServeFamily& f = s->fam[fi];
            if (!f.launched) continue;
            const cudaError_t q = cudaEventQuery(f.ev);
            if (q == cudaErrorNotReady) continue;
            if (q != cudaSuccess) {
                cudaGetLastError();
                return sfail(s, RELU_QP_ERR_CUDA, std::string("server chunk: ") + cudaGetErrorString(q));
            }
            RQ_TRY(family_collect(s, f, (int)fi));
            RQ_TRY(family_launch(s, f));
            progressed = true;
        }
        if (!progressed) std::this_thread::yield();
    }
    int a = 0, q = 0;
    for (auto& f : s->fam) {
        a += f.active;
        q += (int)f.queue.size();
    }
    if (active) *active = a;
    if (waiting) *waiting = q;
    return RELU_QP_OK;
}

int server_poll(relu_qp_server_t s, int max_results, relu_qp_result* results, float* x_out, int x_stride) {
    int k = 0;
    while (k < max_results && !s->results.empty()) {
        ServeResult& r = s->results.front();
        if (results) results[k] = r.r;
        if (x_out) std::memcpy(x_out + (size_t)k * x_stride, r.x.data(), sizeof(float) * r.x.size());
        s->results.pop_front();
        ++k;
    }
    return k;
}

void server_destroy(relu_qp_server_t s) {
    for (auto& f : s->fam) {
        if (f.stream) cudaStreamSynchronize(f.stream);
        if (f.h) {
            f.h->stream = f.saved_stream;
            f.h->bw.tiles_hint = 0;
        }
        for (void* p : f.dev_allocs) cudaFree(p);
        for (void* p : f.host_allocs) cudaFreeHost(p);
        if (f.ev) cudaEventDestroy(f.ev);
        if (f.stream) cudaStreamDestroy(f.stream);
    }
    delete s;
}

const char* server_error(relu_qp_server_t s) { return s->err.c_str(); }
int server_families(relu_qp_server_t s) { return (int)s->fam.size(); }
int server_clients(relu_qp_server_t s, int family) { return s->fam[family].clients; }
int server_nx(relu_qp_server_t s, int family) { return s->fam[family].h->bw.nx; }
double server_clock(relu_qp_server_t s) { return s->now(); }

}  // namespace rq
