// Single-QP online stage of Algorithm 1 (Sec. III-B) in one cooperative
// kernel: the layer of Eq. gpu_update every iteration, the residuals of Eqs.
// primal and dual every check_interval layers, the penalty rule of Eq.
// rho_update with the nearest bank entry (Sec. III-C), and the stop test.
//
// Layer in factored form (the algebra is in setup_fp64.cu): with
//   s = [x; 2 rho z - lam'],   t = Wt s + b,
//   r = (Ax) - z + lam'/rho          (carried Ax from the previous layer)
//   x+ = t_x,  (Ax)+ = t_Ax,  z+ = clamp(t_Ax + r, l, u),  lam'+ = rho r,
// which equals v+ = clamp(W v + b) with v = [x; z; lam'].
//
// Work split: each CTA owns a slice of the rows of x and a slice of the rows of
// A x, keeps as many of their rows of Wt as fit in shared memory (the rest
// stream from L2) and their state for the whole solve; a warp computes up to
// 4 consecutive rows at once (coalesced 128-bit loads, one shuffle reduction
// per row).  The check of a row of x and the dual residual of that row stay in
// the same CTA, so a check exchanges only lam_std and the residual maxima.
//
// Exchange.  What bounds a layer is not the product (a few hundred clocks) but
// handing every CTA the new operand, so the operand's entries carry their own
// arrival and no barrier stands between layers.  Three forms, chosen by timing
// at setup; a row's arithmetic, and so every bit of the result, is the same:
//  - one CTA: shared memory and a CTA barrier;
//  - one cluster: st.async writes each entry into every CTA's copy and counts
//    its bytes on that CTA's mbarrier (one trip; a store, a release and an
//    arrival one after the other before);
//  - a cooperative grid: every entry is one 64-bit word in global memory, value
//    and exchange number together, and the readers poll the words themselves;
//    or, where that many words would crowd the L2, plain entries and a count of
//    the CTAs that have stored theirs, polled before the entries are read.
// Two operand buffers suffice: a CTA publishes exchange e + 1 (over e - 1) only
// after it has all of e, and a row's part of e is sent only once its warp has
// read all of e - 1 that it needs.
// A row's remaining state (z, lam', r) is updated after its entry has left, and stays in
// registers while every warp has one group of rows; a check's FP64 decision is one warp's.
//
// Measured, us per layer at n = m = 20 / 160 / 320 / 640 / 800 / 1600 (200 fixed layers,
// best shape): 0.55 / 0.90 / 1.22 / 2.04 / 2.47 / 4.34; with a barrier between layers and
// the operand loaded after it 1.61 / 1.98 / 2.23 / 2.72 / 2.92 / 4.75.  They are bound by the
// exchange: 0.25 (one CTA), 0.6 (cluster), 1.2 (words), 2.2 (count); the last by that and by
// reading the rows, about half each (a CTA's 22 rows, 16 from shared memory and 6 from L2).
//
// Every wait has a deadline after which the kernel records RELU_QP_ERR_TIMEOUT
// in the error word; the other waits see it and leave too.
#include "common.h"
#include "grid_sync.h"
#include "shape_search.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <mutex>

namespace rq {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;

enum { RED_RP = 0, RED_RD, RED_AX, RED_Z, RED_PX, RED_ATL, RED_WORDS = 8 };
enum { DEC_STOP = 6, DEC_RHO = 7 };   // of the decision's words: 1 + the status to stop with, or 0; bank entry
enum { OUT_STATUS = 0, OUT_ITERS, OUT_RHO, OUT_SWITCHES, OUT_LAST, OUT_GAVE_UP, OUT_WORDS = 8 };
// FORM_GRID and FORM_COUNT are cooperative grids: tagged words, or plain operand buffers and a
// count of the CTAs that have written theirs.
enum Form { FORM_GRID = 0, FORM_CLUSTER = 1, FORM_ONE = 2, FORM_COUNT = 3 };
constexpr int kState = 9;   // floats of state per row (see solve_body)

struct SP {
    int n, m, R, ldw, ldp, ldt, nr;
    const float* Wt[RQ_MAX_RHO];
    const float* bias[RQ_MAX_RHO];
    double rho[RQ_MAX_RHO];
    const float *P, *A, *At, *q, *l, *u, *rs;
    const float *rsx, *rsz;   // scaled problems: residual factors 1/(c D), 1/E (else nullptr)
    const float *xin, *lin;   // warm start (or nullptr)
    float *xo, *zo, *lo;      // results (zo, lo may be nullptr)
    // grid form: tagged words of the operand [2][R], of lam_std [m] and of the maxima [ctas][8]
    unsigned long long *wop, *wls, *wred;
    unsigned tag0;            // exchange e is tagged tag0 + 1 + e
    // count form: the operand buffers [2][ldw] and the arrivals so far, from count0 on
    float* sop;
    unsigned *count, count0;
    int *err, *out_i;
    float* out_f;
    int rho_index0, check_interval, adaptive, max_iter;
    double eps_abs, eps_rel, qnorm;
    int xr, ar, ctas;         // rows of x and of A x per CTA, CTAs with rows
    int gs, gu, cached_rows;  // rows of a warp's group, of a group outside shared memory
    int share;                // count form, where both do not fit: lam_std staged over the operand
    long long timeout_ns;
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

constexpr int kRows = 4;   // rows of a warp whose dot products run together (a group)

// Dot products of NR (1, 2 or 4) padded rows (w[j], in shared or global memory) with one
// padded vector in shared memory, in one pass over k, so that the rows' loads overlap.  Rows and
// vector are 16-byte aligned and zero padded to a multiple of 4 floats.  Every row keeps four
// accumulators and one summation tree of its own, whatever NR is, so that a row's bits do not
// depend on its group.  The sums are scattered as they are formed (a lane keeps half of its rows at each
// of the first steps: 6 shuffles for 4 rows where one reduction per row takes 20, and a
// CTA's shuffles go one warp a clock): lane l returns row l / (32 / NR).
template <int NR, bool LDG>
__device__ __forceinline__ float rows_dot(const float* const (&w)[kRows], const float* __restrict__ s, int ld, int lane) {
    const float4* s4 = reinterpret_cast<const float4*>(s);
    const int n4 = ld >> 2;
    float a[NR][4];
#pragma unroll
    for (int j = 0; j < NR; ++j) a[j][0] = a[j][1] = a[j][2] = a[j][3] = 0.f;
    int k = lane;
    if (LDG) {
        // rows in global memory: U steps' loads before the first product (an L2 trip is some
        // 700 clocks, the step's products a few)
        constexpr int U = NR == 1 ? 8 : NR == 2 ? 4 : 2;
        for (; k + 32 * (U - 1) < n4; k += 32 * U) {
            float4 x[U][NR];
#pragma unroll
            for (int t = 0; t < U; ++t)
#pragma unroll
                for (int j = 0; j < NR; ++j) x[t][j] = __ldg(reinterpret_cast<const float4*>(w[j]) + k + 32 * t);
#pragma unroll
            for (int t = 0; t < U; ++t) {
                const float4 b = s4[k + 32 * t];
#pragma unroll
                for (int j = 0; j < NR; ++j) {
                    a[j][0] = fmaf(x[t][j].x, b.x, a[j][0]);
                    a[j][1] = fmaf(x[t][j].y, b.y, a[j][1]);
                    a[j][2] = fmaf(x[t][j].z, b.z, a[j][2]);
                    a[j][3] = fmaf(x[t][j].w, b.w, a[j][3]);
                }
            }
        }
    }
    for (; k < n4; k += 32) {
        const float4 b = s4[k];
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            const float4* wj = reinterpret_cast<const float4*>(w[j]) + k;
            const float4 x = LDG ? __ldg(wj) : *wj;
            a[j][0] = fmaf(x.x, b.x, a[j][0]);
            a[j][1] = fmaf(x.y, b.y, a[j][1]);
            a[j][2] = fmaf(x.z, b.z, a[j][2]);
            a[j][3] = fmaf(x.w, b.w, a[j][3]);
        }
    }
    float v[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) v[j] = (a[j][0] + a[j][1]) + (a[j][2] + a[j][3]);
    int o = 16;
#pragma unroll
    for (int h = NR / 2; h >= 1; h /= 2, o /= 2) {
        const bool up = (lane & o) != 0;   // keeps the upper half of its rows
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const float give = up ? v[j] : v[j + h], keep = up ? v[j + h] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    for (; o > 0; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// LDG: every row is in global memory (read-only loads); else in shared memory or mixed.
template <bool LDG>
__device__ __forceinline__ float group_dot(int gs, const float* const (&w)[kRows], const float* s, int ld, int lane) {
    if (gs == 4) return rows_dot<4, LDG>(w, s, ld, lane);
    if (gs == 2) return rows_dot<2, LDG>(w, s, ld, lane);
    return rows_dot<1, LDG>(w, s, ld, lane);
}

constexpr bool is_grid(int form) { return form == FORM_GRID || form == FORM_COUNT; }

// ---- exchanges -------------------------------------------------------------
// The `count` values of the tagged words w into dst, by the whole CTA.
__device__ __forceinline__ bool gather(const SP& p, const unsigned long long* w, float* dst, int count, unsigned tag) {
    return gather_words<kThreads>(w, count, tag, p.err, p.timeout_ns, [&](int k, unsigned a, unsigned b, bool two) {
        dst[k] = __uint_as_float(a);
        if (two) dst[k + 1] = __uint_as_float(b);
    });
}

// The first ncache rows of the CTA (x rows x0 .., then A x rows a0 ..) of bank entry ri.
__device__ void load_w_cache(const SP& p, float* wcache, int ri, int x0, int nx, int a0, int ncache) {
    const int c4 = p.ldw >> 2;
    for (int e = threadIdx.x; e < ncache * c4; e += kThreads) {
        const int lr = e / c4, k = e - lr * c4, r = lr < nx ? x0 + lr : p.n + a0 + (lr - nx);
        reinterpret_cast<float4*>(wcache)[e] = __ldg(reinterpret_cast<const float4*>(p.Wt[ri] + (size_t)r * p.ldw) + k);
    }
}

__device__ __forceinline__ void red_max(unsigned* slot, int word, float v) {
    atomicMax(slot + word, __float_as_uint(fabsf(v)));
}

// The solve; false if a wait gave up.
template <int F>
__device__ __forceinline__ bool solve_body(const SP& p, float* smem, unsigned long long* mbar, unsigned* s_red,
                                           unsigned* s_dec) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int n = p.n, m = p.m, R = p.R, ldw = p.ldw, cta = blockIdx.x;
    // this CTA's rows: lr < nx are x0 + lr, the others A x rows a0 + lr - nx
    const int x0 = cta * p.xr, nx = max(0, min(p.xr, n - x0));
    const int a0 = cta * p.ar, na = max(0, min(p.ar, m - a0));
    const int rows = nx + na, gs = p.gs;
    const int ncache = min(p.cached_rows, rows);
    const int ngu = (rows - ncache + p.gu - 1) / p.gu, ng = ngu + (ncache + gs - 1) / gs;
    const int per = p.xr + p.ar;
    float* wcache = smem;
    float* sv = smem + (size_t)p.cached_rows * ldw;        // operand: two buffers (grids: one)
    float* svk = sv + (size_t)(is_grid(F) ? 1 : 2) * ldw;  // lam_std (ldt floats)
    float* reds = svk + (p.share ? 0 : p.ldt);             // every CTA's maxima [ctas][8]
    if (F == FORM_COUNT && p.share) svk = sv;              // (read again after the check)
    float* st_bias = reds + RED_WORDS * p.ctas;
    // per row: bias, r = (Ax) - z + lam'/rho of the next layer, z (x of a row of x), lam', rho, l, u,
    // the check's product, lam_std
    float *st_rr = st_bias + per, *st_z = st_rr + per, *st_lam = st_z + per, *st_rho = st_lam + per,
          *st_l = st_rho + per, *st_u = st_l + per, *st_chk = st_u + per, *st_ls = st_chk + per;
    // (from the rounded lam' in every layer, as the batched FP32 path forms it: with t - z + r instead
    // a multiplier that is zero keeps other rounding noise)
    auto carry = [&](float ax, float z, float lam, float rho_i) { return ax - z + lam / rho_i; };
    // barriers (cluster form): operand buffers 0 and 1, lam_std, maxima
    const uint32_t bar0 = cl_smem(mbar);
    const uint32_t sv_a = cl_smem(sv), svk_a = cl_smem(svk), reds_a = cl_smem(reds);
    auto row_of = [&](int lr) { return lr < nx ? x0 + lr : n + a0 + (lr - nx); };
    bool failed = false;
    unsigned e = 0;      // exchange whose operand is current
    auto cur = [&]() { return sv + (is_grid(F) ? 0 : (size_t)(e & 1) * ldw); };
    // one entry of exchange x
    auto publish = [&](unsigned x, int r, float v) {
        if (F == FORM_GRID) {
            put_word(p.wop + (size_t)(x & 1) * ((R + 1) & ~1) + r, __float_as_uint(v), p.tag0 + 1 + x);
        } else if (F == FORM_COUNT) {
            p.sop[(size_t)(x & 1) * ldw + r] = v;
        } else if (F == FORM_ONE) {
            sv[(size_t)(x & 1) * ldw + r] = v;
        } else {
            for (int q = 0; q < p.ctas; ++q) cl_send1(sv_a + 4u * ((x & 1) * ldw + r), bar0 + 8 * (x & 1), q, v);
        }
    };
    // all of exchange x (cluster form: a warp's own wait, by the warps that compute rows; whole
    // warps call it, and `failed` is the same in every lane)
    auto wait_bar = [&](uint32_t bar, uint32_t parity) {
        if (!failed && !cl_wait_warp(bar, parity, p.err, p.timeout_ns)) failed = true;
    };
    // (count form) exchange x, all of it stored, into shared memory
    auto load_operand = [&](unsigned x) {
        const float4* src = reinterpret_cast<const float4*>(p.sop + (size_t)(x & 1) * ldw);
        for (int k = tid; k < (ldw >> 2); k += kThreads) reinterpret_cast<float4*>(sv)[k] = __ldcg(src + k);
        __syncthreads();
    };
    auto receive = [&](unsigned x) -> bool {
        if (F == FORM_GRID) {
            __syncthreads();   // the buffer's readers are done
            return gather(p, p.wop + (size_t)(x & 1) * ((R + 1) & ~1), sv, R, p.tag0 + 1 + x);
        }
        if (F == FORM_COUNT) {
            // every CTA has stored its entries and read the last operand
            if (!count_wait(p.count, p.count0 + (x + 1) * (unsigned)p.ctas, p.err, p.timeout_ns)) return false;
            load_operand(x);
            return true;
        }
        if (F == FORM_ONE) {
            __syncthreads();
            return true;
        }
        if (warp < ng) wait_bar(bar0 + 8 * (x & 1), (x >> 1) & 1);
        if (tid == 0 && !failed) cl_expect(bar0 + 8 * (x & 1), 4u * R);   // the buffer's next use
        return true;
    };

    int ri = p.rho_index0, switches = 0;
    unsigned checks = 0;
    // ---------------- start state ----------------
    for (int k = tid; k < ldw; k += kThreads) {   // the padding's zeros, and x for z = A x
        const float v = k < n && p.xin ? p.xin[k] : 0.f;
        // (cluster form: exchange 0 may already be arriving in the first buffer)
        if (F != FORM_CLUSTER || k >= R) sv[k] = v;
        if (!is_grid(F)) sv[ldw + k] = v;
    }
    if (!p.share)
        for (int k = tid; k < p.ldt; k += kThreads) svk[k] = 0.f;
    if (tid < RED_WORDS) s_red[tid] = 0u;
    for (int lr = tid; lr < rows; lr += kThreads) {
        st_bias[lr] = __ldg(p.bias[ri] + row_of(lr));
        if (lr >= nx) {
            const int i = a0 + lr - nx;
            st_rho[lr] = (float)(p.rho[ri] * (double)__ldg(p.rs + i));
            st_l[lr] = __ldg(p.l + i);
            st_u[lr] = __ldg(p.u + i);
            st_lam[lr] = p.lin ? p.lin[i] : 0.f;
            st_z[lr] = 0.f;
        }
    }
    __syncthreads();
    if (p.xin) {
        // z = A x
        const float* x = is_grid(F) ? sv : sv + ldw;
        for (int lr = nx + warp; lr < rows; lr += kWarps) {
            const float* a = p.A + (size_t)(a0 + lr - nx) * p.ldp;
            float v = 0.f;
#pragma unroll 4
            for (int k = lane; k < n; k += 32) v = fmaf(__ldg(a + k), x[k], v);
            v = warp_sum(v);
            if (lane == 0) st_z[lr] = v;
        }
        __syncthreads();
    }
    for (int lr = tid; lr < rows; lr += kThreads) {
        const int r = row_of(lr);
        if (lr >= nx) st_rr[lr] = carry(st_z[lr], st_z[lr], st_lam[lr], st_rho[lr]);
        publish(0, r, lr < nx ? (p.xin ? p.xin[r] : 0.f) : fmaf(2.0f * st_rho[lr], st_z[lr], -st_lam[lr]));
    }
    load_w_cache(p, wcache, ri, x0, nx, a0, ncache);
    if (F == FORM_CLUSTER) {
        __syncthreads();
        if (tid < 32) wait_bar(bar0, 0);
        failed = __syncthreads_or(failed ? 1 : 0) != 0;
        if (tid == 0 && !failed) cl_expect(bar0, 4u * R);
    } else if (!receive(0)) {
        return false;
    }

    // Groups: the rows that are not in shared memory first (their loads take longest), one to
    // gu of them to a warp, then gs of the cached ones; group g is warp g % kWarps's.  A
    // group's lanes split by row: lane l updates row l / (32 / its rows), one lane per row
    // publishes and stores.
    struct Group {
        int lr0, cnt, gr;      // first row, rows, lanes' rows (gs or gu)
        bool global;
        const float* w[kRows];
    };
    auto group = [&](int g) {
        Group G;
        G.global = g < ngu;
        G.gr = G.global ? p.gu : gs;
        G.lr0 = G.global ? ncache + g * p.gu : (g - ngu) * gs;
        G.cnt = min(G.gr, (G.global ? rows : ncache) - G.lr0);
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
            const int lr = G.lr0 + (j < G.cnt ? j : 0);
            G.w[j] = G.global ? p.Wt[ri] + (size_t)row_of(lr) * ldw : wcache + (size_t)lr * ldw;
        }
        return G;
    };
    auto product = [&](const Group& G, const float* s) {
        return G.global ? group_dot<true>(G.gr, G.w, s, ldw, lane) : group_dot<false>(G.gr, G.w, s, ldw, lane);
    };
    // a group's new operand entries: row lr's in its lanes, `one` set in one of them
    auto hand_on = [&](const Group& G, int lr, bool valid, bool one, float snew) {
        if (F != FORM_CLUSTER) {
            if (one) publish(e + 1, row_of(lr), snew);
            return;
        }
        const int r = row_of(G.lr0), b = (int)((e + 1) & 1);
        const uint32_t bar = bar0 + 8 * b, base = sv_a + 4u * (uint32_t)(b * ldw);
        if (G.cnt == 4 && (r & 3) == 0 && (G.lr0 + 3 < nx || G.lr0 >= nx)) {
            const float v0 = __shfl_sync(0xffffffffu, snew, 0), v1 = __shfl_sync(0xffffffffu, snew, 8),
                        v2 = __shfl_sync(0xffffffffu, snew, 16), v3 = __shfl_sync(0xffffffffu, snew, 24);
            if (lane < p.ctas) cl_send4(base + 4u * (uint32_t)r, bar, lane, v0, v1, v2, v3);
        } else if (valid) {
            const int per_row = 32 / G.gr;
            for (int q = lane % per_row; q < p.ctas; q += per_row) cl_send1(base + 4u * (uint32_t)row_of(lr), bar, q, snew);
        }
    };

    int it = 0;
    while (true) {
        // ---------------- the layers up to the next check, or the last one ----------------
        const int len = p.check_interval > 0 ? min(p.check_interval, p.max_iter - it) : p.max_iter - it;
        if (ng <= kWarps) {
            // one group a warp: its rows' state stays in registers
            const bool work = warp < ng;
            const Group G = group(work ? warp : 0);
            const int per_row = 32 / G.gr, jl = lane / per_row;
            const bool valid = work && jl < G.cnt, one = valid && lane % per_row == 0;
            const int lr = G.lr0 + (jl < G.cnt ? jl : 0);
            const bool ax = work && lr >= nx;
            const float bias = work ? st_bias[lr] : 0.f, rho_i = ax ? st_rho[lr] : 0.f, lo = ax ? st_l[lr] : 0.f,
                        up = ax ? st_u[lr] : 0.f, rho2 = 2.0f * rho_i;
            float rr = ax ? st_rr[lr] : 0.f, t = 0.f, z = 0.f, lam = 0.f;
            for (int k = 0; k < len; ++k) {
                if (work && !failed) {
                    if (ax && k > 0) rr = carry(t, z, lam, rho_i);   // (beside the product, not after it)
                    t = product(G, cur()) + bias;
                    z = t;
                    float snew = z;
                    if (ax) {
                        z = fminf(fmaxf(t + rr, lo), up);
                        lam = __fmul_rn(rho_i, rr);
                        snew = fmaf(rho2, z, -lam);
                    }
                    hand_on(G, lr, valid, one, snew);
                }
                ++e;
                if (!receive(e)) return false;
            }
            if (one) {
                st_z[lr] = z;
                if (ax) st_lam[lr] = lam;
            }
        } else {
            for (int k = 0; k < len; ++k) {
                const float* svc = cur();
                for (int g = warp; g < ng && !failed; g += kWarps) {
                    const Group G = group(g);
                    const int per_row = 32 / G.gr, jl = lane / per_row;
                    const bool valid = jl < G.cnt, one = valid && lane % per_row == 0;
                    const int lr = G.lr0 + (valid ? jl : 0);
                    const float t = product(G, svc) + st_bias[lr];
                    float z = t, lam = 0.f, snew = t, rr = 0.f;
                    const bool ax = lr >= nx;
                    if (ax) {
                        rr = st_rr[lr];
                        z = fminf(fmaxf(t + rr, st_l[lr]), st_u[lr]);
                        lam = __fmul_rn(st_rho[lr], rr);
                        snew = fmaf(2.0f * st_rho[lr], z, -lam);
                    }
                    hand_on(G, lr, valid, one, snew);
                    if (one) {
                        st_z[lr] = z;
                        if (ax) {
                            st_lam[lr] = lam;
                            st_rr[lr] = carry(t, z, lam, st_rho[lr]);
                        }
                    }
                    __syncwarp();
                }
                ++e;
                if (!receive(e)) return false;
            }
        }
        it += len;
        const bool is_check = p.check_interval > 0 && it % p.check_interval == 0;
        const bool last = (it == p.max_iter);

        // ---------------- residuals (Eqs. primal, dual) ----------------
        // (a warp of the cluster form that gave up leaves here, with its CTA)
        if (__syncthreads_or(failed ? 1 : 0)) return false;
        const float* svc = cur();
        const unsigned tag = p.tag0 + 1 + e;
        constexpr int kC = 2, kPer = 32 / kC;   // rows of a warp (in global memory: P, A, A^T)
        const int jc = lane / kPer;
        const bool lead = lane % kPer == 0;
        for (int lr0 = warp * kC; lr0 < rows; lr0 += kWarps * kC) {
            const int lr = lr0 + jc;
            const float* c[kRows];
#pragma unroll
            for (int j = 0; j < kRows; ++j) {
                const int k = min(lr0 + (j < kC ? j : 0), rows - 1);
                c[j] = k < nx ? p.P + (size_t)(x0 + k) * p.ldp : p.A + (size_t)(a0 + k - nx) * p.ldp;
            }
            const float v = rows_dot<kC, true>(c, svc, p.ldp, lane);
            if (lr < nx) {
                if (lead) {
                    st_chk[lr] = v;
                    red_max(s_red, RED_PX, p.rsx ? v * p.rsx[x0 + lr] : v);
                }
            } else if (lr < rows) {
                const int i = a0 + lr - nx;
                const float zi = st_z[lr], f = p.rsz ? p.rsz[i] : 1.f, ls = fmaf(st_rho[lr], v - zi, st_lam[lr]);
                if (lead) {
                    st_chk[lr] = v;
                    st_ls[lr] = ls;
                    red_max(s_red, RED_RP, (v - zi) * f);
                    red_max(s_red, RED_AX, v * f);
                    red_max(s_red, RED_Z, zi * f);
                    if (is_grid(F)) put_word(p.wls + i, __float_as_uint(ls), tag);
                    else if (F == FORM_ONE) svk[i] = ls;
                }
                if (F == FORM_CLUSTER)
                    for (int q = lane % kPer; q < p.ctas; q += kPer) cl_send1(svk_a + 4u * (uint32_t)i, bar0 + 16, q, ls);
            }
        }
        if (is_grid(F)) {
            if (F == FORM_COUNT && p.share) {
                __syncthreads();
                for (int k = m + tid; k < p.ldt; k += kThreads) svk[k] = 0.f;
            }
            if (m > 0 && !gather(p, p.wls, svk, m, tag)) return false;
        } else if (F == FORM_ONE) {
            __syncthreads();
        } else if (m > 0) {
            wait_bar(bar0 + 16, checks & 1);
            if (__syncthreads_or(failed ? 1 : 0)) return false;
            if (tid == 0) cl_expect(bar0 + 16, 4u * m);
        }
        for (int lr0 = warp * kC; lr0 < nx; lr0 += kWarps * kC) {
            const int lr = lr0 + jc;
            float v = 0.f;
            if (m > 0) {
                const float* c[kRows];
#pragma unroll
                for (int j = 0; j < kRows; ++j) c[j] = p.At + (size_t)(x0 + min(lr0 + (j < kC ? j : 0), nx - 1)) * p.ldt;
                v = rows_dot<kC, true>(c, svk, p.ldt, lane);
            }
            if (lr < nx && lead) {
                const float f = p.rsx ? p.rsx[x0 + lr] : 1.f;
                red_max(s_red, RED_RD, (st_chk[lr] + __ldg(p.q + x0 + lr) + v) * f);
                red_max(s_red, RED_ATL, v * f);
            }
        }
        __syncthreads();
        // every CTA's maxima
        if (is_grid(F)) {
            if (tid < RED_WORDS) put_word(p.wred + RED_WORDS * cta + tid, s_red[tid], tag);
            if (!gather(p, p.wred, reds, RED_WORDS * p.ctas, tag)) return false;
        } else if (F == FORM_CLUSTER) {
            for (int t = tid; t < 2 * p.ctas; t += kThreads) {
                const float* v = reinterpret_cast<const float*>(s_red) + 4 * (t & 1);
                cl_send4(reds_a + 4u * (uint32_t)(RED_WORDS * cta + 4 * (t & 1)), bar0 + 24, t >> 1, v[0], v[1], v[2], v[3]);
            }
            wait_bar(bar0 + 24, checks & 1);
            if (__syncthreads_or(failed ? 1 : 0)) return false;
            if (tid == 0) cl_expect(bar0 + 24, 4u * RED_WORDS * p.ctas);
        } else {
            if (tid < RED_WORDS) reinterpret_cast<unsigned*>(reds)[tid] = s_red[tid];
            __syncthreads();
        }
        ++checks;
        if (warp < 6) {
            unsigned v = 0;
            for (int q = lane; q < p.ctas; q += 32) v = max(v, reinterpret_cast<const unsigned*>(reds)[RED_WORDS * q + warp]);
            v = __reduce_max_sync(0xffffffffu, v);
            if (lane == 0) s_dec[warp] = v;
        }
        __syncthreads();
        if (tid < RED_WORDS) s_red[tid] = 0u;

        // ---------------- decision (identical in every CTA) ----------------
        // One warp takes it: an FP64 instruction holds an SM's FP64 pipe for 16 clocks a warp.
        if (warp == 0) {
            const double rp = __uint_as_float(s_dec[RED_RP]), rd = __uint_as_float(s_dec[RED_RD]);
            const double nAx = __uint_as_float(s_dec[RED_AX]), nz = __uint_as_float(s_dec[RED_Z]);
            const double nPx = __uint_as_float(s_dec[RED_PX]), nAtl = __uint_as_float(s_dec[RED_ATL]);
            const bool numerical = !(isfinite(rp) && isfinite(rd) && isfinite(nPx) && isfinite(nAtl));
            const double eps_p = p.eps_abs + p.eps_rel * fmax(nAx, nz);
            const double eps_d = p.eps_abs + p.eps_rel * fmax(fmax(nPx, nAtl), p.qnorm);
            const bool converged = is_check && !numerical && rp <= eps_p && rd <= eps_d;
            int nri = ri;
            if (p.adaptive && is_check && !converged && !numerical) {
                // Eq. rho_update (inf-norms, 1e-4 floors), nearest bank entry in log distance
                const double num = rp * fmax(fmax(nPx, nAtl), fmax(p.qnorm, 1e-4));
                const double den = rd * fmax(fmax(nAx, nz), 1e-4);
                if (num > 0.0 && den > 0.0) nri = nearest_entry(p.rho, p.nr, ri, p.rho[ri] * p.rho[ri] * (num / den));
            }
            if (lane == 0) {
                s_dec[DEC_STOP] = numerical ? 1 + RELU_QP_NUMERICAL : converged ? 1 + RELU_QP_SOLVED : last ? 1 + RELU_QP_MAX_ITER : 0;
                s_dec[DEC_RHO] = (unsigned)nri;
            }
        }
        __syncthreads();
        const int stop = (int)s_dec[DEC_STOP];
        if (stop) {
            for (int lr = tid; lr < rows; lr += kThreads) {
                if (lr < nx) {
                    p.xo[x0 + lr] = st_z[lr];
                } else {
                    const int i = a0 + lr - nx;
                    if (p.zo) p.zo[i] = st_z[lr];
                    if (p.lo) p.lo[i] = st_ls[lr];
                }
            }
            if (cta == 0 && tid == 0) {
                p.out_i[OUT_STATUS] = stop - 1;
                p.out_i[OUT_ITERS] = it;
                p.out_i[OUT_RHO] = ri;
                p.out_i[OUT_SWITCHES] = switches;
                p.out_i[OUT_LAST] = (int)e;
                p.out_f[0] = __uint_as_float(s_dec[RED_RP]);
                p.out_f[1] = __uint_as_float(s_dec[RED_RD]);
            }
            return true;
        }
        const int nri = (int)s_dec[DEC_RHO];
        if (nri == ri) {
            // the directly computed Ax replaces the carried one
            for (int lr = nx + tid; lr < rows; lr += kThreads) st_rr[lr] = carry(st_chk[lr], st_z[lr], st_lam[lr], st_rho[lr]);
            // lam_std was staged over the operand: read that again.  Without another arrival: the
            // exchange is complete, and its buffer is stored to again (e + 2) only after every CTA
            // has arrived at e + 1, which it does after this.
            if (F == FORM_COUNT && p.share) load_operand(e);
            else __syncthreads();   // the state above is read by the rows' warps
            continue;
        }
        // switch: rebase lam' so that the next layer is standard ADMM with the new rho, and
        // hand the operand on with the new penalties
        ri = nri;
        ++switches;
        for (int lr = tid; lr < rows; lr += kThreads) {
            const int r = row_of(lr);
            float v;
            if (lr < nx) {
                v = st_z[lr];
            } else {
                const float rho_i = (float)(p.rho[ri] * (double)__ldg(p.rs + (r - n)));
                const float lnew = fmaf(-rho_i, st_chk[lr] - st_z[lr], st_ls[lr]);
                st_lam[lr] = lnew;
                st_rho[lr] = rho_i;
                st_rr[lr] = carry(st_chk[lr], st_z[lr], lnew, rho_i);
                v = fmaf(2.0f * rho_i, st_z[lr], -lnew);
            }
            publish(e + 1, r, v);
            st_bias[lr] = __ldg(p.bias[ri] + r);
        }
        load_w_cache(p, wcache, ri, x0, nx, a0, ncache);
        __syncthreads();
        ++e;
        if (!receive(e)) return false;
    }
}

template <int F>
__global__ void __launch_bounds__(kThreads, 1) single_solve_kernel(const __grid_constant__ SP p) {
    extern __shared__ __align__(16) float smem[];
    __shared__ __align__(8) unsigned long long s_bar[4];
    __shared__ __align__(16) unsigned s_red[RED_WORDS];
    __shared__ unsigned s_dec[RED_WORDS];
    if (F == FORM_CLUSTER) {
        if (threadIdx.x == 0 && blockIdx.x < p.ctas) {
            const uint32_t b = cl_smem(s_bar);
            for (int k = 0; k < 4; ++k) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b + 8 * k) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            cl_expect(b, 4u * p.R);
            cl_expect(b + 8, 4u * p.R);
            if (p.m > 0) cl_expect(b + 16, 4u * p.m);
            cl_expect(b + 24, 4u * RED_WORDS * p.ctas);
        }
        cl_sync_hw();   // every CTA's barriers stand before anything is sent
    }
    const bool done = (int)blockIdx.x >= p.ctas || solve_body<F>(p, smem, s_bar, s_red, s_dec);
    // (the CTA that reports the results may have had all it waits for when another had not)
    if (!done && threadIdx.x == 0) p.out_i[OUT_GAVE_UP] = 1;
    if (F == FORM_CLUSTER) cl_close(!done);   // (every wait before has a deadline, so every CTA gets here)
}

// b_r = Bop_r q for every bank entry (blockIdx.y), one warp per row.
struct BiasPtrs {
    const float* Bop[RQ_MAX_RHO];
    float* bias[RQ_MAX_RHO];
};

__global__ void __launch_bounds__(256) bias_kernel(BiasPtrs b, int rows, int n, const float* __restrict__ q) {
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (r >= rows) return;
    const float* w = b.Bop[blockIdx.y] + (size_t)r * n;
    float v = 0.f;
    int k = lane;
    for (; k + 7 * 32 < n; k += 8 * 32) {      // eight loads in flight, the products in order
        float x[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = __ldg(w + k + 32 * t);
#pragma unroll
        for (int t = 0; t < 8; ++t) v = fmaf(x[t], __ldg(q + k + 32 * t), v);
    }
    for (; k < n; k += 32) v = fmaf(__ldg(w + k), __ldg(q + k), v);
    v = warp_sum(v);
    if (lane == 0) b.bias[blockIdx.y][r] = v;
}

// Slices of the rows: per CTA xr rows of x and ar rows of A x (the cluster form: multiples
// of 4, so that a warp's 4 entries leave as one 16-byte store); CTAs with rows: a prefix.
void slices(relu_qp_t h, int ctas, bool cl, int* xr, int* ar, int* used) {
    int a = ceil_div(h->n, ctas), b = h->m > 0 ? ceil_div(h->m, ctas) : 0;
    if (cl) {
        a = (int)round_up(a, 4);
        b = (int)round_up(b, 4);
    }
    *xr = a;
    *ar = b;
    *used = std::max(ceil_div(h->n, a), b > 0 ? ceil_div(h->m, b) : 0);
}

// Above this many entries the grid counts its CTAs instead of tagging the entries: every CTA
// polls all of the words (measured per layer, words against count: 1.80 / 2.73 us at 1280
// entries, 2.54 / 3.05 at 1600, 7.7 / 5.2 at 3200).
constexpr int kTagMax = 2048;

Form form_of(relu_qp_t h, int ctas, int cluster) {
    return cluster > 1 ? FORM_CLUSTER : ctas == 1 ? FORM_ONE : h->R <= kTagMax ? FORM_GRID : FORM_COUNT;
}

// lam_std is staged over the operand where the two together pass 208 KB: of a CTA's 227 KB the
// maxima and the state of its rows take up to 15 KB on 152 CTAs (n + m = 40000).
constexpr size_t kStageMax = 53248;
bool share_lam(relu_qp_t h, int ctas, int cluster) {
    return form_of(h, ctas, cluster) == FORM_COUNT && h->ldw + round_up(h->m, 4) > kStageMax;
}

// gs: rows of a warp's group (the cluster form: 4, one 16-byte store)
void fill_params(relu_qp_t h, SP& p, int ctas, int cluster, int gs, int cached) {
    const int n = h->n, m = h->m;
    p.n = n; p.m = m; p.R = h->R; p.ldw = h->ldw;
    p.ldp = (int)round_up(n, 4);
    p.ldt = (int)round_up(m > 0 ? m : 1, 4);
    p.nr = h->nr;
    for (int r = 0; r < h->nr; ++r) {
        p.Wt[r] = h->be[r].Wt;
        p.bias[r] = h->be[r].bias;
        p.rho[r] = h->be[r].rho;
    }
    p.P = h->P32; p.A = h->A32; p.At = h->At32;
    p.q = h->q32; p.l = h->l32; p.u = h->u32; p.rs = h->rs32;
    p.rsx = h->sc_rx; p.rsz = h->sc_z;
    p.qnorm = h->qnorm;
    slices(h, ctas, cluster > 1, &p.xr, &p.ar, &p.ctas);
    p.cached_rows = cached;
    // the rows outside shared memory over as many warps as the cached ones leave
    const int out = p.xr + p.ar - cached, free_warps = std::max(1, kWarps - ceil_div(cached, gs));
    p.gu = out <= free_warps ? 1 : out <= 2 * free_warps ? 2 : 4;
    p.gs = gs;
    p.share = share_lam(h, ctas, cluster) ? 1 : 0;
    p.timeout_ns = 2000000000LL;
}

// cached rows of W + the operand (two buffers but in the grid form) + lam_std + every CTA's
// maxima + the state of the CTA's rows
size_t smem_bytes(relu_qp_t h, int cached_rows, int ctas, int cluster) {
    int xr, ar, used;
    slices(h, ctas, cluster > 1, &xr, &ar, &used);
    return (((size_t)cached_rows + (is_grid(form_of(h, ctas, cluster)) ? 1 : 2)) * h->ldw +
            (share_lam(h, ctas, cluster) ? 0 : round_up(h->m > 0 ? h->m : 1, 4)) + RED_WORDS * (size_t)used +
            kState * (size_t)(xr + ar)) *
           sizeof(float);
}

const void* kernel_of(relu_qp_t h, int ctas, int cluster) {
    switch (form_of(h, ctas, cluster)) {
        case FORM_COUNT: return (const void*)single_solve_kernel<FORM_COUNT>;
        case FORM_CLUSTER: return (const void*)single_solve_kernel<FORM_CLUSTER>;
        case FORM_ONE: return (const void*)single_solve_kernel<FORM_ONE>;
        default: return (const void*)single_solve_kernel<FORM_GRID>;
    }
}

// Rows of Wt a CTA can cache: what the opt-in shared memory holds beside the rest; -1 when
// not even the rest fits.  (Also readies the shape's kernel for its launches.)
int cached_rows_for(relu_qp_t h, int ctas, int cluster) {
    int room = 0;
    if (allow_shared(h, kernel_of(h, ctas, cluster), &room) != RELU_QP_OK) return -1;
    int xr, ar, used;
    slices(h, ctas, cluster > 1, &xr, &ar, &used);
    const long left = (long)room - 256 - (long)smem_bytes(h, 0, ctas, cluster);
    if (left < 0) return -1;
    return (int)std::min<long>(xr + ar, left / (long)((size_t)h->ldw * sizeof(float)));
}

cudaLaunchConfig_t cluster_config(relu_qp_t h, int ctas, size_t smem, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = h->stream;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)ctas;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// Launch the solve kernel: a cooperative grid of `ctas` CTAs, one CTA, or (cluster > 1) one
// cluster of `ctas` CTAs.
int launch_kernel(relu_qp_t h, SP& p, int ctas, int cluster) {
    const size_t smem = smem_bytes(h, p.cached_rows, ctas, cluster);
    const void* k = kernel_of(h, ctas, cluster);
    void* args[] = {&p};
    if (cluster > 1) {
        cudaLaunchAttribute at[1];
        const cudaLaunchConfig_t cfg = cluster_config(h, ctas, smem, at);
        RQ_CUDA(h, cudaLaunchKernelExC(&cfg, k, args));
    } else if (ctas == 1) {
        RQ_CUDA(h, cudaLaunchKernel(k, dim3(1), dim3(kThreads), args, smem, h->stream));
    } else {
        RQ_CUDA(h, cudaLaunchCooperativeKernel(k, dim3(ctas), dim3(kThreads), args, smem, h->stream));
    }
    return RELU_QP_OK;
}

// Whether the shape can be resident.
bool fits(relu_qp_t h, int ctas, int cluster, int cached) {
    if (cached < 0) return false;
    const size_t smem = smem_bytes(h, cached, ctas, cluster);
    const void* k = kernel_of(h, ctas, cluster);
    bool ok;
    int n = 0;
    if (cluster > 1) {
        ok = cluster <= 8 || cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        cudaLaunchAttribute at[1];
        const cudaLaunchConfig_t cfg = cluster_config(h, ctas, smem, at);
        ok = ok && cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n >= 1;
    } else {
        ok = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kThreads, smem) == cudaSuccess && n >= 1 &&
             ctas <= n * h->num_sms;
    }
    cudaGetLastError();
    return ok;
}

// Words of the grids' exchanges for this problem, and the pointers into them: the operand
// (tagged words, or plain buffers of ldw floats), lam_std, the maxima, the count.
size_t operand_words(relu_qp_t h) { return std::max(2 * round_up(h->R, 2), (size_t)h->ldw); }
size_t exchange_words(relu_qp_t h, int max_ctas) {
    return operand_words(h) + round_up(h->m, 2) + RED_WORDS * (size_t)max_ctas + 2;
}
void set_words(relu_qp_t h, SP& p, unsigned long long* w) {
    p.wop = w;
    p.sop = reinterpret_cast<float*>(w);
    p.wls = w + operand_words(h);
    p.wred = p.wls + round_up(h->m, 2);
    p.count = reinterpret_cast<unsigned*>(p.wred + RED_WORDS * (size_t)h->sw.max_ctas);
}

// The exchange numbers start above every tag an earlier launch left in the words; the words
// are zeroed (numbers start over) after a failure and before the numbers wrap around.
int reset_words(relu_qp_t h) {
    SingleWork& w = h->sw;
    RQ_CUDA(h, cudaMemsetAsync(w.words, 0, sizeof(unsigned long long) * exchange_words(h, w.max_ctas), h->stream));
    RQ_CUDA(h, cudaMemsetAsync(w.err, 0, sizeof(int), h->stream));
    w.tag = w.count = 0;
    return RELU_QP_OK;
}

int launch(relu_qp_t h, int ctas, int cluster, int cached, int gs, const float* xin, const float* lin, int rho_index,
           double eps_abs, double eps_rel, int max_iter, int check_interval, int adaptive) {
    SingleWork& w = h->sw;
    if (w.tag > 0xC0000000u) RQ_TRY(reset_words(h));
    SP p{};
    fill_params(h, p, ctas, cluster, gs, cached);
    set_words(h, p, w.words);
    p.rho_index0 = rho_index;
    p.check_interval = check_interval;
    p.adaptive = adaptive;
    p.max_iter = max_iter;
    p.eps_abs = eps_abs;
    p.eps_rel = eps_rel;
    p.xin = xin;
    p.lin = lin;
    p.xo = w.out;
    p.zo = w.out + h->n;
    p.lo = w.out + h->n + h->m;
    p.tag0 = w.tag;
    p.count0 = w.count;
    w.last_ctas = p.ctas;
    w.counted = form_of(h, ctas, cluster) == FORM_COUNT;
    p.err = w.err;
    p.out_i = w.out_i;
    p.out_f = w.out_f;
    w.out_i[OUT_LAST] = -1;    // the kernel's results go to host memory
    w.out_i[OUT_GAVE_UP] = 0;
    return launch_kernel(h, p, ctas, cluster);
}

// After the launch has been waited for: its error, or the next free exchange number.
int finish(relu_qp_t h, const char* what) {
    SingleWork& w = h->sw;
    if (w.out_i[OUT_LAST] < 0 || w.out_i[OUT_GAVE_UP]) {
        RQ_TRY(reset_words(h));
        RQ_CUDA(h, cudaStreamSynchronize(h->stream));
        return fail(h, RELU_QP_ERR_TIMEOUT, std::string("a wait passed its deadline ") + what);
    }
    w.tag += (unsigned)w.out_i[OUT_LAST] + 2u;
    if (w.counted) w.count += ((unsigned)w.out_i[OUT_LAST] + 1u) * (unsigned)w.last_ctas;
    return RELU_QP_OK;
}

}  // namespace

static int compute_bias(relu_qp_t h) {
    BiasPtrs b{};
    for (int r = 0; r < h->nr; ++r) {
        b.Bop[r] = h->be[r].Bop;
        b.bias[r] = h->be[r].bias;
    }
    bias_kernel<<<dim3(ceil_div(h->R, 8), h->nr), 256, 0, h->stream>>>(b, h->R, h->n, h->q32);
    RQ_CUDA(h, cudaGetLastError());
    return RELU_QP_OK;
}

int single_alloc(relu_qp_t h) {
    SingleWork& w = h->sw;
    const size_t n = h->n, m = h->m;
    w.max_ctas = 4 * h->num_sms;
    RQ_TRY(alloc(h, &w.words, exchange_words(h, w.max_ctas)));
    RQ_TRY(alloc(h, &w.err, 4));
    RQ_TRY(alloc(h, &w.in, n + m));
    // pinned: staging of q, l, u, staging of a warm start, the results the kernel writes
    const size_t floats = 2 * (n + 2 * m) + (n + m) + 2 * RED_WORDS;
    RQ_CUDA(h, cudaHostAlloc(reinterpret_cast<void**>(&w.pin), sizeof(float) * floats, cudaHostAllocDefault));
    w.pin_in = w.pin + (n + 2 * m);
    w.out = w.pin_in + (n + m);
    w.out_f = w.out + (n + 2 * m);
    w.out_i = reinterpret_cast<int*>(w.out_f + RED_WORDS);
    return RELU_QP_OK;
}

void single_release(relu_qp_t h) {
    if (h->sw.pin) cudaFreeHost(h->sw.pin);
    h->sw.pin = nullptr;
}

// Group size of a shape before it is tuned: the fewest rows that give every warp a group.
int default_gs(relu_qp_t h, int ctas, int cluster) {
    int xr, ar, used;
    slices(h, ctas, cluster > 1, &xr, &ar, &used);
    const int want = ceil_div(xr + ar, kWarps);
    return cluster > 1 || want > 2 ? 4 : want;
}

// Choose the launch shape by timing 50 fixed-rho layers (no checks) of every candidate that
// can be resident, then the rows of a warp's group.
int single_prepare(relu_qp_t h) {
    SingleWork& w = h->sw;
    w.grid = 0;
    auto time = [&](int g, int cl, int cached, int gs, bool warm, float* ms) -> int {
        RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
        RQ_TRY(launch(h, g, cl, cached, gs, nullptr, nullptr, 0, 0.0, 0.0, warm ? 10 : 50, 0, 0));
        RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
        RQ_CUDA(h, cudaStreamSynchronize(h->stream));
        RQ_TRY(finish(h, "while tuning the solve"));
        RQ_CUDA(h, cudaEventElapsedTime(ms, h->ev0, h->ev1));
        return RELU_QP_OK;
    };
    // Grids, then clusters, the largest first: beyond its minimum the time rises with the rows
    // per CTA (a small grid or cluster of a large problem takes 100 times the best: 25 ms of the
    // setup at n = m = 800).
    struct Shape {
        int ctas, cluster, cached;
    };
    std::vector<Shape> shapes{{h->num_sms, 0, -1}};
    for (int g = 1; g <= 4 * h->num_sms; g *= 2) shapes.push_back({g, 0, -1});
    std::sort(shapes.begin(), shapes.end(), [](const Shape& a, const Shape& b) { return a.ctas > b.ctas; });
    const int grids = (int)shapes.size();
    for (int c : {16, 8, 4, 2}) shapes.push_back({c, c, -1});
    auto possible = [&](Shape& s) {
        s.cached = s.ctas <= h->R ? cached_rows_for(h, s.ctas, s.cluster) : -1;
        return fits(h, s.ctas, s.cluster, s.cached);
    };
    auto use = [&](const Shape& s) {
        w.grid = s.ctas;
        w.cluster = s.cluster;
        w.cached_rows = s.cached;
        w.gs = default_gs(h, s.ctas, s.cluster);
    };
    if (h->opts.single_precision != RELU_QP_PREC_FP32) {
        // a handle of FP64 solves never launches this one: any shape that fits
        for (Shape& s : shapes)
            if (possible(s)) {
                use(s);
                return RELU_QP_OK;
            }
        return fail(h, RELU_QP_ERR_UNSUPPORTED, "the single-QP solve does not fit on an SM");
    }
    auto shape_time = [&](int k, bool warm, float* ms) -> int {
        Shape& s = shapes[k];
        *ms = -1.f;
        if (warm && !possible(s)) return RELU_QP_OK;
        return time(s.ctas, s.cluster, s.cached, default_gs(h, s.ctas, s.cluster), warm, ms);
    };
    float best = 1e30f;
    int chosen = -1;
    std::vector<ShapeTime> timed, clusters;
    RQ_TRY(search_family(grids, shape_time, &best, timed));
    RQ_TRY(search_family((int)shapes.size() - grids,
                         [&](int k, bool warm, float* ms) { return shape_time(grids + k, warm, ms); }, &best, clusters));
    for (const ShapeTime& t : clusters) timed.push_back({grids + t.k, t.ms});
    RQ_TRY(pick_shape(timed, shape_time, &chosen));
    if (chosen < 0) return fail(h, RELU_QP_ERR_UNSUPPORTED, "the single-QP solve does not fit on an SM");
    const Shape s = shapes[chosen];
    use(s);
    if (w.cluster > 1) return RELU_QP_OK;
    // (groups of other sizes are within some 5 %: one run each)
    float least = 1e30f;
    for (const ShapeTime& t : timed)
        if (t.k == chosen) least = t.ms;
    const int gs0 = w.gs;
    for (int gs : {1, 2, 4}) {
        float ms = 0.f;
        if (gs == gs0) continue;
        RQ_TRY(time(s.ctas, 0, s.cached, gs, true, &ms));
        RQ_TRY(time(s.ctas, 0, s.cached, gs, false, &ms));
        if (ms >= least) continue;
        least = ms;
        w.gs = gs;
    }
    return RELU_QP_OK;
}

int single_get_config(relu_qp_t h, int* ctas, int* cluster, int* cached_rows) {
    if (h->sw.grid <= 0) return fail(h, RELU_QP_ERR_INVALID, "the single-QP solve is not set up");
    if (ctas) *ctas = h->sw.grid;
    if (cluster) *cluster = h->sw.cluster > 1 ? h->sw.cluster : 0;
    if (cached_rows) *cached_rows = h->sw.cached_rows;
    return RELU_QP_OK;
}

int single_set_config(relu_qp_t h, int ctas, int cluster) {
    if (h->sw.grid <= 0) return fail(h, RELU_QP_ERR_INVALID, "the single-QP solve is not set up");
    if (ctas < 1 || ctas > h->R || cluster < 0 || (cluster > 1 && cluster != ctas) ||
        (cluster > 1 && cluster != 2 && cluster != 4 && cluster != 8 && cluster != 16))
        return fail(h, RELU_QP_ERR_INVALID, "ctas in [1, n + m]; cluster 0 or cluster = ctas in {2, 4, 8, 16}");
    const int cl = cluster > 1 ? cluster : 0;
    const int cached = cached_rows_for(h, ctas, cl);
    if (ctas > h->sw.max_ctas || !fits(h, ctas, cl, cached))
        return fail(h, RELU_QP_ERR_UNSUPPORTED, cl ? "a cluster of this size cannot be resident"
                                                   : "that many CTAs cannot be co-resident");
    h->sw.grid = ctas;
    h->sw.cluster = cl;
    h->sw.cached_rows = cached;
    h->sw.gs = default_gs(h, ctas, cl);
    return RELU_QP_OK;
}

int single_update(relu_qp_t h) {
    RQ_CUDA(h, cudaMemcpyAsync(h->q32, h->sw.pin, sizeof(float) * (h->n + 2 * (size_t)h->m), cudaMemcpyHostToDevice,
                               h->stream));
    return compute_bias(h);
}

void fill_info(relu_qp_t h, relu_qp_info* info) {
    if (!info) return;
    const SingleWork& w = h->sw;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, h->ev0, h->ev1);
    info->status = w.out_i[OUT_STATUS];
    info->iters = w.out_i[OUT_ITERS];
    info->rho_index = w.out_i[OUT_RHO];
    info->rho_switches = w.out_i[OUT_SWITCHES];
    info->r_prim = w.out_f[0];
    info->r_dual = w.out_f[1];
    info->solve_ms = ms;
}

// x_warm, lam_warm: the host's FP32 warm start (lam_warm may be nullptr: zeros).  The
// results are in h->sw.out: x, z, lam.
int single_solve(relu_qp_t h, const float* x_warm, const float* lam_warm, int rho_index, double eps_abs,
                 double eps_rel, int max_iter, relu_qp_info* info) {
    SingleWork& w = h->sw;
    const size_t n = h->n, m = h->m;
    const bool lam = x_warm && lam_warm && m > 0;
    if (x_warm) {
        std::memcpy(w.pin_in, x_warm, sizeof(float) * n);
        if (lam) std::memcpy(w.pin_in + n, lam_warm, sizeof(float) * m);
        RQ_CUDA(h, cudaMemcpyAsync(w.in, w.pin_in, sizeof(float) * (n + (lam ? m : 0)), cudaMemcpyHostToDevice, h->stream));
    }
    RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
    RQ_TRY(launch(h, w.grid, w.cluster, w.cached_rows, w.gs, x_warm ? w.in : nullptr, lam ? w.in + n : nullptr, rho_index, eps_abs,
                  eps_rel, max_iter, h->opts.check_interval, h->opts.adaptive_rho));
    h->launches += 1;
    RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    RQ_TRY(finish(h, "in relu_qp_solve"));
    fill_info(h, info);
    return RELU_QP_OK;
}


// ---------------------------------------------------------------------------
// Solve without allocating: the scratch of the cooperative solve lives in a
// fixed, file-scope device array instead of buffers allocated at setup.
//
// Some callers cannot allocate device memory at the time they solve: a
// real-time control loop whose cycle must not stall on cudaMalloc (which can
// synchronise the device and take unbounded time), or a host application
// whose allocator owns all device memory.  They set the problem up once (the
// layer bank is still built by relu_qp_setup) and then solve with
// relu_qp_solve_noalloc, which only launches kernels and copies.
//
// Every GPU that loads the library holds this array until the process exits.
// All calls share it, so two calls whose GPU work overlaps (on different
// streams, or from different threads) race on it; calls must be ordered.
// It keeps the contents of the last call; each call clears the parts that
// must start at zero.
// ---------------------------------------------------------------------------
namespace {

// the grid form's exchange words for n + m <= kNoAllocMaxRows and the error word; 49152
// floats = 192 KiB.
constexpr int kNoAllocMaxRows = 4096;
constexpr size_t kNoAllocWords = 49152;
static __device__ __align__(256) float g_noalloc_scratch[kNoAllocWords];

constexpr int kMaxDevices = 64;
float* g_noalloc_ptr[kMaxDevices] = {};
std::mutex g_noalloc_mutex;

// Device address of the array on the handle's device, looked up once per
// device (a host-side use of the symbol itself would not be a device address).
// The lookup is made with h->device current, whatever device the calling
// thread has made current, because the stream and every buffer of the solve
// belong to h->device.
int noalloc_scratch(relu_qp_t h, float** out) {
    const int dev = h->device;
    if (dev < 0 || dev >= kMaxDevices) return fail(h, RELU_QP_ERR_UNSUPPORTED, "device ordinal >= 64");
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        int cur = 0;
        RQ_CUDA(h, cudaGetDevice(&cur));
        if (cur != dev) RQ_CUDA(h, cudaSetDevice(dev));
        void* ptr = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (cur != dev) cudaSetDevice(cur);
        if (e != cudaSuccess || !ptr) {
            cudaGetLastError();
            return fail(h, RELU_QP_ERR_CUDA, std::string("cudaGetSymbolAddress(scratch): ") + cudaGetErrorString(e));
        }
        g_noalloc_ptr[dev] = static_cast<float*>(ptr);
    }
    *out = g_noalloc_ptr[dev];
    return RELU_QP_OK;
}

// The caller's warm-start and output pointers must be device (or managed)
// memory of the handle's device: anything else would reach the kernels and
// the device-to-device copies unchecked.  NULL passes (optional arguments are
// checked by the caller).
int noalloc_check_ptr(relu_qp_t h, const void* ptr, const char* name) {
    if (!ptr) return RELU_QP_OK;
    cudaPointerAttributes a{};
    const cudaError_t e = cudaPointerGetAttributes(&a, ptr);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(h, RELU_QP_ERR_INVALID, std::string(name) + " is not a CUDA pointer");
    }
    const bool on_device = a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
    if (!on_device || (a.type == cudaMemoryTypeDevice && a.device != h->device))
        return fail(h, RELU_QP_ERR_INVALID,
                    std::string(name) + " must be device FP32 memory of device " + std::to_string(h->device));
    return RELU_QP_OK;
}

}  // namespace

int single_solve_noalloc(relu_qp_t h, const float* x_warm, const float* lam_warm, int rho_index, double eps_abs,
                         double eps_rel, int max_iter, float* x_out, float* z_out, float* lam_out,
                         relu_qp_info* info) {
    const size_t words = exchange_words(h, h->sw.max_ctas);
    if (h->R > kNoAllocMaxRows || 2 * words + 4 > kNoAllocWords)
        return fail(h, RELU_QP_ERR_INVALID, "relu_qp_solve_noalloc supports n + m <= " +
                                                std::to_string(kNoAllocMaxRows) + " (fixed scratch of " +
                                                std::to_string(kNoAllocWords * 4 / 1024) + " KiB)");
    RQ_TRY(noalloc_check_ptr(h, x_warm, "x_warm"));
    RQ_TRY(noalloc_check_ptr(h, lam_warm, "lam_warm"));
    RQ_TRY(noalloc_check_ptr(h, x_out, "x_out"));
    RQ_TRY(noalloc_check_ptr(h, z_out, "z_out"));
    RQ_TRY(noalloc_check_ptr(h, lam_out, "lam_out"));
    float* base = nullptr;
    RQ_TRY(noalloc_scratch(h, &base));
    SingleWork& w = h->sw;
    SP p{};
    fill_params(h, p, w.grid, w.cluster, w.gs, w.cached_rows);
    set_words(h, p, reinterpret_cast<unsigned long long*>(base));
    p.err = reinterpret_cast<int*>(base + 2 * words);
    p.rho_index0 = rho_index;
    p.check_interval = h->opts.check_interval;
    p.adaptive = h->opts.adaptive_rho;
    p.max_iter = max_iter;
    p.eps_abs = eps_abs;
    p.eps_rel = eps_rel;
    p.xin = x_warm;
    p.lin = lam_warm;
    p.xo = x_out;
    p.zo = h->m > 0 ? z_out : nullptr;
    p.lo = h->m > 0 ? lam_out : nullptr;
    p.tag0 = 0;                    // the words start at zero: other handles leave theirs in the array
    p.out_i = w.out_i;
    p.out_f = w.out_f;
    w.out_i[OUT_LAST] = -1;
    w.out_i[OUT_GAVE_UP] = 0;
    RQ_CUDA(h, cudaMemsetAsync(base, 0, sizeof(float) * (2 * words + 4), h->stream));
    RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
    RQ_TRY(launch_kernel(h, p, w.grid, w.cluster));
    RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    if (w.out_i[OUT_LAST] < 0 || w.out_i[OUT_GAVE_UP])
        return fail(h, RELU_QP_ERR_TIMEOUT, "a wait passed its deadline in relu_qp_solve_noalloc");
    fill_info(h, info);
    return RELU_QP_OK;
}

}  // namespace rq
