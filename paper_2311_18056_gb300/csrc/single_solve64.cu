// Single-QP online stage of Algorithm 1 (Sec. III-B) in FP64: the same loop as
// single_solve.cu (layer of Eq. gpu_update in factored form every iteration,
// residuals of Eqs. primal and dual every check_interval layers, penalty rule
// of Eq. rho_update with the nearest bank entry, stop test) with every
// product, state vector and residual in FP64.
//
// Why a second arithmetic: an equality row carries 1000x the penalty of an
// inequality row (Sec. II-B), so the rounding of (Ax - z) enters its
// multiplier step multiplied by up to 1000 rho every layer.  In FP32 that
// noise (~6e-8 |Ax| rho_eq) leaves the dual residual of random QPs with n/4
// equality rows near 1e-5..1e-4, above the 1e-6 tolerance of the random-QP
// benchmark (Sec. V-A); in FP64 the same noise is ~1e-16 |Ax| rho_eq.
//
// Refined form (opts.single_precision = RELU_QP_PREC_FP64R): the FP64 layer
// product is computed once per check interval (the anchor), c = Wt s_ref + b,
// and the other layers apply the FP32 bank to the increment only,
// t = c + Wt32 (s - s_ref), with the element-wise step, the state and the
// checks in FP64.  The FP32 rounding then scales with |s - s_ref|, which
// shrinks as the solve converges, and each layer costs an FP32 row product
// instead of an FP64 one (GB300's FP64 rate is ~1/60 of its FP32 rate).
//
// Work split and exchange as in single_solve.cu: each CTA owns a slice of the rows
// of x and of A x with their state in shared memory, a warp takes a row at a time,
// and the operand's entries carry their own arrival (an FP64 entry is two tagged
// words side by side, an increment one), or, above kTagMax words, the CTAs are
// counted.  The rows of the layer that fit are cached in shared memory: the FP32
// bank's for the increments, else the FP64 bank's; FP64 rows otherwise stream from
// L2 (the FP64 bank of n + m = 3000 is 72 MB).  An FP64 entry goes out only where
// the next layer, or a check, reads it.
//
// Bound: n + m = 513 by the exchange and the chain of FP64 operations behind a row's
// sum (an SM issues one FP64 warp instruction in 16 clocks); n + m = 3000 by the FP64
// pipe, 59 k FMAs per SM and layer at two a clock.  A solve of 100 layers: n = 342 (FP64)
// 599 us with a grid barrier and the rows' state in global memory, 320 us so; n = 1110
// (anchored) 817 and 340 us.
#include "common.h"
#include "grid_sync.h"
#include "shape_search.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>

namespace rq {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
// operand s in shared memory: n + m doubles at most
constexpr int kMaxRows64 = 24576;
// words of an exchange up to which they are tagged
constexpr int kTagMax = 2048;
constexpr int kState = 11;   // doubles of state per row

enum { RED_RP = 0, RED_RD, RED_AX, RED_Z, RED_PX, RED_ATL, RED_WORDS = 8 };
enum { DEC_STOP = 6, DEC_RHO = 7 };   // of the decision's words: 1 + the status to stop with, or 0; bank entry
enum { OUT_STATUS = 0, OUT_ITERS, OUT_RHO, OUT_SWITCHES, OUT_LAST, OUT_COUNTED, OUT_GAVE_UP, OUT_WORDS = 8 };

struct SP64 {
    int n, m, R, nr;
    const double* Wt[RQ_MAX_RHO];
    const float* Wt32[RQ_MAX_RHO];   // refined form: FP32 bank, rows of ldw floats (zero padded)
    int ldw, anchor_every;
    const double* bias[RQ_MAX_RHO];
    double rho[RQ_MAX_RHO];
    const double *P, *A, *At, *q, *l, *u;
    const float* rs;              // per-row penalty scale (1 or eq_scale)
    const double *rsx, *rsz;      // scaled problems: residual factors 1/(c D), 1/E (else nullptr)
    const double *xin, *lin;      // warm start (or nullptr)
    double *xo, *zo, *lo;         // results
    // exchanges: the operand buffers [2] of 2 R words (tagged words, FP64 entries or FP32
    // increments), lam_std, the maxima of three checks, the count of arrivals from count0 on
    unsigned long long* wop;
    double* ls;
    unsigned long long* red;
    unsigned *count, count0;
    unsigned tag0;                // exchange e is tagged tag0 + 1 + e
    int *err, *out_i;
    double* out_f;
    int rho_index0, check_interval, adaptive, max_iter, xr, ar, ctas, cached, share;
    double eps_abs, eps_rel, qnorm;
    long long timeout_ns;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Dot product of a row (in global or, GLOBAL false, in shared memory) with a vector in
// shared memory; the result is valid in every lane.  Eight independent loads per lane are in
// flight per step: a row streams from L2, and fewer leave the FP64 pipe waiting on it.
template <bool GLOBAL>
__device__ __forceinline__ double row_dot(const double* __restrict__ w, const double* __restrict__ s, int len, int lane) {
    double a[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    int k = lane;
    for (; k + 7 * 32 < len; k += 8 * 32) {
        double wv[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) wv[t] = GLOBAL ? __ldg(w + k + 32 * t) : w[k + 32 * t];
#pragma unroll
        for (int t = 0; t < 8; ++t) a[t] = fma(wv[t], s[k + 32 * t], a[t]);
    }
#pragma unroll
    for (int t = 0; t < 7; ++t, k += 32)   // at most 7 steps
        if (k < len) a[t] = fma(GLOBAL ? __ldg(w + k) : w[k], s[k], a[t]);
    return warp_sum(((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7])));
}

// FP32 row (ld floats, 16-byte aligned, zero padded) times an FP32 vector in
// shared memory; the result is valid in every lane.
template <bool GLOBAL>
__device__ __forceinline__ float row_dot32(const float* __restrict__ w, const float* __restrict__ s, int ld, int lane) {
    const float4* w4 = reinterpret_cast<const float4*>(w);
    const float4* s4 = reinterpret_cast<const float4*>(s);
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 4
    for (int k = lane; k < (ld >> 2); k += 32) {
        const float4 a = GLOBAL ? __ldg(w4 + k) : w4[k];
        const float4 b = s4[k];
        a0 = fmaf(a.x, b.x, a0);
        a1 = fmaf(a.y, b.y, a1);
        a2 = fmaf(a.z, b.z, a2);
        a3 = fmaf(a.w, b.w, a3);
    }
    float v = (a0 + a1) + (a2 + a3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void red_max(unsigned long long* slot, int word, double v) {
    atomicMax(slot + word, (unsigned long long)__double_as_longlong(fabs(v)));
}

__device__ __forceinline__ double red_get(const unsigned long long* slot, int word) {
    return __longlong_as_double((long long)__ldcg(slot + word));
}

// TAG: tagged words, else counted CTAs.  False if a wait gave up.
template <bool REFINED, bool TAG>
__device__ __forceinline__ bool solve64_body(const SP64& p, double* smem, double* s_dec, unsigned long long* s_red) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int n = p.n, m = p.m, R = p.R, cta = blockIdx.x;
    const int x0 = cta * p.xr, nx = max(0, min(p.xr, n - x0));
    const int a0 = cta * p.ar, na = max(0, min(p.ar, m - a0));
    const int rows = nx + na, per = p.xr + p.ar, ncache = min(p.cached, rows);
    // the operand (R doubles, or ldw floats of increments), lam_std, the rows' state, cached rows
    double* sv = smem;
    float* dv = reinterpret_cast<float*>(sv);
    const int op = (max(R, (p.ldw + 1) / 2) + 1) & ~1;
    double* svk = p.share ? sv : sv + op;
    double* st = sv + op + (p.share ? 0 : (m + 1) & ~1);
    double *st_bias = st, *st_rr = st + per, *st_z = st_rr + per, *st_lam = st_z + per, *st_rho = st_lam + per,
           *st_l = st_rho + per, *st_u = st_l + per, *st_chk = st_u + per, *st_ls = st_chk + per, *st_c = st_ls + per,
           *st_sref = st_c + per;
    double* wc64 = st + kState * (size_t)per + ((kState * per) & 1);
    float* wc32 = reinterpret_cast<float*>(wc64);
    auto row_of = [&](int lr) { return lr < nx ? x0 + lr : n + a0 + (lr - nx); };
    int ri = p.rho_index0, switches = 0;
    unsigned e = 0, counted = 0, checks = 0;
    // ---- exchange x: FP64 entries or FP32 increments ----
    auto publish64 = [&](unsigned x, int r, double v) {
        if (TAG) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(v);
            put_words2(p.wop + ((size_t)(x & 1) * R + r) * 2, (unsigned)b, (unsigned)(b >> 32), p.tag0 + 1 + x);
        } else {
            reinterpret_cast<double*>(p.wop)[(size_t)(x & 1) * R + r] = v;
        }
    };
    auto publish32 = [&](unsigned x, int r, float v) {
        if (TAG) put_word(p.wop + (size_t)(x & 1) * R * 2 + r, __float_as_uint(v), p.tag0 + 1 + x);
        else reinterpret_cast<float*>(p.wop)[(size_t)(x & 1) * R * 4 + r] = v;
    };
    auto all_arrived = [&]() { return count_wait(p.count, p.count0 + ++counted * (unsigned)p.ctas, p.err, p.timeout_ns); };
    auto receive64 = [&](unsigned x) -> bool {
        if (TAG) {
            __syncthreads();   // the operand's readers are done
            return gather_words<kThreads>(p.wop + (size_t)(x & 1) * R * 2, 2 * R, p.tag0 + 1 + x, p.err, p.timeout_ns,
                                          [&](int k, unsigned a, unsigned b, bool) {
                                              sv[k >> 1] = __longlong_as_double((long long)(((unsigned long long)b << 32) | a));
                                          });
        }
        if (!all_arrived()) return false;
        for (int k = tid; k < R; k += kThreads) sv[k] = __ldcg(reinterpret_cast<const double*>(p.wop) + (size_t)(x & 1) * R + k);
        __syncthreads();
        return true;
    };
    auto receive32 = [&](unsigned x) -> bool {
        if (TAG) {
            __syncthreads();
            for (int k = R + tid; k < p.ldw; k += kThreads) dv[k] = 0.f;
            return gather_words<kThreads>(p.wop + (size_t)(x & 1) * R * 2, R, p.tag0 + 1 + x, p.err, p.timeout_ns,
                                          [&](int k, unsigned a, unsigned b, bool two) {
                                              dv[k] = __uint_as_float(a);
                                              if (two) dv[k + 1] = __uint_as_float(b);
                                          });
        }
        if (!all_arrived()) return false;
        for (int k = tid; k < p.ldw; k += kThreads)
            dv[k] = k < R ? __ldcg(reinterpret_cast<const float*>(p.wop) + (size_t)(x & 1) * R * 4 + k) : 0.f;
        __syncthreads();
        return true;
    };
    auto load_bank = [&]() {
        if (REFINED) {
            const int c4 = p.ldw >> 2;
            for (int k = tid; k < ncache * c4; k += kThreads)
                reinterpret_cast<float4*>(wc32)[k] =
                    __ldg(reinterpret_cast<const float4*>(p.Wt32[ri] + (size_t)row_of(k / c4) * p.ldw) + k % c4);
        } else {
            for (int lr = warp; lr < ncache; lr += kWarps)
                for (int k = lane; k < R; k += 32) wc64[(size_t)lr * R + k] = __ldg(p.Wt[ri] + (size_t)row_of(lr) * R + k);
        }
        for (int lr = tid; lr < rows; lr += kThreads) st_bias[lr] = __ldg(p.bias[ri] + row_of(lr));
    };

    // ---------------- start state ----------------
    if (p.xin)
        for (int k = tid; k < n; k += kThreads) sv[k] = p.xin[k];
    if (tid < RED_WORDS) s_red[tid] = 0ull;
    for (int lr = nx + tid; lr < rows; lr += kThreads) {
        const int i = a0 + lr - nx;
        st_rho[lr] = p.rho[ri] * (double)__ldg(p.rs + i);
        st_l[lr] = __ldg(p.l + i);
        st_u[lr] = __ldg(p.u + i);
        st_lam[lr] = p.lin ? p.lin[i] : 0.0;
        st_z[lr] = 0.0;
    }
    load_bank();
    __syncthreads();
    if (p.xin) {
        for (int lr = nx + warp; lr < rows; lr += kWarps) {
            const double v = row_dot<true>(p.A + (size_t)(a0 + lr - nx) * n, sv, n, lane);
            if (lane == 0) st_z[lr] = v;
        }
        __syncthreads();
    }
    for (int lr = tid; lr < rows; lr += kThreads) {
        const int r = row_of(lr);
        if (lr >= nx) st_rr[lr] = st_lam[lr] / st_rho[lr];   // A x - z = 0
        publish64(0, r, lr < nx ? (p.xin ? p.xin[r] : 0.0) : 2.0 * st_rho[lr] * st_z[lr] - st_lam[lr]);
    }
    if (!receive64(0)) return false;

    for (int it = 1; it <= p.max_iter; ++it) {
        // ---------------- one layer ----------------
        // refined form: an FP64 anchor layer at the start of every check interval (so also
        // after every bank switch), FP32 increment layers in between
        const bool anchor = !REFINED || (it - 1) % p.anchor_every == 0;
        const bool last = it == p.max_iter;
        // the next layer is an anchor, or a check reads x
        const bool full = !REFINED || it % p.anchor_every == 0 || last;
        for (int lr = warp; lr < rows; lr += kWarps) {
            const int r = row_of(lr);
            double t;
            if (anchor) {
                t = !REFINED && lr < ncache ? row_dot<false>(wc64 + (size_t)lr * R, sv, R, lane)
                                            : row_dot<true>(p.Wt[ri] + (size_t)r * R, sv, R, lane);
            } else {
                t = (double)(lr < ncache ? row_dot32<false>(wc32 + (size_t)lr * p.ldw, dv, p.ldw, lane)
                                         : row_dot32<true>(p.Wt32[ri] + (size_t)r * p.ldw, dv, p.ldw, lane));
            }
            if (lane == 0) {
                t += anchor ? st_bias[lr] : st_c[lr];
                if (REFINED && anchor) {
                    st_c[lr] = t;
                    st_sref[lr] = sv[r];
                }
                double snew = t, z = t;
                if (lr >= nx) {
                    const double rr = st_rr[lr], lam = st_rho[lr] * rr;
                    z = fmin(fmax(t + rr, st_l[lr]), st_u[lr]);
                    snew = 2.0 * st_rho[lr] * z - lam;
                    if (full) publish64(e + 1, r, snew);
                    else publish32(e + 1, r, (float)(snew - st_sref[lr]));
                    st_lam[lr] = lam;
                    // (t - z + lam / rho, as the FP32 solve has it, would put an FP64 division
                    // into every layer: n = 342 450 us against 415, n = 1110 anchored 480 against
                    // 425, and the same error against more digits, 2.0e-10 and 3.8e-10)
                    st_rr[lr] = t - z + rr;
                } else if (full) {
                    publish64(e + 1, r, snew);
                } else {
                    publish32(e + 1, r, (float)(snew - st_sref[lr]));
                }
                st_z[lr] = z;
            }
        }
        ++e;
        if (!(full ? receive64(e) : receive32(e))) return false;

        const bool is_check = (p.check_interval > 0) && (it % p.check_interval == 0);
        if (!is_check && !last) continue;

        // ---------------- residuals (Eqs. primal, dual) ----------------
        unsigned long long* slot = p.red + (checks % 3) * RED_WORDS;
        if (cta == 0 && tid < RED_WORDS) p.red[((checks + 1) % 3) * RED_WORDS + tid] = 0ull;
        ++checks;
        for (int lr = warp; lr < rows; lr += kWarps) {
            const int i = a0 + lr - nx;
            const double v = row_dot<true>(lr < nx ? p.P + (size_t)(x0 + lr) * n : p.A + (size_t)i * n, sv, n, lane);
            if (lane != 0) continue;
            st_chk[lr] = v;
            if (lr < nx) {
                red_max(s_red, RED_PX, p.rsx ? v * p.rsx[x0 + lr] : v);
            } else {
                const double zi = st_z[lr], f = p.rsz ? p.rsz[i] : 1.0, ls = st_lam[lr] + st_rho[lr] * (v - zi);
                st_ls[lr] = ls;
                p.ls[i] = ls;
                red_max(s_red, RED_RP, (v - zi) * f);
                red_max(s_red, RED_AX, v * f);
                red_max(s_red, RED_Z, zi * f);
            }
        }
        if (!all_arrived()) return false;
        for (int k = tid; k < m; k += kThreads) svk[k] = __ldcg(p.ls + k);
        __syncthreads();
        for (int lr = warp; lr < nx; lr += kWarps) {
            const int j = x0 + lr;
            const double v = (m > 0) ? row_dot<true>(p.At + (size_t)j * m, svk, m, lane) : 0.0;
            if (lane == 0) {
                const double f = p.rsx ? p.rsx[j] : 1.0;
                red_max(s_red, RED_RD, (st_chk[lr] + __ldg(p.q + j) + v) * f);
                red_max(s_red, RED_ATL, v * f);
            }
        }
        __syncthreads();
        if (tid < RED_WORDS) {
            atomicMax(slot + tid, s_red[tid]);
            s_red[tid] = 0ull;
        }
        if (!all_arrived()) return false;

        // ---------------- decision (identical in every CTA; one warp's FP64) ----------------
        if (warp == 0) {
            const double rp = red_get(slot, RED_RP), rd = red_get(slot, RED_RD);
            const double nAx = red_get(slot, RED_AX), nz = red_get(slot, RED_Z);
            const double nPx = red_get(slot, RED_PX), nAtl = red_get(slot, RED_ATL);
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
                s_dec[RED_RP] = rp;
                s_dec[RED_RD] = rd;
                s_dec[DEC_STOP] = numerical ? 1 + RELU_QP_NUMERICAL : converged ? 1 + RELU_QP_SOLVED : last ? 1 + RELU_QP_MAX_ITER : 0;
                s_dec[DEC_RHO] = nri;
            }
        }
        __syncthreads();
        const int stop = (int)s_dec[DEC_STOP], nri = (int)s_dec[DEC_RHO];
        if (stop) {
            for (int lr = tid; lr < rows; lr += kThreads) {
                if (lr < nx) {
                    p.xo[x0 + lr] = st_z[lr];
                } else {
                    p.zo[a0 + lr - nx] = st_z[lr];
                    p.lo[a0 + lr - nx] = st_ls[lr];
                }
            }
            if (cta == 0 && tid == 0) {
                p.out_i[OUT_STATUS] = stop - 1;
                p.out_i[OUT_ITERS] = it;
                p.out_i[OUT_RHO] = ri;
                p.out_i[OUT_SWITCHES] = switches;
                p.out_i[OUT_COUNTED] = (int)counted;
                p.out_i[OUT_LAST] = (int)e;
                p.out_f[0] = s_dec[RED_RP];
                p.out_f[1] = s_dec[RED_RD];
            }
            return true;
        }
        if (nri == ri) {
            // the directly computed Ax replaces the carried one
            for (int lr = nx + tid; lr < rows; lr += kThreads)
                st_rr[lr] = st_chk[lr] - st_z[lr] + st_lam[lr] / st_rho[lr];
            if (p.share) {
                if (!receive64(e)) return false;   // (lam_std was staged over the operand)
            } else {
                __syncthreads();
            }
            continue;
        }
        // switch: rebase lam' so that the next layer is standard ADMM with the new rho
        ri = nri;
        ++switches;
        for (int lr = tid; lr < rows; lr += kThreads) {
            const int r = row_of(lr);
            double v = st_z[lr];
            if (lr >= nx) {
                const double rho_i = p.rho[ri] * (double)__ldg(p.rs + (r - n)), d = st_chk[lr] - v;
                const double lnew = st_ls[lr] - rho_i * d;
                st_lam[lr] = lnew;
                st_rho[lr] = rho_i;
                st_rr[lr] = d + lnew / rho_i;
                v = 2.0 * rho_i * v - lnew;
            }
            publish64(e + 1, r, v);
        }
        load_bank();
        ++e;
        if (!receive64(e)) return false;
    }
    return true;
}

template <bool REFINED, bool TAG>
__global__ void __launch_bounds__(kThreads, 1) single64_kernel(const __grid_constant__ SP64 p) {
    extern __shared__ __align__(16) double smem[];
    __shared__ double s_dec[RED_WORDS];
    __shared__ unsigned long long s_red[RED_WORDS];
    if ((int)blockIdx.x >= p.ctas) return;
    // (the CTA that reports the results may have had all it waits for when another had not)
    if (!solve64_body<REFINED, TAG>(p, smem, s_dec, s_red) && threadIdx.x == 0) p.out_i[OUT_GAVE_UP] = 1;
}

// b_r = Bop_r q for every bank entry (blockIdx.y), one warp per row.
struct Bias64 {
    const double* Bop[RQ_MAX_RHO];
    double* bias[RQ_MAX_RHO];
};

__global__ void __launch_bounds__(256) bias64_kernel(Bias64 b, int rows, int n, const double* __restrict__ q) {
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (r >= rows) return;
    const double* w = b.Bop[blockIdx.y] + (size_t)r * n;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    int k = lane;
    for (; k + 96 < n; k += 128)
#pragma unroll
        for (int t = 0; t < 4; ++t) a[t] = fma(__ldg(w + k + 32 * t), __ldg(q + k + 32 * t), a[t]);
    for (; k < n; k += 32) a[0] = fma(__ldg(w + k), __ldg(q + k), a[0]);
    const double v = warp_sum((a[0] + a[1]) + (a[2] + a[3]));
    if (lane == 0) b.bias[blockIdx.y][r] = v;
}

bool refined(relu_qp_t h) { return h->opts.single_precision == RELU_QP_PREC_FP64R; }
// (an FP64 exchange is 2 R words; the refined form's common exchange R)
bool tagged(relu_qp_t h) { return (refined(h) ? 1 : 2) * h->R <= kTagMax; }
bool share_lam(relu_qp_t h) { return h->R + h->m > 20000; }

const void* kernel_for(relu_qp_t h) {
    if (refined(h)) return tagged(h) ? (const void*)single64_kernel<true, true> : (const void*)single64_kernel<true, false>;
    return tagged(h) ? (const void*)single64_kernel<false, true> : (const void*)single64_kernel<false, false>;
}

// bytes of a cached row, and of everything else
size_t row_bytes(relu_qp_t h) { return refined(h) ? sizeof(float) * h->ldw : sizeof(double) * h->R; }
size_t smem64(relu_qp_t h, int grid, int cached) {
    const size_t per = ceil_div(h->n, grid) + (h->m > 0 ? ceil_div(h->m, grid) : 0);
    const size_t op = round_up(std::max(h->R, (h->ldw + 1) / 2), 2), lam = share_lam(h) ? 0 : round_up(h->m, 2);
    return sizeof(double) * (op + lam + round_up(kState * per, 2)) + round_up(cached * row_bytes(h), 16);
}

int reset_words(relu_qp_t h) {
    SingleWork64& w = h->sw64;
    RQ_CUDA(h, cudaMemsetAsync(w.words, 0, sizeof(unsigned long long) * 4 * h->R, h->stream));
    RQ_CUDA(h, cudaMemsetAsync(w.count, 0, sizeof(unsigned) * 4, h->stream));
    w.tag = w.counted = 0;
    return RELU_QP_OK;
}

int launch(relu_qp_t h, int grid, const double* xin, const double* lin, int rho_index, double eps_abs, double eps_rel,
           int max_iter, int check_interval, int adaptive) {
    SingleWork64& w = h->sw64;
    if (w.tag > 0xC0000000u) RQ_TRY(reset_words(h));
    SP64 p{};
    p.n = h->n;
    p.m = h->m;
    p.R = h->R;
    p.nr = h->nr;
    p.ldw = h->ldw;
    p.anchor_every = h->opts.check_interval > 0 ? h->opts.check_interval : 25;
    for (int r = 0; r < h->nr; ++r) {
        p.Wt32[r] = h->be[r].Wt;
        p.Wt[r] = h->be[r].Wt64;
        p.bias[r] = h->be[r].bias64;
        p.rho[r] = h->be[r].rho;
    }
    p.P = h->P64; p.A = h->A64; p.At = h->At64;
    p.q = h->q64; p.l = h->l64; p.u = h->u64; p.rs = h->rs32;
    p.rsx = h->sc64_rx;
    p.rsz = h->sc64_z;
    p.xin = xin;
    p.lin = lin;
    p.xo = w.out;
    p.zo = w.out + h->n;
    p.lo = w.out + h->n + h->m;
    p.wop = w.words;
    p.ls = w.lstd;
    p.red = w.red;
    p.count = w.count;
    p.err = reinterpret_cast<int*>(w.count + 2);
    p.count0 = w.counted;
    p.tag0 = w.tag;
    p.out_i = w.out_i;
    p.out_f = w.out_f;
    p.rho_index0 = rho_index;
    p.check_interval = check_interval;
    p.adaptive = adaptive;
    p.max_iter = max_iter;
    p.eps_abs = eps_abs;
    p.eps_rel = eps_rel;
    p.qnorm = h->qnorm;
    p.xr = ceil_div(h->n, grid);
    p.ar = h->m > 0 ? ceil_div(h->m, grid) : 0;
    p.ctas = std::max(ceil_div(h->n, p.xr), p.ar > 0 ? ceil_div(h->m, p.ar) : 0);
    p.share = share_lam(h) ? 1 : 0;
    p.timeout_ns = 2000000000LL;
    // the rows of the bank that fit beside the rest
    const size_t room = w.smem_max - smem64(h, grid, 0);
    p.cached = (int)std::min<size_t>(p.xr + p.ar, room / row_bytes(h));
    const size_t smem = smem64(h, grid, p.cached);
    w.last_ctas = p.ctas;
    w.out_i[OUT_LAST] = -1;   // the kernel's results go to host memory
    w.out_i[OUT_GAVE_UP] = 0;
    RQ_CUDA(h, cudaMemsetAsync(w.red, 0, sizeof(unsigned long long) * 3 * RED_WORDS, h->stream));
    void* args[] = {&p};
    RQ_CUDA(h, cudaLaunchCooperativeKernel(kernel_for(h), dim3(grid), dim3(kThreads), args, smem, h->stream));
    return RELU_QP_OK;
}

// After the launch has been waited for: its error, or the next free exchange numbers.
int finish(relu_qp_t h, const char* what) {
    SingleWork64& w = h->sw64;
    if (w.out_i[OUT_LAST] < 0 || w.out_i[OUT_GAVE_UP]) {
        RQ_TRY(reset_words(h));
        RQ_CUDA(h, cudaStreamSynchronize(h->stream));
        return fail(h, RELU_QP_ERR_TIMEOUT, std::string("a wait passed its deadline ") + what);
    }
    w.tag += (unsigned)w.out_i[OUT_LAST] + 2u;
    w.counted += (unsigned)w.out_i[OUT_COUNTED] * (unsigned)w.last_ctas;
    return RELU_QP_OK;
}

}  // namespace

int single64_alloc(relu_qp_t h, const double* P, const double* A) {
    const int n = h->n, m = h->m, R = h->R, mm = m > 0 ? m : 1;
    if (R > kMaxRows64)
        return fail(h, RELU_QP_ERR_INVALID,
                    "single_precision FP64 supports n + m <= " + std::to_string(kMaxRows64));
    RQ_TRY(alloc(h, &h->P64, (size_t)n * n));
    RQ_TRY(alloc(h, &h->A64, (size_t)mm * n));
    RQ_TRY(alloc(h, &h->At64, (size_t)n * mm));
    RQ_TRY(alloc(h, &h->q64, (size_t)n + 2 * (size_t)m));   // q, l, u
    h->l64 = h->q64 + n;
    h->u64 = h->l64 + m;
    for (int r = 0; r < h->nr; ++r) RQ_TRY(alloc(h, &h->be[r].bias64, (size_t)R));
    SingleWork64& w = h->sw64;
    RQ_TRY(alloc(h, &w.words, 4 * (size_t)R));
    RQ_TRY(alloc(h, &w.lstd, (size_t)mm));
    RQ_TRY(alloc(h, &w.in, (size_t)R));
    RQ_TRY(alloc(h, &w.red, 3 * RED_WORDS));
    RQ_TRY(alloc(h, &w.count, 4));
    // pinned: staging of q, l, u, staging of a warm start, the results the kernel writes
    const size_t doubles = 2 * ((size_t)n + 2 * m) + (size_t)R + 2 * RED_WORDS;
    RQ_CUDA(h, cudaHostAlloc(reinterpret_cast<void**>(&w.pin), sizeof(double) * doubles, cudaHostAllocDefault));
    w.pin_in = w.pin + n + 2 * (size_t)m;
    w.out = w.pin_in + R;
    w.out_f = w.out + n + 2 * (size_t)m;
    w.out_i = reinterpret_cast<int*>(w.out_f + RED_WORDS);
    RQ_CUDA(h, cudaMemcpy(h->P64, P, sizeof(double) * n * n, cudaMemcpyHostToDevice));
    if (m > 0) {
        std::vector<double> At((size_t)n * m);
        for (int i = 0; i < m; ++i)
            for (int j = 0; j < n; ++j) At[(size_t)j * m + i] = A[(size_t)i * n + j];
        RQ_CUDA(h, cudaMemcpy(h->A64, A, sizeof(double) * (size_t)m * n, cudaMemcpyHostToDevice));
        RQ_CUDA(h, cudaMemcpy(h->At64, At.data(), sizeof(double) * At.size(), cudaMemcpyHostToDevice));
    }
    if (h->scaled) {
        std::vector<double> fx(n), fz(mm, 1.0);
        for (int j = 0; j < n; ++j) fx[j] = 1.0 / (h->sC * h->sD[j]);
        for (int i = 0; i < m; ++i) fz[i] = 1.0 / h->sE[i];
        RQ_TRY(alloc(h, &h->sc64_rx, (size_t)n));
        RQ_TRY(alloc(h, &h->sc64_z, (size_t)mm));
        RQ_CUDA(h, cudaMemcpy(h->sc64_rx, fx.data(), sizeof(double) * n, cudaMemcpyHostToDevice));
        RQ_CUDA(h, cudaMemcpy(h->sc64_z, fz.data(), sizeof(double) * mm, cudaMemcpyHostToDevice));
    }
    return RELU_QP_OK;
}

void single64_release(relu_qp_t h) {
    if (h->sw64.pin) cudaFreeHost(h->sw64.pin);
    h->sw64.pin = nullptr;
}

int single64_update(relu_qp_t h) {
    RQ_CUDA(h, cudaMemcpyAsync(h->q64, h->sw64.pin, sizeof(double) * (h->n + 2 * (size_t)h->m), cudaMemcpyHostToDevice,
                               h->stream));
    Bias64 b{};
    for (int r = 0; r < h->nr; ++r) {
        b.Bop[r] = h->be[r].Bop64;
        b.bias[r] = h->be[r].bias64;
    }
    bias64_kernel<<<dim3(ceil_div(h->R, 8), h->nr), 256, 0, h->stream>>>(b, h->R, h->n, h->q64);
    RQ_CUDA(h, cudaGetLastError());
    return RELU_QP_OK;
}

// CTA count of the cooperative launch: the fastest of the co-resident candidates over 50
// fixed-rho layers (no checks), the largest first.
int single64_prepare(relu_qp_t h) {
    SingleWork64& w = h->sw64;
    int room = 0;
    RQ_TRY(allow_shared(h, kernel_for(h), &room));
    w.smem_max = (size_t)room - 256;
    std::vector<int> cands{h->num_sms};
    for (int g = 1; g < h->num_sms; g *= 2) cands.push_back(g);
    std::sort(cands.begin(), cands.end(), std::greater<int>());
    float best = 1e30f;
    int chosen = -1;
    std::vector<ShapeTime> timed;
    auto time = [&](int k, bool warm, float* ms) -> int {
        const int g = cands[k];
        *ms = -1.f;
        if (g > h->R || smem64(h, g, 0) > w.smem_max) return RELU_QP_OK;
        RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
        RQ_TRY(launch(h, g, nullptr, nullptr, 0, 0.0, 0.0, warm ? 10 : 50, 0, 0));
        RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
        RQ_CUDA(h, cudaStreamSynchronize(h->stream));
        RQ_TRY(finish(h, "while tuning the FP64 solve"));
        RQ_CUDA(h, cudaEventElapsedTime(ms, h->ev0, h->ev1));
        return RELU_QP_OK;
    };
    RQ_TRY(search_family((int)cands.size(), time, &best, timed));
    RQ_TRY(pick_shape(timed, time, &chosen));
    if (chosen < 0) return fail(h, RELU_QP_ERR_UNSUPPORTED, "FP64 solve kernel does not fit on an SM");
    w.grid = cands[chosen];
    return RELU_QP_OK;
}

int single64_solve(relu_qp_t h, const double* x_warm, const double* lam_warm, int rho_index, double eps_abs,
                   double eps_rel, int max_iter, double* x_out, double* z_out, double* lam_out,
                   relu_qp_info* info) {
    SingleWork64& w = h->sw64;
    const size_t n = h->n, m = h->m;
    const bool lam = x_warm && lam_warm && m > 0;
    if (x_warm) {
        std::memcpy(w.pin_in, x_warm, sizeof(double) * n);
        if (lam) std::memcpy(w.pin_in + n, lam_warm, sizeof(double) * m);
        RQ_CUDA(h, cudaMemcpyAsync(w.in, w.pin_in, sizeof(double) * (n + (lam ? m : 0)), cudaMemcpyHostToDevice, h->stream));
    }
    RQ_CUDA(h, cudaEventRecord(h->ev0, h->stream));
    RQ_TRY(launch(h, w.grid, x_warm ? w.in : nullptr, lam ? w.in + n : nullptr, rho_index, eps_abs, eps_rel, max_iter,
                  h->opts.check_interval, h->opts.adaptive_rho));
    h->launches += 1;
    RQ_CUDA(h, cudaEventRecord(h->ev1, h->stream));
    RQ_CUDA(h, cudaStreamSynchronize(h->stream));
    RQ_TRY(finish(h, "in the FP64 solve"));
    std::memcpy(x_out, w.out, sizeof(double) * n);
    if (z_out && m > 0) std::memcpy(z_out, w.out + n, sizeof(double) * m);
    if (lam_out && m > 0) std::memcpy(lam_out, w.out + n + m, sizeof(double) * m);
    if (info) {
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
    return RELU_QP_OK;
}

}  // namespace rq
