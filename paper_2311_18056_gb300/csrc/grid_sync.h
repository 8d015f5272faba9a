// Grid-wide barrier of the cooperative kernels (batch_tail.cu): every CTA of the launch must be
// co-resident.  bar[0] counts every arrival of the launch (zeroed before the
// launch, never reset during it); each CTA keeps the number of barriers it has
// passed (its epoch), so barrier e is complete once the count reaches
// e * expected.  Thread 0 of each CTA arrives with a release reduction (no
// return value to wait for; the release covers the CTA's stores, ordered before
// it by __syncthreads) and polls the count with acquire loads, each issued
// together with a relaxed load of the error word.  Every wait has a deadline:
// past it the kernel's error word is set to RELU_QP_ERR_TIMEOUT; a CTA that
// sees the error word set leaves at once, and the barrier returns false in
// every thread of the CTA, so the caller returns from the kernel.
//
// The same header holds the exchange of the kernels that run as one
// thread-block cluster (below), which waits on mbarriers.
//
// The arrival and wait logic is written once (barrier_arrive_wait) over a
// policy of memory operations: the device policy below uses PTX atomics at GPU
// scope and %globaltimer; diag.cu instantiates it with host atomics so that
// host threads can exercise the same logic, deadline included.
#pragma once

#include "../../include/relu_qp.h"

namespace rq {

// One arrival of `expected` participants on the arrival counter *count;
// `epoch` is the caller's number of barriers passed on it.  False if the wait
// passed timeout_ns (err set to RELU_QP_ERR_TIMEOUT) or another participant
// has set err.
#pragma nv_exec_check_disable
template <class Ops>
__host__ __device__ inline bool barrier_arrive_wait(Ops& o, unsigned* count, int* err, unsigned expected,
                                                    unsigned& epoch, long long timeout_ns) {
    const unsigned target = (++epoch) * expected;   // modulo 2^32, as the count
    o.add_release(count, 1u);
    long long t0 = 0;
    bool timing = false;
    while (true) {
        const int e = o.load_error(err);
        const unsigned v = o.load_acquire(count);
        if (e != 0) return false;
        if (static_cast<int>(v - target) >= 0) return true;
        const long long t = o.now_ns();
        if (!timing) {
            t0 = t;
            timing = true;
        } else if (t - t0 > timeout_ns) {
            o.set_error(err, RELU_QP_ERR_TIMEOUT);
            return false;
        }
        o.relax();
    }
}

#ifdef __CUDACC__
__device__ __forceinline__ long long grid_sync_timer() {
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Device policy of barrier_arrive_wait: atomics at GPU scope.
struct GridSyncDeviceOps {
    __device__ __forceinline__ void add_release(unsigned* p, unsigned v) {
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
    }
    __device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return v;
    }
    __device__ __forceinline__ int load_error(const int* p) {
        int v;
        asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return v;
    }
    __device__ __forceinline__ long long now_ns() { return grid_sync_timer(); }
    __device__ __forceinline__ void relax() {}
    __device__ __forceinline__ void set_error(int* err, int code) { atomicExch(err, code); }
};

// Per-CTA state of the grid barrier, in shared memory: `epoch` (read and
// written by thread 0 only) counts the barriers the CTA has passed; `ok` carries
// thread 0's verdict to the CTA.  grid_sync_init runs once at kernel start.
struct GridSyncState {
    unsigned epoch;
    int ok;
};

__device__ __forceinline__ void grid_sync_init(GridSyncState* s) {
    if (threadIdx.x == 0) s->epoch = 0u;
}

// Barrier over `expected` CTAs (gridDim.x for the kernels' own barriers).
__device__ __forceinline__ bool grid_sync_n(unsigned* bar, int* err, long long timeout_ns, GridSyncState* s,
                                            unsigned expected) {
    __syncthreads();
    if (threadIdx.x == 0) {
        GridSyncDeviceOps o;
        int ok = 1;
        if (expected > 1)
            ok = barrier_arrive_wait(o, bar, err, expected, s->epoch, timeout_ns) ? 1 : 0;
        else if (o.load_error(err) != 0)
            ok = 0;
        s->ok = ok;
    }
    __syncthreads();
    return s->ok != 0;
}

__device__ __forceinline__ bool grid_sync(unsigned* bar, int* err, long long timeout_ns, GridSyncState* s) {
    return grid_sync_n(bar, err, timeout_ns, s, gridDim.x);
}

// The error word is set, or the deadline has passed (which sets it).
__device__ __forceinline__ bool sync_give_up(int* err, long long t0, long long timeout_ns) {
    int e;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(e) : "l"(err) : "memory");
    if (e != 0) return true;
    if (grid_sync_timer() - t0 <= timeout_ns) return false;
    atomicExch(err, RELU_QP_ERR_TIMEOUT);
    return true;
}

// ---- exchanges of a cooperative grid ----
// One 64-bit word in global memory: 32 bits of value and the exchange's number, which a
// reader polls together (a 64-bit access is one access; no ordering between words is needed).
__device__ __forceinline__ void put_word(unsigned long long* w, unsigned v, unsigned tag) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(((unsigned long long)tag << 32) | v) : "memory");
}
__device__ __forceinline__ void put_words2(unsigned long long* w, unsigned a, unsigned b, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(w), "l"(t | a), "l"(t | b) : "memory");
}
__device__ __forceinline__ void get_words(const unsigned long long* w, unsigned long long& a, unsigned long long& b) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(w) : "memory");
}

// `count` tagged words from w on (16-byte aligned), by a CTA of THREADS threads: store(k, a, b,
// two) gets words k and (two) k + 1.  False in every thread if a wait gave up.  Four pairs a
// thread are in flight; only pairs that are not there yet are read again.
template <int THREADS, class Store>
__device__ __forceinline__ bool gather_words(const unsigned long long* w, int count, unsigned tag, int* err,
                                             long long timeout_ns, Store store) {
    constexpr int U = 4;
    bool ok = true;
    const int pairs = (count + 1) >> 1;
    for (int b = threadIdx.x; b < pairs && ok; b += U * THREADS) {
        unsigned todo = 0;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (b + u * THREADS < pairs) todo |= 1u << u;
        long long t0 = 0;
        for (int tries = 0; todo; ++tries) {
            unsigned long long a[U], c[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if ((todo >> u) & 1u) get_words(w + 2 * (b + u * THREADS), a[u], c[u]);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!((todo >> u) & 1u)) continue;
                const int k = 2 * (b + u * THREADS);
                const bool two = k + 1 < count;
                if ((unsigned)(a[u] >> 32) != tag || (two && (unsigned)(c[u] >> 32) != tag)) continue;
                todo &= ~(1u << u);
                store(k, (unsigned)a[u], (unsigned)c[u], two);
            }
            if (todo && (tries & 63) == 63) {
                if (t0 == 0) t0 = grid_sync_timer();
                if (sync_give_up(err, t0, timeout_ns)) {
                    ok = false;
                    break;
                }
            }
        }
    }
    return __syncthreads_or(ok ? 0 : 1) == 0;
}

// Arrive (the release covers the CTA's stores) and wait until the count reaches `target`
// (modulo 2^32); false in every thread if the wait gave up.
__device__ __forceinline__ bool count_wait(unsigned* count, unsigned target, int* err, long long timeout_ns) {
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        long long t0 = 0;
        while (ok) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
            if ((int)(v - target) >= 0) break;
            if (t0 == 0) t0 = grid_sync_timer();
            ok = !sync_give_up(err, t0, timeout_ns);
        }
    }
    return __syncthreads_or(ok ? 0 : 1) == 0;
}

// ---- one thread-block cluster instead of a cooperative grid ----
// A CTA's mbarrier counts the bytes that st.async writes into its shared memory:
// one arrival per phase (cl_expect, by the receiver, with the phase's bytes) and
// the bytes themselves.  The receiver arms the next phase once it has seen the
// current one complete, so a phase never completes before its reader has left
// the one before.
__device__ __forceinline__ uint32_t cl_smem(const void* ptr) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(ptr));
}
// shared::cluster address of the shared::cta address `addr` in CTA `rank`
__device__ __forceinline__ uint32_t cl_mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// values into CTA q's copy of this CTA's address, their bytes counted on its mbarrier
__device__ __forceinline__ void cl_send1(uint32_t addr, uint32_t bar, int q, float v) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(cl_mapa(addr, q)),
                 "f"(v), "r"(cl_mapa(bar, q))
                 : "memory");
}
__device__ __forceinline__ void cl_send4(uint32_t addr, uint32_t bar, int q, float a, float b, float c, float d) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                     cl_mapa(addr, q)),
                 "f"(a), "f"(b), "f"(c), "f"(d), "r"(cl_mapa(bar, q))
                 : "memory");
}
__device__ __forceinline__ bool cl_try(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
// false once the error word is set or the deadline has passed
__device__ __forceinline__ bool cl_wait(uint32_t bar, uint32_t parity, int* err, long long timeout_ns) {
    long long t0 = 0;
    while (!cl_try(bar, parity)) {
        if (t0 == 0) t0 = grid_sync_timer();
        if (sync_give_up(err, t0, timeout_ns)) return false;
    }
    return true;
}
// The same by a whole warp, with one verdict for it: lanes poll apart, so that the word of an
// error elsewhere can reach some before the phase completes and find the others done, and a
// warp that went on in part would wait for ever in its next shuffle or barrier.
__device__ __forceinline__ bool cl_wait_warp(uint32_t bar, uint32_t parity, int* err, long long timeout_ns) {
    return __all_sync(0xffffffffu, cl_wait(bar, parity, err, timeout_ns)) != 0;
}
// hardware barrier of every thread of the cluster (no deadline: only where every CTA is
// known to arrive, at the start and at the end of a kernel)
__device__ __forceinline__ void cl_sync_hw() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// What partners sent before a closing cluster barrier lands some us later at most.  A CTA that has
// waited for every byte sent to it can leave after the barrier; one whose wait gave up stays this
// long before its shared memory goes to another.
__device__ __forceinline__ void cl_settle() {
    for (const long long t0 = grid_sync_timer(); grid_sync_timer() - t0 < 50000;) {}
}
// The end of a kernel whose CTAs write into each other's shared memory: reached by every thread
// of the cluster, so that no CTA leaves while a partner may still send to it (a lifetime, no
// order of memory).  `failed`: a wait of this thread gave up; one thread that stays keeps the
// CTA's shared memory.
__device__ __forceinline__ void cl_close(bool failed) {
    __syncthreads();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (failed) cl_settle();
}
#endif

}  // namespace rq
