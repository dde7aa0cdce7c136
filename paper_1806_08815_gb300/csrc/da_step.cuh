// da_step.cuh -- the Digital Annealer's parallel-trial Monte Carlo step
// (Algorithm 2 of arXiv:1806.08815) for many replicas at once.
//
// One group of G warps anneals one replica.  Lane l of warp w owns the V
// consecutive variables i = w*32V + l*V + v (v < V) and keeps their effective
// fields g_i = Q_ii + sum_j W_ij x_j and bits x_i in registers for the whole
// launch.  Per step:
//   (a) every lane forms Delta E_i = (1 - 2 x_i) g_i for its V variables (all
//       N trials of the step run in parallel, Sec. II);
//   (b) Metropolis against the dynamic offset: delta = Delta E - E_off is
//       accepted when delta <= 0, else when u < exp(-beta delta).  u comes from
//       Philox block (i/4, t, replica, 0).  The test is made in the log
//       domain, t = delta beta log2(e) + log2(2^24 u) - 24 < 0, with a
//       hardware log2 of the draw; trials with |t| within a band of 2^-15,
//       wider than the error of that estimate, take the exact test with the
//       library's exponential instead, so every decision equals the exact one;
//   (c) each lane's acceptance bits are already in index order, so the counts of
//       the lanes below (from votes; shuffles at V = 32) locate the j-th accepted
//       variable, j = floor(u * count); the chosen x_k flips while every lane
//       adds +-W[k][i] (16-byte loads of row k, which equals column k, from L2;
//       the fp32 forms read a copy of W in the warp row order, where each load
//       of a warp covers 512 contiguous bytes) to its fields.  The next step's
//       Philox words are computed in the latency of the votes and of that row.
//       E_off returns to 0 on a flip and grows by inc otherwise.
// The energy and the best state are not touched by a step: it appends the flip
// to a log in shared memory, settled 32 flips at a time (settle_log).  A G = 1
// group needs no barrier.  A G > 1 group publishes its lanes' acceptance and
// state masks in shared memory behind one named barrier per step.  The
// best-state test of a launch's last step is left pending
// (ReplicaScalars::check) so that it sees the energy after any recompute
// between launches, as Algorithm 2's result is defined after each complete step;
// a recompute sets it too, for it can lower the energy below the best one
// although the step before it flipped nothing.
//
// Launches cover steps [t0, t1) and keep the state in global memory between
// launches (the fp32 path recomputes the fields between launches).
#pragma once
#include <cstddef>

#include "da_device.cuh"
#include "da_internal.h"
#include "da_replica.cuh"
#include "da_step_common.cuh"
#include "da_tc.cuh"

namespace da {
namespace step_detail {

// A launch whose stop flag is set (a cancelled request of the request loop)
// returns at once and leaves the replica state as it was.  One thread reads
// the flag for the block, so that every warp of the block takes the same
// branch (the G > 1 groups meet at barriers).
__device__ __forceinline__ bool launch_stopped(const StepParams& p)
{
    __shared__ int s_stop;
    if (threadIdx.x == 0) s_stop = p.stop ? *reinterpret_cast<const volatile int*>(p.stop) : 0;
    __syncthreads();
    return s_stop != 0;
}

// What a lane publishes for the choice: its acceptance mask, its state bits and the
// accepted trials on the lanes of its warp below it.
template <int V> struct Published {   // V = 32
    using T = uint4;
    static __device__ __forceinline__ T pack(uint32_t acc, uint32_t x, int excl) { return make_uint4(acc, x, excl, 0); }
    static __device__ __forceinline__ uint32_t acc(const T& e) { return e.x; }
    static __device__ __forceinline__ uint32_t x(const T& e) { return e.y; }
    static __device__ __forceinline__ int excl(const T& e) { return (int)e.z; }
};
template <> struct Published<16> {
    using T = uint2;
    static __device__ __forceinline__ T pack(uint32_t acc, uint32_t x, int excl) { return make_uint2(acc | x << 16, excl); }
    static __device__ __forceinline__ uint32_t acc(const T& e) { return e.x & 0xFFFFu; }
    static __device__ __forceinline__ uint32_t x(const T& e) { return e.x >> 16; }
    static __device__ __forceinline__ int excl(const T& e) { return (int)e.y; }
};
template <> struct Published<8> {
    using T = uint32_t;
    static __device__ __forceinline__ T pack(uint32_t acc, uint32_t x, int excl) { return acc | x << 8 | (uint32_t)excl << 16; }
    static __device__ __forceinline__ uint32_t acc(const T& e) { return e & 0xFFu; }
    static __device__ __forceinline__ uint32_t x(const T& e) { return (e >> 8) & 0xFFu; }
    static __device__ __forceinline__ int excl(const T& e) { return (int)(e >> 16); }
};
template <> struct Published<4> : Published<8> {};

// Of the GA warps of a replica, G of them in this block.
template <typename E, int V, int GA, int G> struct GroupShared {
    uint64_t arrived[2];                         // clusters: a step's entries are here, by step parity
    typename Published<V>::T lanes[2][32 * GA];  // by step parity
    alignas(16) int total[2][(GA + 3) / 4 * 4];  // accepted trials of each warp, by step parity
    FlipEntry log[2][32];                        // by window parity
    FlipHead<E> head[G];
};

// ---- one replica on the blocks of a cluster ---------------------------------------
// Every block of the cluster gets every warp's entries by asynchronous stores into its own
// shared memory, which count their bytes on a barrier there: one way through the cluster
// and no acknowledgement (stores followed by the cluster's barrier took 0.3 us longer per
// step, reading the owner's entries from its block 0.35 us more again).
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_address(uint32_t shared_address, uint32_t rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(shared_address), "r"(rank));
    return a;
}
// bar: the barrier in the block that a lies in
__device__ __forceinline__ void cluster_send(uint32_t a, uint32_t v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a), "r"(v),
                 "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void cluster_send(uint32_t a, uint2 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(a),
                 "r"(v.x), "r"(v.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// A bounded wait for the phase of the given parity (tc::mbar_wait), acquiring what the
// cluster's blocks stored.
__device__ __forceinline__ bool cluster_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
constexpr uint32_t kClusterPolls = 1u << 26;
constexpr uint64_t kClusterNs = 2000000000ull;
__device__ __forceinline__ bool cluster_await(uint32_t bar, uint32_t parity)
{
    if (cluster_try(bar, parity)) return true;
    const uint64_t t0 = tc::global_ns();
    for (uint32_t i = 0; i < kClusterPolls; ++i) {
        if (cluster_try(bar, parity)) return true;
        if ((i & 255u) == 255u && tc::global_ns() - t0 > kClusterNs) return false;
    }
    return false;
}

// After a wait that gave up: time for asynchronous stores on their way to this block, before
// its shared memory goes to another (they take about a microsecond).
__device__ __forceinline__ void cluster_drain()
{
    const uint64_t t0 = tc::global_ns();
    for (uint32_t i = 0; i < (1u << 20) && tc::global_ns() - t0 < 1000000ull; ++i) {}
}

// G > 1 warps per replica: warp w owns the slice [32 V w, 32 V (w + 1)) of the variables.
// One barrier per step: every lane publishes its mask, state bits and in-warp prefix
// count, every warp its total; after the barrier each warp finds the owner warp from the
// G totals and reads only that warp's 32 entries.  Bound by the latency of the step's
// chain (one to two warps per scheduler).  us per step, fp32 with 32 replicas, against
// the form in which every warp scanned all 32 G masks and booked the energy in fp64:
// N = 1024 (G = 4, V = 8) 1.015 -> 0.611, N = 2048 (G = 4, V = 16) 1.168 -> 0.755,
// N = 4096 (G = 8, V = 16) 1.564 -> 1.000, N = 8192 (G = 8, V = 32) 2.712 -> 1.606
// (there the rows of W come from HBM).  16 warps in one block are no faster: N = 2048
// 0.978, N = 4096 1.314, N = 8192 1.955; on several SMs they are (kClusterReplicas in
// da_api.cu).
// C > 1: the replica on the C blocks of a cluster, G warps in each (warp w of block c is
// warp c G + w); published to every block by asynchronous stores, and the wait for the bytes
// they bring (await_step) in the place of the block's barrier.
template <typename Tw, int V, int G, bool FULL, bool TRACE, int C = 1>
__global__ void __launch_bounds__(32 * G * OccupancyGV<G, V>::rpb, OccupancyGV<G, V>::min_blocks)
    step_kernel(const __grid_constant__ StepParams p)
{
    constexpr bool kCoal = sizeof(Tw) == 4 && V >= 8;   // fp32 forms: rows from p.Wc (step_uses_coal)
    constexpr int kRegCap = 65536 / (32 * G * OccupancyGV<G, V>::rpb * OccupancyGV<G, V>::min_blocks);
    constexpr bool kPre = kRegCap >= (V <= 8 ? 96 : V == 16 ? 128 : 255);
    constexpr int GA = G * C;                       // warps of the replica
    using R_ = WarpReplica<Tw, V, false, kPre, kCoal, (V * GA < 32 ? V * GA : 32)>;
    using A = Arith<Tw>;
    using H = typename R_::H;
    using Pub = Published<V>;
    using Shared = GroupShared<typename R_::E, V, GA, G>;
    __shared__ Shared shared[C > 1 ? 1 : OccupancyGV<G, V>::rpb];
    uint32_t rank = 0, peer[C];
    if constexpr (C > 1) {
        rank = cluster_rank();
        if (threadIdx.x == 0) {
            tc::mbar_init(&shared[0].arrived[0], 1);
            tc::mbar_init(&shared[0].arrived[1], 1);
            tc::mbar_init_fence();
        }
        __syncwarp();
        cluster_arrive();                                // every block is there, its barriers initialised
        cluster_wait();
#pragma unroll
        for (int c = 0; c < C; ++c) peer[c] = cluster_address((uint32_t)__cvta_generic_to_shared(&shared[0]), c);
    } else {
        if (launch_stopped(p)) return;
    }
    const int wib = threadIdx.x >> 5;
    const int g = C > 1 ? 0 : wib / G;              // group (replica) within the block
    const int wb = wib - g * G;                     // warp of the group within the block
    const int w = (int)rank * G + wb;               // and within the replica
    const int r = C > 1 ? blockIdx.x / C : blockIdx.x * (blockDim.x / (32 * G)) + g;
    if (r >= p.R) return;
    auto& gs = shared[g];

    R_ rp;
    rp.init(static_cast<const Tw*>(kCoal ? p.Wc : p.W), p.N, kCoal ? p.npad : p.ldw, p.rep_base + (uint32_t)r,
            p.bestx + (size_t)r * p.nw, gs.log[0], &gs.head[wb], w * 32 * V);
    const int lane = rp.lane;
    H* hg = static_cast<H*>(p.h) + (size_t)r * p.npad + rp.base;
    uint32_t* xg = p.x + (size_t)r * p.nw;
    rp.load_fields(hg);
    rp.xm = (xg[rp.base >> 5] >> (rp.base & 31)) & R_::VMASK;
    ReplicaScalars sc = p.sc[r];
    rp.m = sc.m;
    const PhiloxKeys& keys = *reinterpret_cast<const PhiloxKeys*>(&p.round_key[0][0]);
    const bool per_rep = p.betas != nullptr;
    rp.begin(p.t0, p.t1, per_rep ? nullptr : p.beta, per_rep ? p.betas[p.temp_of[r]] : 0.f, A::load_e(sc.E),
             A::load_e(sc.best), sc.flips, keys);
    bool held = sc.check != 0;
    if (held && p.t0 < p.t1) rp.test_current();
    if constexpr (kPre) {
        rp.prep_draws(keys);
        if (p.t0 < p.t1) rp.draw_pre((uint32_t)p.t0, keys);
    } else {
        if (p.t0 < p.t1) rp.draw((uint32_t)p.t0, keys);
    }
    int window = 0;
    // clusters: the number of the step in the launch, its bytes beside the entries (the flip
    // of the step before), whether a wait gave up
    uint32_t sent = 0, extra = 0;
    bool lost = false;
    constexpr uint32_t kStepBytes = 32 * GA * sizeof(typename Pub::T) + GA * sizeof(int);
    auto await_step = [&](uint32_t bytes) {
        if (threadIdx.x == 0) tc::mbar_arrive_expect_tx(&gs.arrived[sent & 1], bytes);
        return cluster_await((uint32_t)__cvta_generic_to_shared(&gs.arrived[sent & 1]), (sent >> 1) & 1);
    };

    auto one_step = [&](uint32_t t, auto& slots) -> int {
        const float Eoff = __fmul_rn(__uint2float_rn(rp.m), p.inc);
        bool unsure;
        uint32_t accm = decide_log<A, V>(rp.h, rp.xm, Eoff, __fmul_rn(rp.beta, kLog2e), rp.lg, unsure);
        const bool any_unsure = __any_sync(0xffffffffu, unsure);
        // the rare exact test: at V = 16 in one block without padding before the count and out
        // of line (N = 2048 with 32 replicas 0.728 -> 0.720 us per step, with 1024 2.80 -> 2.72),
        // else after a first count (N = 500 with 128 replicas 0.487, before it 0.494; N = 8192
        // with 64 1.557, 1.569) and at V = 16 inline (N = 2000 with 64 replicas 0.812, as a call
        // 0.866; N = 8192 on clusters 1.32, 1.44)
        constexpr bool kFirst = V == 16 && C == 1 && FULL, kOut = V != 16 || kFirst;
        auto exact = [&] {
            accm = decide_exact_out<A, V, kOut>(rp.h, rp.xm, Eoff, rp.beta, rp.lg, accm, rp.base, t, rp.rep, keys);
        };
        if (kFirst && any_unsure) exact();
        if constexpr (!FULL) accm &= rp.valid;
        int excl, mine;
        rp.count_below(accm, excl, mine);
        if constexpr (C == 1) slots.template at<0>();
        if (!kFirst && any_unsure) {
            exact();
            if constexpr (!FULL) accm &= rp.valid;
            rp.count_below(accm, excl, mine);
        }
        if constexpr (C > 1) {
            // buffers and barriers by the parity of `sent`; a buffer is free again when the
            // step after it has arrived, for which every warp has left it
            const uint32_t at_lane = (uint32_t)(offsetof(Shared, lanes) +
                                                ((t & 1) * 32 * GA + w * 32 + lane) * sizeof(typename Pub::T));
            const uint32_t at_total = (uint32_t)(offsetof(Shared, total) +
                                                 ((t & 1) * ((GA + 3) / 4 * 4) + w) * sizeof(int));
            const uint32_t at_bar = (uint32_t)(offsetof(Shared, arrived) + (sent & 1) * sizeof(uint64_t));
            const typename Pub::T e = Pub::pack(accm, rp.xm, excl);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                cluster_send(peer[c] + at_lane, e, peer[c] + at_bar);
                if (lane == c) cluster_send(peer[c] + at_total, (uint32_t)mine, peer[c] + at_bar);
            }
            slots.template at<0>();
            const bool ok = await_step(kStepBytes + extra);
            ++sent;
            if (!__all_sync(0xffffffffu, ok)) {
                lost = true;
                return -1;
            }
        } else {
            gs.lanes[t & 1][w * 32 + lane] = Pub::pack(accm, rp.xm, excl);
            if (lane == 0) gs.total[t & 1][w] = mine;
            group_barrier(1 + g, 32 * G);
        }
        // the flips up to the step before are in the log of every warp: settled here, by
        // every warp for its own words
        if (rp.n == 32) {
            rp.settle();
            window ^= 1;
            rp.log = gs.log[window];
        }
        int before[GA];                             // accepted trials on the warps below u
        int total = 0;
#pragma unroll
        for (int u = 0; u < GA; ++u) {
            before[u] = total;
            total += gs.total[t & 1][u];
        }
        if (total == 0) {
            rp.m += 1;
            slots.rest_none();
            rp.next_inputs(t, keys);
            return -1;
        }
        int j = (int)__umulhi(rp.cw, (uint32_t)total);
        int ow = 0, skip = 0;
#pragma unroll
        for (int u = 1; u < GA; ++u)
            if (j >= before[u]) {
                ow = u;
                skip = before[u];
            }
        j -= skip;
        const typename Pub::T e = gs.lanes[t & 1][ow * 32 + lane];
        const uint32_t lower = __ballot_sync(0xffffffffu, Pub::excl(e) + __popc(Pub::acc(e)) <= j);
        slots.template at<1>();
        const int ent = ow * 32 + __popc(lower);
        const typename Pub::T o = gs.lanes[t & 1][ent];
        slots.template at<2>();
        const uint32_t pre = bits_before(Pub::acc(o), j - Pub::excl(o), lane);
        slots.template at<3>();
        const int vk = __popc(pre);
        const uint32_t xold = (Pub::x(o) >> vk) & 1u;
        const int k = ent * V + vk;
        Tw cv[V];
        if (FULL || rp.base < p.N) R_::load_row(rp.W + (size_t)k * rp.ldw + rp.rowoff, cv);
        const bool own = w * 32 + lane == ent;
        if (w == ow) {                              // warp-uniform
            const H gk = select_slot<H, V>(rp.h, vk);
            const FlipEntry f{A::log_bits(A::signed_field(gk, xold)), k};
            if constexpr (C > 1) {
                const uint32_t at = (uint32_t)(offsetof(Shared, log) + (window * 32 + rp.n) * sizeof(FlipEntry));
                if (own) {                          // counted with the next step
                    const uint32_t at_bar = (uint32_t)(offsetof(Shared, arrived) + (sent & 1) * sizeof(uint64_t));
#pragma unroll
                    for (int c = 0; c < C; ++c)
                        cluster_send(peer[c] + at, make_uint2(f.dE, (uint32_t)f.k), peer[c] + at_bar);
                }
            } else {
                if (own) rp.log[rp.n] = f;
            }
        }
        ++rp.n;
        slots.rest_flip();
        rp.next_inputs(t, keys);
        if (FULL || rp.base < p.N) {
            const typename A::Sign sg = A::sign(xold);
#pragma unroll
            for (int v = 0; v < V; ++v) rp.h[v] = A::apply_signed(rp.h[v], cv[v], sg);
        }
        if (own) rp.xm ^= 1u << vk;
        rp.m = 0;
        return k;
    };
    for (uint32_t t = (uint32_t)p.t0; t < (uint32_t)p.t1; ++t) {
        int k;
        if constexpr (kPre) {
            // where the draws' rounds go, measured: V <= 8 and V = 32 have the row load (and V = 32
            // its HBM latency) to fill; N = 1024 (G = 4, V = 8) 0.637 -> 0.620 us per step, N = 4096
            // (G = 8, V = 16) 1.048 -> 1.000, N = 8192 1.743 -> 1.606 against the one-warp split;
            // on clusters the wait for the other blocks takes the first two, at N = 8192 the rest
            // belongs under the row load (1.406 -> 1.356)
            constexpr bool kMid = V == 16 && C == 1;
            constexpr int kR0 = V == 16 ? 5 : 3, kR1 = kMid ? 6 : 5, kR2 = kMid ? 7 : 5,
                          kR3 = C > 1 && V == 16 ? 5 : kMid && G < 8 ? 8 : 7;
            typename R_::template DrawSlots<PhiloxKeys, kR0, kR1, kR2, kR3> s{rp, keys, t + 1};
            k = one_step(t, s);
        } else {
            auto f = [&] { rp.draw(t + 1, keys); };
            typename R_::template RestOnly<decltype(f)> s{f};
            k = one_step(t, s);
        }
        held = k >= 0;
        if constexpr (C > 1) {
            extra = held ? (uint32_t)sizeof(FlipEntry) : 0u;
            if (lost) break;
        }
        if constexpr (TRACE) {
            if (w == 0 && lane == 0) p.trace[(size_t)r * p.trace_T + t] = k;
        }
    }
    // the last flip is in the log
    if constexpr (C > 1) {
        if (!lost && !__all_sync(0xffffffffu, await_step(extra))) lost = true;
        if (lost && lane == 0 && p.err) atomicExch(p.err, 2);
        __syncwarp();
        cluster_arrive();                           // no block leaves while another may still store to it
        cluster_wait();
        if (lost) {                                 // a store sent before that, which no wait here counted, lands
            cluster_drain();
            return;
        }
    } else {
        group_barrier(1 + g, 32 * G);
    }
    if (rp.n > 0) rp.settle(held);

    rp.store_fields(hg);
    const uint32_t word = rp.word();
    if (lane % R_::P == 0) xg[rp.base >> 5] = word;
    if (w == 0 && lane == 0) {
        sc.E = A::store_e(rp.head->E);
        sc.best = A::store_e(rp.head->best);
        sc.flips = rp.head->flips;
        sc.m = rp.m;
        sc.check = held ? 1u : 0u;
        p.sc[r] = sc;
    }
}

// G = 1: one warp per replica, the body of WarpReplica.  The fp32 forms at V >= 8 read their rows from p.Wc
// (the warp row order, pitch 32 V).
template <typename Tw, int V, bool FULL, bool TRACE>
__global__ void __launch_bounds__(32 * OccupancyGV<1, V>::rpb, OccupancyGV<1, V>::min_blocks)
    step_kernel_g1(const __grid_constant__ StepParams p)
{
    constexpr bool kCoal = sizeof(Tw) == 4 && V >= 8;   // float and f32e
    using R_ = WarpReplica<Tw, V, false, true, kCoal, V, V == 32 || (V == 16 && FULL)>;
    using H = typename R_::H;
    __shared__ FlipLog<typename R_::E> logs[OccupancyGV<1, V>::rpb];
    if (launch_stopped(p)) return;
    const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= p.R) return;
    R_ rp;
    rp.init(static_cast<const Tw*>(kCoal ? p.Wc : p.W), p.N, kCoal ? 32 * V : p.ldw, p.rep_base + (uint32_t)r,
            p.bestx + (size_t)r * p.nw, logs[threadIdx.x >> 5].f,
            &logs[threadIdx.x >> 5].head);
    H* hg = static_cast<H*>(p.h) + (size_t)r * p.npad + rp.base;
    uint32_t* xg = p.x + (size_t)r * p.nw;
    rp.load_fields(hg);
    rp.xm = (xg[rp.base >> 5] >> (rp.base & 31)) & R_::VMASK;
    ReplicaScalars sc = p.sc[r];
    rp.m = sc.m;
    const PhiloxKeys& keys = *reinterpret_cast<const PhiloxKeys*>(&p.round_key[0][0]);
    const bool per_rep = p.betas != nullptr;
    rp.begin(p.t0, p.t1, per_rep ? nullptr : p.beta, per_rep ? p.betas[p.temp_of[r]] : 0.f, Arith<Tw>::load_e(sc.E),
             Arith<Tw>::load_e(sc.best), sc.flips, keys);
    bool held = sc.check != 0;       // the best-state test of the last step is still to be made
    if (held && p.t0 < p.t1) rp.test_current();
    rp.prep_draws(keys);
    if (p.t0 < p.t1) rp.draw_pre((uint32_t)p.t0, keys);
    for (uint32_t t = (uint32_t)p.t0; t < (uint32_t)p.t1; ++t) {
        const int k = rp.template step<FULL>(t, t + 1 < p.t1, p.inc, keys);
        held = k >= 0;
        if constexpr (TRACE) {
            if (rp.lane == 0) p.trace[(size_t)r * p.trace_T + t] = k;
        }
    }
    rp.store_fields(hg);
    const uint32_t word = rp.word();
    if (rp.lane % R_::P == 0) xg[rp.base >> 5] = word;
    if (rp.n > 0) rp.settle(held);
    if (rp.lane == 0) {
        sc.E = Arith<Tw>::store_e(rp.head->E);
        sc.best = Arith<Tw>::store_e(rp.head->best);
        sc.flips = rp.head->flips;
        sc.m = rp.m;
        sc.check = held ? 1u : 0u;
        p.sc[r] = sc;
    }
}

// G = 1 with warp specialisation: block = one replica = an annealer warp
// (WarpReplica::step_log) and a producer warp that computes the acceptance
// draws of the coming steps, L = log2 U for every trial, into a ring of
// kWsRing shared-memory buffers.  The producer depends on nothing the
// annealer computes, so it runs up to kWsRing steps ahead; the annealer reads
// the next step's buffer while its row load is in flight.  Full/empty
// handshakes are mbarriers whose waits are bounded (a wait that gives up
// sets *p.err and ends the launch; the replica's results are then invalid,
// and later launches that see the flag leave at once).
//
// Seven blocks per SM, so that 1024 replicas run in one wave, leave 128 registers; at V = 32
// the exact test is inline and the row load unconditional (SLACK) to fit them: 32 bytes of
// spills without padding and 40 with it, 300 and 440 with the test out of line and the load
// under its condition.  us per step with 128 (1024) replicas, fp32: N = 1024 0.99 (1.63), 1.00 (1.83) before,
// N = 1000 1.02 (1.63), 1.44 (2.59) before.
constexpr int kWsRing = 4;
constexpr uint32_t kWsWaitPolls = 1u << 26;
constexpr uint64_t kWsWaitNs = 2000000000ull;

template <typename Tw, int V, bool FULL, bool TRACE>
__global__ void __launch_bounds__(64, 7) step_kernel_ws(const __grid_constant__ StepParams p)
{
    using R_ = WarpReplica<Tw, V, false, false, false, V, V == 32, (V < 16), V == 32>;
    using H = typename R_::H;
    constexpr int NQ = V / 4;
    __shared__ float4 ring[kWsRing][NQ][32];
    __shared__ uint64_t full[kWsRing], empty[kWsRing];
    __shared__ int failed;
    __shared__ FlipLog<typename R_::E> log;
    const int r = blockIdx.x;
    if (r >= p.R) return;   // whole block
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int b = 0; b < kWsRing; ++b) {
            tc::mbar_init(&full[b], 32);
            tc::mbar_init(&empty[b], 32);
        }
        failed = (p.err ? *reinterpret_cast<volatile int*>(p.err) : 0) |
                 (p.stop ? *reinterpret_cast<const volatile int*>(p.stop) : 0);
    }
    __syncthreads();
    if (failed) return;     // whole block
    const PhiloxKeys& keys = *reinterpret_cast<const PhiloxKeys*>(&p.round_key[0][0]);
    const uint32_t rep = p.rep_base + (uint32_t)r;
    const long long n = p.t1 - p.t0;

    if (warp == 1) {   // producer: draws of steps t0 .. t1 - 1, in order
        const uint32_t q0 = (uint32_t)(lane * V) >> 2;
        for (long long i = 0; i < n; ++i) {
            const int b = (int)(i % kWsRing);
            const uint32_t ph = (uint32_t)(i / kWsRing);
            if (ph > 0 && !tc::mbar_wait(&empty[b], (ph - 1) & 1u, kWsWaitPolls, kWsWaitNs)) {
                if (p.err) atomicExch(p.err, 2);
                break;
            }
            const uint32_t tt = (uint32_t)(p.t0 + i);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const u32x4 w = philox4x32_10(q0 + q, tt, rep, 0u, keys);
                ring[b][q][lane] = make_float4(lg2_draw(w.x), lg2_draw(w.y), lg2_draw(w.z), lg2_draw(w.w));
            }
            tc::mbar_arrive(&full[b]);
        }
        return;
    }

    R_ rp;
    rp.init(static_cast<const Tw*>(p.W), p.N, p.ldw, rep, p.bestx + (size_t)r * p.nw, log.f, &log.head);
    H* hg = static_cast<H*>(p.h) + (size_t)r * p.npad + rp.base;
    uint32_t* xg = p.x + (size_t)r * p.nw;
    rp.load_fields(hg);
    rp.xm = (xg[rp.base >> 5] >> (rp.base & 31)) & R_::VMASK;
    ReplicaScalars sc = p.sc[r];
    rp.m = sc.m;
    const bool per_rep = p.betas != nullptr;
    rp.begin(p.t0, p.t1, per_rep ? nullptr : p.beta, per_rep ? p.betas[p.temp_of[r]] : 0.f, Arith<Tw>::load_e(sc.E),
             Arith<Tw>::load_e(sc.best), sc.flips, keys);
    bool held = sc.check != 0;       // the best-state test of the last step is still to be made
    if (held && p.t0 < p.t1) rp.test_current();

    float L[V];
    bool ok = true;
    auto fetch = [&](long long i) {   // the draws of step t0 + i, then release the buffer
        const int b = (int)(i % kWsRing);
        if (!tc::mbar_wait(&full[b], (uint32_t)(i / kWsRing) & 1u, kWsWaitPolls, kWsWaitNs)) {
            ok = false;
            return;
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 f = ring[b][q][lane];
            L[4 * q] = f.x; L[4 * q + 1] = f.y; L[4 * q + 2] = f.z; L[4 * q + 3] = f.w;
        }
        tc::mbar_arrive(&empty[b]);
    };
    if (n > 0) fetch(0);
    for (long long i = 0; i < n && __all_sync(0xffffffffu, ok); ++i) {
        const long long t = p.t0 + i;
        const int k = rp.template step_log<FULL>(t, p.inc, L, keys, [&] {
            if (i + 1 < n) fetch(i + 1);
        });
        held = k >= 0;
        if constexpr (TRACE) {
            if (lane == 0) p.trace[(size_t)r * p.trace_T + t] = k;
        }
    }
    if (!__all_sync(0xffffffffu, ok) && lane == 0 && p.err) atomicExch(p.err, 2);
    rp.store_fields(hg);
    const uint32_t word = rp.word();
    if (lane % R_::P == 0) xg[rp.base >> 5] = word;
    if (rp.n > 0) rp.settle(held);
    if (lane == 0) {
        sc.E = Arith<Tw>::store_e(rp.head->E);
        sc.best = Arith<Tw>::store_e(rp.head->best);
        sc.flips = rp.head->flips;
        sc.m = rp.m;
        sc.check = held ? 1u : 0u;
        p.sc[r] = sc;
    }
}

// One launch of kernel K with the on-chip memory split of prefer_shared; with
// no blocks (p.R = 0) only the attribute is set, which also loads the kernel.
template <auto K>
inline void launch_shared(int blocks, int threads, cudaStream_t st, const StepParams& p)
{
    prefer_shared<K>();
    if (blocks > 0) K<<<blocks, threads, 0, st>>>(p);
}

// One launch on clusters of C blocks per replica, G warps in each.
template <auto K>
inline cudaError_t launch_cluster(int C, int threads, cudaStream_t st, const StepParams& p)
{
    prefer_shared<K>();
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)p.R * C);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, K, p);
}

template <typename Tw, int V, int G, int C>
cudaError_t launch_on_clusters(const StepParams& p, bool trace, cudaStream_t st)
{
    if (p.N == 32 * V * G * C)
        return trace ? launch_cluster<step_kernel<Tw, V, G, true, true, C>>(C, 32 * G, st, p)
                     : launch_cluster<step_kernel<Tw, V, G, true, false, C>>(C, 32 * G, st, p);
    return trace ? launch_cluster<step_kernel<Tw, V, G, false, true, C>>(C, 32 * G, st, p)
                 : launch_cluster<step_kernel<Tw, V, G, false, false, C>>(C, 32 * G, st, p);
}

template <typename Tw, int V, int G>
cudaError_t launch_vg(const StepShape& s, const StepParams& p, bool trace, cudaStream_t st)
{
    const int threads = 32 * G * s.rpb;
    const int blocks = (p.R + s.rpb - 1) / s.rpb;
    const bool full = p.N == 32 * V * G;
    if constexpr (G == 1) {
        if (s.ws) {
            if (blocks == 0) return cudaSuccess;
            if (full) {
                if (trace) step_kernel_ws<Tw, V, true, true><<<p.R, 64, 0, st>>>(p);
                else step_kernel_ws<Tw, V, true, false><<<p.R, 64, 0, st>>>(p);
            } else {
                if (trace) step_kernel_ws<Tw, V, false, true><<<p.R, 64, 0, st>>>(p);
                else step_kernel_ws<Tw, V, false, false><<<p.R, 64, 0, st>>>(p);
            }
            return cudaGetLastError();
        }
        if (blocks > 0 && sizeof(Tw) == 4 && V >= 8 && p.Wc == nullptr) return cudaErrorInvalidValue;
        if (full) {
            if (trace) launch_shared<step_kernel_g1<Tw, V, true, true>>(blocks, threads, st, p);
            else launch_shared<step_kernel_g1<Tw, V, true, false>>(blocks, threads, st, p);
        } else {
            if (trace) launch_shared<step_kernel_g1<Tw, V, false, true>>(blocks, threads, st, p);
            else launch_shared<step_kernel_g1<Tw, V, false, false>>(blocks, threads, st, p);
        }
        return cudaGetLastError();
    } else {
        if (blocks > 0 && sizeof(Tw) == 4 && V >= 8 && p.Wc == nullptr) return cudaErrorInvalidValue;
        if constexpr (G == 8 && V >= 16) {
            if (s.cluster > 1) {                    // its blocks do not look at a stop flag
                if (p.R > 0 && p.stop) return cudaErrorInvalidValue;
                return p.R > 0 ? launch_on_clusters<Tw, V / 2, 4, 4>(p, trace, st) : cudaSuccess;
            }
        }
        if (full) {
            if (trace) launch_shared<step_kernel<Tw, V, G, true, true>>(blocks, threads, st, p);
            else launch_shared<step_kernel<Tw, V, G, true, false>>(blocks, threads, st, p);
        } else {
            if (trace) launch_shared<step_kernel<Tw, V, G, false, true>>(blocks, threads, st, p);
            else launch_shared<step_kernel<Tw, V, G, false, false>>(blocks, threads, st, p);
        }
        return cudaGetLastError();
    }
}

template <typename Tw>
cudaError_t launch_typed(const StepShape& s, const StepParams& p, bool trace, cudaStream_t st)
{
#define DA_CASE(VV, GG) \
    if (s.V == VV && s.G == GG) return launch_vg<Tw, VV, GG>(s, p, trace, st);
    DA_CASE(4, 1) DA_CASE(8, 1) DA_CASE(16, 1) DA_CASE(32, 1)
    DA_CASE(4, 2) DA_CASE(8, 2) DA_CASE(16, 2) DA_CASE(32, 2)
    DA_CASE(4, 4) DA_CASE(8, 4) DA_CASE(16, 4) DA_CASE(32, 4)
    DA_CASE(8, 8) DA_CASE(16, 8) DA_CASE(32, 8)
#undef DA_CASE
    return cudaErrorInvalidConfiguration;
}

}  // namespace step_detail
}  // namespace da
