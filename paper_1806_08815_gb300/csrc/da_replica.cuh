// da_replica.cuh -- one replica annealed by one warp (the G = 1 form of the
// step in da_step.cuh), packaged so that the chunked step kernel and the
// persistent batched kernel share it.
//
// What bounds a step is the latency of its dependent chain: 809 cycles for 217
// instructions of one warp at N = 64, 1865 for 701 at N = 1024 (2 warps per scheduler
// at 1024 replicas: 2600).  So the chain holds as few long-latency operations as
// possible: the count of accepted trials and the position of the chosen one come from
// votes instead of chains of shuffles, the inputs of the next step (draws, choice word,
// beta) are made in the shadow of this one, and the fp64 energy and the best state are
// settled 32 flips at a time (FlipLog).  us per step before and after, 64 replicas
// (1024): fp32 N = 64 0.555 -> 0.33 (0.613 -> 0.395), N = 256 0.670 -> 0.426
// (0.761 -> 0.516), N = 512 0.781 -> 0.56 (0.918 -> 0.717), N = 1024 0.961 -> 0.89
// (1.327 -> 1.182).  With two warps per scheduler (the last) the pipes bind as much as
// the chain: a 32 x 32 -> 64 bit product holds the integer multiplier for 4 cycles, and
// 120 of them with the other multiplications are 1400 of the 2550 cycles.
//
// Lane l owns the V consecutive variables i = l*V + v of the replica and keeps
// their effective fields g_i, bits x_i and the Philox words of the current step
// in registers.  step() performs one step of Algorithm 2 (see da_step.cuh for
// the decomposition); recompute() replaces the fp32 fields and the tracked
// energy by their exact fixed-point values (the same definition as the tiled
// recompute in da_fields.cu, evaluated by the warp itself).
#pragma once
#include <type_traits>

#include "da_device.cuh"
#include "da_fixed.cuh"
#include "da_internal.h"
#include "da_step_common.cuh"

namespace da {
namespace step_detail {

// SW: the rows of W are read from a copy staged in shared memory (W points
// there) instead of from global memory.
// PRE: the step-invariant part of each Philox block is computed once per launch
// (prep_draws) and the draws of every step start from it (draw_pre); four more
// words per block live in registers, for kernels that have them to spare.
// COAL: W points at the couplings in the warp row order (row pitch ldw, slices of 32 V0
// entries; step_uses_coal in da_internal.h) and rows are read with RowCoal.
// WIDE: the form of a step whose instructions count for more than its latency, for one warp
// per replica at V = 32 and, without padding, at V = 16, where the default shapes put one to
// two warps on a scheduler: counts by shuffles, packed field updates, most of the draws'
// rounds before the choice, the rare parts out of line.  At V = 16 against the other form:
// N = 512 with 1024 replicas 0.755 -> 0.717 us per step (int8 0.738 -> 0.714, PTDA 0.774 ->
// 0.737), with 512 0.586 -> 0.564; with padding it is slower (N = 500 with 512 replicas 0.607 ->
// 0.626), and so it is at V = 8 (N = 256 with 1024 replicas 0.516 -> 0.554).
// RARE_OUT: the rare parts of a step (exact test, choice draws' refill) out of line.
// SLACK: lanes wholly beyond N load their part of a row too, and leave it: a load under a
// condition stays before the code that follows it, its registers live throughout, where an
// unconditional one moves down to its use.  W in the plain order has the room for it
// (instance_W_bytes).
template <typename Tw, int V, bool SW = false, bool PRE = false, bool COAL = false, int V0 = V, bool WIDE = V == 32,
          bool RARE_OUT = V != 16 || WIDE, bool SLACK = false>
struct WarpReplica {
    using A = Arith<Tw>;
    using H = typename A::H;
    using E = typename A::E;
    static_assert(V % 4 == 0 && V <= 32, "V must be 4, 8, 16 or 32");
    static constexpr int NQ = V / 4;
    static constexpr uint32_t VMASK = V == 32 ? 0xffffffffu : ((1u << V) - 1u);
    static constexpr int P = 32 / V;

    H h[V];
    float lg[V];      // log2 U of this lane's draws for the current step (lg2_draw)
    u32x4 cr;         // choice words of the steps [t & ~127, + 128): lane l holds those of 4 l .. 4 l + 3
    uint32_t cw;      // the choice word of the current step
    float bwin, bnext;   // the schedule of the steps [t & ~31, + 32) and of the 32 after, one per lane
    float beta;       // of the current step
    uint32_t xm, valid, m;
    FlipEntry* log;   // the replica's flip log and this warp's energies, in shared memory
    FlipHead<E>* head;
    int n;            // flips in the log
    int lane, base, N, ldw;
    int rowoff;       // this lane's first entry in a row of W
    uint32_t rep;
    const Tw* __restrict__ W;
    uint32_t* bestg;  // best-state words of this replica
    // Step-invariant Philox words of the lane's blocks (prep_draws): kq1..kq4 per
    // block, ku0 shared by the lane's blocks.
    uint32_t kq1[PRE ? NQ : 1], kq2[PRE ? NQ : 1], kq3[PRE ? NQ : 1], kq4[PRE ? NQ : 1];
    uint32_t ku0;

    __device__ __forceinline__ void init(const Tw* W_, int N_, int ldw_, uint32_t rep_, uint32_t* bestg_,
                                         FlipEntry* log_, FlipHead<E>* head_, int slice = 0)
    {
        lane = threadIdx.x & 31;
        base = slice + lane * V;
        rowoff = COAL ? base / (32 * V0) * (32 * V0) + base % V0 * 32 + base % (32 * V0) / V0 * 4 : base;
        N = N_;
        ldw = ldw_;
        rep = rep_;
        W = W_;
        bestg = bestg_;
        valid = base >= N ? 0u : (N - base >= V ? VMASK : ((1u << (N - base)) - 1u));
        log = log_;
        head = head_;
    }

    // Before the first step t0 of a launch over [t0, t1): the energies, and the step
    // inputs that depend on nothing in a step (next_inputs).  sched: the schedule, or
    // null for a fixed beta0.
    const float* __restrict__ sched;
    long long t_end;
    template <class Keys>
    __device__ __forceinline__ void begin(long long t0, long long t1, const float* sched_, float beta0, E e0, E best0,
                                          long long flips0, const Keys& keys)
    {
        if (lane == 0) *head = FlipHead<E>{e0, best0, flips0};
        __syncwarp();
        n = 0;
        sched = sched_;
        t_end = t1;
        bwin = bnext = beta = beta0;
        if (sched && t0 < t1) {
            bwin = sched_window(t0 & ~31ll);
            bnext = sched_window((t0 & ~31ll) + 32);
            beta = __shfl_sync(0xffffffffu, bwin, (int)t0 & 31);
        }
        fill_choice(t0, keys);
        cw = choice_word(t0);
    }
    __device__ __forceinline__ float sched_window(long long tb) const
    {
        const long long t = tb + lane;
        return ldx(sched + (t < t_end ? t : t_end - 1));
    }

    // The uniform-choice draws (block (0, t & ~3, rep, 1), lane t % 4): each lane
    // computes one block, so that one Philox evaluation serves 128 steps and a
    // step's word comes by a shuffle that depends on nothing in the step; likewise
    // beta from a window of the schedule.  Both are fetched one step ahead, under
    // the row load: a load of beta every step had cost 0.06 of 0.51 us per step at
    // N = 64.
    template <class Keys>
    __device__ __forceinline__ void fill_choice(long long t, const Keys& keys)
    {
        const uint32_t c = (uint32_t)((t & ~127ll) + 4 * lane);
        if constexpr (RARE_OUT) cr = choice_block(c, rep, keys);
        else cr = philox4x32_10(0u, c, rep, 1u, keys);
    }
    template <class Keys>
    static __device__ __noinline__ u32x4 choice_block(uint32_t c, uint32_t rep, const Keys& keys)
    {
        return philox4x32_10(0u, c, rep, 1u, keys);
    }
    __device__ __forceinline__ uint32_t choice_word(uint32_t t) const
    {
        return __shfl_sync(0xffffffffu, pick(cr, (int)(t & 3)), (int)(t >> 2) & 31);
    }
    template <class Keys>
    __device__ __forceinline__ void next_inputs(uint32_t t, const Keys& keys)   // of step t + 1
    {
        const uint32_t t1 = t + 1;
        if ((t1 & 31) == 0) {
            if (sched) {
                bwin = bnext;
                bnext = sched_window((long long)t1 + 32);
            }
            if ((t1 & 127) == 0) fill_choice(t1, keys);
        }
        beta = __shfl_sync(0xffffffffu, bwin, (int)(t1 & 31));
        cw = choice_word(t1);
    }

    // The flips logged so far into the tracked energy, and the test of Algorithm 2's
    // result after each: a strictly lower energy than any seen makes that state the
    // best one.  hold_last: the test of the last flip is left to the caller (a
    // recompute follows it, and the test comes after the recompute).
    __device__ __forceinline__ void settle(bool hold_last = false)
    {
        settle_impl(head, log, n, hold_last, xm, lane, base, bestg);
        n = 0;
    }
    // Once per 32 flips: out of line, so that the step's code stays short (the
    // instruction fetch of a one-warp step is part of its latency: N = 512 fp32, 64
    // replicas 0.604 us per step inlined, 0.586 not).
    static __device__ __noinline__ void settle_impl(FlipHead<E>* head, const FlipEntry* log, int n, bool hold_last,
                                                    uint32_t xm, int lane, int base, uint32_t* bestg)
    {
        __syncwarp();
        E e = head->E, b = head->best;
        const int at = settle_log<A>(log, n, hold_last ? n - 1 : n, lane, e, b);
        if (at >= 0) {                        // the state after flip `at`: the later ones undone
            uint32_t x = xm;
            for (int q = at + 1; q < n; ++q) {
                const int k = log[q].k - base;
                if (k >= 0 && k < V) x ^= 1u << k;
            }
            const uint32_t wv = gather_word<V>(x, lane);
            if (lane % P == 0) bestg[base >> 5] = wv;
        }
        __syncwarp();
        if (lane == 0) *head = FlipHead<E>{e, b, head->flips + n};
        __syncwarp();
    }

    // The best-state test of the current state (no flips pending) at the energy head->E.
    __device__ __forceinline__ void test_current()
    {
        __syncwarp();
        if (head->E < head->best) {             // uniform
            const uint32_t wv = word();
            if (lane % P == 0) bestg[base >> 5] = wv;
            __syncwarp();
            if (lane == 0) head->best = head->E;
        }
        __syncwarp();
    }

    __device__ __forceinline__ uint32_t word() const { return gather_word<V>(xm, lane); }

    // The lane's V fields between launches (16-byte aligned).  From V = 16 on, where the
    // lanes' slices are 64 bytes or more apart, as 16-byte accesses: 4-byte ones touch up to
    // 32 lines each (5 us of a launch of 1024 replicas at N = 1024).
    __device__ __forceinline__ void load_fields(const H* p)
    {
        static_assert(sizeof(H) == 4, "fields are 4 bytes");
        if constexpr (V < 16) {
#pragma unroll
            for (int v = 0; v < V; ++v) h[v] = p[v];
        } else {
#pragma unroll
            for (int v = 0; v < V; v += 4) {
                const uint4 f = *reinterpret_cast<const uint4*>(p + v);
                h[v] = of_bits(f.x);
                h[v + 1] = of_bits(f.y);
                h[v + 2] = of_bits(f.z);
                h[v + 3] = of_bits(f.w);
            }
        }
    }
    __device__ __forceinline__ void store_fields(H* p) const
    {
        if constexpr (V < 16) {
#pragma unroll
            for (int v = 0; v < V; ++v) p[v] = h[v];
        } else {
#pragma unroll
            for (int v = 0; v < V; v += 4)
                *reinterpret_cast<uint4*>(p + v) =
                    make_uint4(A::log_bits(h[v]), A::log_bits(h[v + 1]), A::log_bits(h[v + 2]), A::log_bits(h[v + 3]));
        }
    }
    static __device__ __forceinline__ H of_bits(uint32_t b)
    {
        if constexpr (std::is_same<H, float>::value) return __uint_as_float(b);
        else return (H)b;
    }

    static __device__ __forceinline__ void load_row(const Tw* p, Tw (&c)[V])
    {
        static_assert(!(SW && COAL), "a staged W is in the plain order");
        if constexpr (SW) RowShared<Tw, V>::load(p, c);
        else if constexpr (COAL) RowCoal<Tw, V>::load(p, c);
        else Row<Tw, V>::load(p, c);
    }

    template <class Keys>
    __device__ __forceinline__ void draw(uint32_t tt, const Keys& keys)
    {
        // the NQ Philox4x32-10 blocks round by round, so that their independent
        // multiply-xor chains interleave
        uint32_t c0[NQ], c1[NQ], c2[NQ], c3[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) { c0[q] = (uint32_t)(base >> 2) + q; c1[q] = tt; c2[q] = rep; c3[q] = 0u; }
#pragma unroll
        for (int round = 0; round < 10; ++round) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const uint64_t pa = (uint64_t)kPhiloxMulA * c0[q];
                const uint64_t pb = (uint64_t)kPhiloxMulB * c2[q];
                const uint32_t n0 = (uint32_t)(pb >> 32) ^ c1[q] ^ keys.a[round];
                const uint32_t n2 = (uint32_t)(pa >> 32) ^ c3[q] ^ keys.b[round];
                c1[q] = (uint32_t)pb;
                c3[q] = (uint32_t)pa;
                c0[q] = n0;
                c2[q] = n2;
            }
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            lg[4 * q] = lg2_draw(c0[q]);
            lg[4 * q + 1] = lg2_draw(c1[q]);
            lg[4 * q + 2] = lg2_draw(c2[q]);
            lg[4 * q + 3] = lg2_draw(c3[q]);
        }
    }

    // The acceptance block q of step t has counter (c0, t, rep, 0), c0 = base/4 + q.
    // Following the words of Philox4x32-10 through its first rounds (round r:
    // products pa = A c0, pb = B c2; c0 <- hi(pb) ^ c1 ^ ka_r, c1 <- lo(pb),
    // c2 <- hi(pa) ^ c3 ^ kb_r, c3 <- lo(pa)):
    //   after round 0: (u ^ t, lo(B rep), y2_q, y3_q) with u = hi(B rep) ^ ka_0,
    //     y2_q = hi(A c0) ^ kb_0, y3_q = lo(A c0): only the first word depends on t;
    //   round 1 multiplies that word (one product per lane and step, P = A (u ^ t))
    //     and y2_q (step-invariant): after it (z0_q, z1_q, hi(P) ^ y3_q ^ kb_1, lo(P))
    //     with z0_q, z1_q step-invariant;
    //   round 2 multiplies z0_q (step-invariant) and the third word (per block).
    // So a step needs one product for the lane and, per block, one product in round
    // 2 and the full rounds 3..9: the words below are the step-invariant operands
    // with their round keys folded in.  draw_pre returns philox4x32_10's words bit
    // for bit.
    template <class Keys>
    __device__ __forceinline__ void prep_draws(const Keys& keys)
    {
        static_assert(PRE, "prep_draws needs PRE");
        const uint64_t pb0 = (uint64_t)kPhiloxMulB * rep;
        ku0 = (uint32_t)(pb0 >> 32) ^ keys.a[0];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const uint64_t pa0 = (uint64_t)kPhiloxMulA * ((uint32_t)(base >> 2) + q);
            const uint64_t pb1 = (uint64_t)kPhiloxMulB * ((uint32_t)(pa0 >> 32) ^ keys.b[0]);
            const uint64_t pa2 = (uint64_t)kPhiloxMulA * ((uint32_t)(pb1 >> 32) ^ (uint32_t)pb0 ^ keys.a[1]);
            kq1[q] = (uint32_t)pa0 ^ keys.b[1];               // y3_q ^ kb_1
            kq2[q] = (uint32_t)pb1 ^ keys.a[2];               // z1_q ^ ka_2
            kq3[q] = (uint32_t)(pa2 >> 32) ^ keys.b[2];       // hi(A z0_q) ^ kb_2
            kq4[q] = (uint32_t)pa2 ^ keys.b[3];               // lo(A z0_q) ^ kb_3
        }
    }

    // The next step's draws in stages (PRE), so that their rounds can fill the
    // latency of the current step's warp collectives: draw_begin (the per-step
    // product and round 2), draw_round<R> (rounds 3..9), draw_end (log2 U of the
    // 4 NQ words into lg).
    uint32_t dq0[PRE ? NQ : 1], dq1[PRE ? NQ : 1], dq2[PRE ? NQ : 1], dq3[PRE ? NQ : 1];

    __device__ __forceinline__ void draw_begin(uint32_t tt)
    {
        const uint64_t P = (uint64_t)kPhiloxMulA * (ku0 ^ tt);
        const uint32_t hP = (uint32_t)(P >> 32), lP = (uint32_t)P;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {            // round 2
            const uint64_t pb = (uint64_t)kPhiloxMulB * (hP ^ kq1[q]);
            dq0[q] = (uint32_t)(pb >> 32) ^ kq2[q];
            dq1[q] = (uint32_t)pb;
            dq2[q] = kq3[q] ^ lP;
            dq3[q] = kq4[q];                       // carries kb_3
        }
    }

    template <int R, class Keys>
    __device__ __forceinline__ void draw_round(const Keys& keys)
    {
        static_assert(R >= 3 && R < 10, "rounds 3..9");
        const uint32_t ka = keys.a[R], kb = R == 3 ? 0u : keys.b[R];   // dq3 of round 2 carries kb_3
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const uint64_t pa = (uint64_t)kPhiloxMulA * dq0[q];
            const uint64_t pb = (uint64_t)kPhiloxMulB * dq2[q];
            dq0[q] = (uint32_t)(pb >> 32) ^ dq1[q] ^ ka;
            dq2[q] = (uint32_t)(pa >> 32) ^ dq3[q] ^ kb;
            dq1[q] = (uint32_t)pb;
            dq3[q] = (uint32_t)pa;
        }
    }

    template <int R0, int R1, class Keys>
    __device__ __forceinline__ void draw_rounds(const Keys& keys)
    {
        if constexpr (R0 < R1) {
            draw_round<R0>(keys);
            draw_rounds<R0 + 1, R1>(keys);
        }
    }

    __device__ __forceinline__ void draw_end()
    {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            lg[4 * q] = lg2_draw(dq0[q]);
            lg[4 * q + 1] = lg2_draw(dq1[q]);
            lg[4 * q + 2] = lg2_draw(dq2[q]);
            lg[4 * q + 3] = lg2_draw(dq3[q]);
        }
    }

    template <class Keys>
    __device__ __forceinline__ void draw_pre(uint32_t tt, const Keys& keys)
    {
        draw_begin(tt);
        draw_rounds<3, 10>(keys);
        draw_end();
    }

    // Work a step places in the latency of its warp collectives (choose_and_flip):
    // at<0>() after the votes on the counts are issued, at<1>() after the owner's
    // vote, at<2>() after the shuffles of the owner's words, at<3>() after the vote
    // on the bit position; rest_flip() while row k is in flight, rest_none() when
    // nothing flips.
    template <class F>
    struct RestOnly {      // everything under the row load (or at once)
        F& f;
        template <int I> __device__ __forceinline__ void at() {}
        __device__ __forceinline__ void rest_flip() { f(); }
        __device__ __forceinline__ void rest_none() { f(); }
    };
    template <class Keys, int kR0 = WIDE ? 7 : 5, int kR1 = WIDE ? 8 : 6, int kR2 = WIDE ? 8 : 7,
              int kR3 = WIDE ? 9 : 8>
    struct DrawSlots {     // the next step's draws (PRE)
        WarpReplica& rp;
        const Keys& keys;
        uint32_t tt;
        // Rounds done after slot 0 .. 3, measured per form: all of them under the row load
        // (3, 3, 3, 3) take N = 512 with 1024 replicas from 0.755 to 0.803 us per step, all of
        // them before it (10, 10, 10, 10) N = 256 from 0.516 to 0.543; in the wide form most
        // belong before the choice (5, 6, 7, 7: 1.25 instead of 1.23 us at N = 1024 with 1024
        // replicas).
        template <int I>
        __device__ __forceinline__ void at()
        {
            if constexpr (I == 0) {
                rp.draw_begin(tt);
                rp.template draw_rounds<3, kR0>(keys);
            } else if constexpr (I == 1) rp.template draw_rounds<kR0, kR1>(keys);
            else if constexpr (I == 2) rp.template draw_rounds<kR1, kR2>(keys);
            else rp.template draw_rounds<kR2, kR3>(keys);
        }
        __device__ __forceinline__ void rest_flip()
        {
            rp.template draw_rounds<kR3, 10>(keys);
            rp.draw_end();
        }
        __device__ __forceinline__ void rest_none()
        {
            rp.template draw_rounds<kR0, 10>(keys);
            rp.draw_end();
        }
    };

    // One step t (the draws of t are in lg).  If draw_next, the draws of t + 1
    // are computed while row k is in flight (PRE: always, spread over the
    // step's collectives as DrawSlots places them).  Returns the flipped index
    // or -1.
    template <bool FULL, class Keys>
    __device__ __forceinline__ int step(uint32_t t, bool draw_next, float inc, const Keys& keys)
    {
        if constexpr (PRE) {
            DrawSlots<Keys> s{*this, keys, (uint32_t)(t + 1)};
            return decide_and_flip<FULL>(t, inc, lg, keys, s);
        } else {
            auto f = [&] {
                if (draw_next) draw((uint32_t)(t + 1), keys);
            };
            RestOnly<decltype(f)> s{f};
            return decide_and_flip<FULL>(t, inc, lg, keys, s);
        }
    }

    // One step t whose acceptance draws are L[v] = log2 U of this lane's trials
    // (lg2_draw; from draw() or from a producer warp), decided in the log domain
    // (decide_log; the rare trials near the threshold by decide_exact).
    // `overlap` runs while row k is in flight.
    template <bool FULL, class Keys, class Overlap>
    __device__ __forceinline__ int step_log(long long t, float inc, const float (&L)[V], const Keys& keys,
                                            Overlap&& overlap)
    {
        RestOnly<Overlap> s{overlap};
        return decide_and_flip<FULL>(t, inc, L, keys, s);
    }

    template <bool FULL, class Keys, class Slots>
    __device__ __forceinline__ int decide_and_flip(uint32_t t, float inc, const float (&L)[V], const Keys& keys,
                                                   Slots& slots)
    {
        // here the draws' and the row's registers are free
        if (n == 32) settle();
        const float Eoff = __fmul_rn(__uint2float_rn(m), inc);
        bool unsure;
        uint32_t accm = decide_log<A, V>(h, xm, Eoff, __fmul_rn(beta, kLog2e), L, unsure);
        const bool any_unsure = __any_sync(0xffffffffu, unsure);
        // the rare exact test before the count: a first count beside the vote on the band and a
        // second one after the test hide one latency, but their code costs more (N = 64 int8
        // 0.341 -> 0.321 us per step without them, fp32 with 1024 replicas 0.411 -> 0.395;
        // N = 256 with 2048 replicas, by its registers, 1.013 -> 0.864), except at V = 16 where
        // the test is inline (N = 500 int8 with 1024 replicas 0.791, 0.813 before the count) and
        // for integer rows at V = 8 (allocation-free, N = 200 0.429, 0.434 before it)
        constexpr bool kFirst = RARE_OUT && !(V == 8 && sizeof(Tw) < 4);
        if (kFirst && any_unsure)
            accm = decide_exact_out<A, V, RARE_OUT>(h, xm, Eoff, beta, L, accm, base, (uint32_t)t, rep, keys);
        if constexpr (!FULL) accm &= valid;
        int excl, total;
        count_below(accm, excl, total);
        slots.template at<0>();
        if (!kFirst && any_unsure) {
            accm = decide_exact_out<A, V, RARE_OUT>(h, xm, Eoff, beta, L, accm, base, (uint32_t)t, rep, keys);
            if constexpr (!FULL) accm &= valid;
            count_below(accm, excl, total);
        }
        return choose_and_flip<FULL>(t, accm, excl, total, keys, slots);
    }

    // Accepted trials on the lanes below this one, and on all lanes: the bits of the
    // lanes' counts as votes, which are independent of one another (one latency of
    // about 20 cycles, then the population counts), beside the warp reduction of the
    // total; a five-shuffle prefix sum is a chain of five 32-cycle latencies.  In the wide
    // form the shuffles are used all the same: a population count takes 8 cycles of the
    // unit that also makes the log2 of the draws (8 cycles each), and with two warps per
    // scheduler that counts for more than the chain (1.25 against 1.29 us per step at
    // N = 1024 with 1024 replicas).
    __device__ __forceinline__ void count_below(uint32_t accm, int& excl, int& total) const
    {
        const int cnt = __popc(accm);
        total = (int)__reduce_add_sync(0xffffffffu, (unsigned)cnt);
        if constexpr (WIDE) {
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            excl = incl - cnt;
        } else {
            constexpr int kBits = V == 4 ? 3 : V == 8 ? 4 : 5;   // of a count 0 .. V
            const uint32_t below = (1u << lane) - 1u;
            excl = 0;
#pragma unroll
            for (int b = 0; b < kBits; ++b) excl += __popc(__ballot_sync(0xffffffffu, (cnt >> b) & 1) & below) << b;
        }
    }

    // (c) of a step with acceptance mask accm (excl accepted trials on lower lanes,
    // total in all): the uniform choice among the accepted trials, the flip and the
    // field update, with `slots` placed as described above.  Returns the flipped index
    // or -1.
    template <bool FULL, class Keys, class Slots>
    __device__ __forceinline__ int choose_and_flip(uint32_t t, uint32_t accm, int excl, int total, const Keys& keys,
                                                   Slots& slots)
    {
        if (total == 0) {
            m += 1;
            slots.rest_none();
            next_inputs(t, keys);
            return -1;
        }
        const int j = (int)__umulhi(cw, (uint32_t)total);
        // inclusive counts ascend, so the lanes with at most j accepted trials up to
        // and including their own are those before the owner
        const uint32_t before = __ballot_sync(0xffffffffu, excl + __popc(accm) <= j);
        slots.template at<1>();
        const int own = __popc(before);
        uint32_t acc_o, x_o;
        int r;
        if constexpr (V <= 8) {
            const uint32_t w = __shfl_sync(0xffffffffu, accm | xm << 8 | (uint32_t)excl << 16, own);
            acc_o = w & 0xFFu;
            x_o = (w >> 8) & 0xFFu;
            r = j - (int)(w >> 16);
        } else {
            acc_o = __shfl_sync(0xffffffffu, accm, own);
            x_o = __shfl_sync(0xffffffffu, xm, own);
            r = j - __shfl_sync(0xffffffffu, excl, own);
        }
        slots.template at<2>();
        const uint32_t pre = bits_before(acc_o, r, lane);
        slots.template at<3>();
        const int vk = __popc(pre);
        const uint32_t xold = (x_o >> vk) & 1u;
        const H gk = select_slot<H, V>(h, vk);
        const int k = own * V + vk;
        Tw cv[V];
        if (FULL || SLACK || base < N) load_row(W + (size_t)k * ldw + rowoff, cv);
        if (lane == own) log[n] = FlipEntry{A::log_bits(A::signed_field(gk, xold)), k};
        ++n;
        slots.rest_flip();
        next_inputs(t, keys);
        if (FULL || base < N) {
            const typename A::Sign sg = A::sign(xold);
#pragma unroll
            for (int v = 0; v < V; v += 2) {
                // packed: the same roundings, half the instructions; V = 8 only with padding
                // (N = 200 0.440 -> 0.420 us per step, but N = 256 0.517 -> 0.521)
                if constexpr (sizeof(Tw) == 4 && (WIDE || (V == 8 && !FULL))) {
                    const float* w = reinterpret_cast<const float*>(&cv[v]);
                    const float2 u = __ffma2_rn(make_float2(sg, sg), make_float2(w[0], w[1]), make_float2(h[v], h[v + 1]));
                    h[v] = u.x;
                    h[v + 1] = u.y;
                } else {
                    h[v] = A::apply_signed(h[v], cv[v], sg);
                    h[v + 1] = A::apply_signed(h[v + 1], cv[v + 1], sg);
                }
            }
        }
        if (lane == own) xm ^= 1u << vk;
        m = 0;
        return k;
    }

    // Exact fixed-point recompute of the fp32 fields and of the tracked
    // energy (no flips pending; same definition as da_fields.cu): g_i = fl32(2^-S (round(d_i 2^S)
    // + sum_{x_j = 1} round(W_ij 2^S))), E = fl64(2^-(S+1) sum_{x_i = 1}
    // (round(d_i 2^S) + sum_i)).
    // The fields of padding variables (beyond N) are set to 0, their value at the
    // start of an anneal, so that no old field stays live across the row loop.
    //
    // Each coupling is split into three integers of at most 22 bits and summed in
    // 32-bit accumulators: adding 1.5 2^23 to w 2^(S-40) leaves round(w 2^(S-40)) in
    // the low mantissa bits (Sum3), the remainder is exact, and so on for 2^(S-20) and
    // 2^S, where the last rounding is the definition's (ties to even: the parts above
    // are multiples of 2^20).  |w| < 2^e with S = 62 - L - e and 2^L > N, so the first
    // part is at most 2^(22-L) and N of them at most 2^22; the others are at most 2^19
    // and N <= 1024 of them at most 2^29.  4 packed fp32 operations per entry and part
    // instead of shifts, negations and carries in 64-bit integers, and the next row is
    // loaded while one is added.  (Scales whose factors leave the fp32 range take the
    // 64-bit form.)  With it the batched fp32 V = 32 class takes 1.39 instead of
    // 1.63 ms per 1024 steps of 512 replicas, 3.65 instead of 4.8 for 2432 (1.34 and 3.39
    // without any recompute).
    __device__ __forceinline__ void recompute(const float* __restrict__ diag, int S)
    {
        static_assert(sizeof(Tw) == 4, "only the fp32 fields are recomputed");
        long long acc[V];
        if (S >= -60 && S <= 100) sum_rows_split(S, acc);
        else sum_rows_wide(S, acc);
#pragma unroll
        for (int v = 0; v < V; ++v)
            acc[v] += ((valid >> v) & 1u) ? fixed_of_f32(ldx(diag + base + v), S) : 0ll;
        // energy: sum over x_i = 1 of (round(d_i 2^S) + acc_i), exact in 128 bits
        unsigned long long lo = 0;
        long long hi = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (((valid & xm) >> v) & 1u) {
                const long long t = fixed_of_f32(ldx(diag + base + v), S) + acc[v];
                const unsigned long long nlo = lo + (unsigned long long)t;
                hi += (t < 0 ? -1ll : 0ll) + (nlo < lo ? 1ll : 0ll);
                lo = nlo;
            }
            h[v] = ((valid >> v) & 1u) ? scaled_f32_of(acc[v], S) : H(0);   // padding: 0, so h is dead above
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long olo = __shfl_xor_sync(0xffffffffu, lo, o);
            const long long ohi = __shfl_xor_sync(0xffffffffu, hi, o);
            const unsigned long long nlo = lo + olo;
            hi = hi + ohi + (nlo < lo ? 1ll : 0ll);
            lo = nlo;
        }
        if (lane == 0) head->E = __longlong_as_double(energy_of_sum<false>(lo, hi, S));
        __syncwarp();
    }

    // The variables with x_j = 1 in ascending order, -1 after the last (warp-uniform).
    struct SetBits {
        uint32_t mine, w;
        int wi, nw;
        __device__ __forceinline__ int next()
        {
            while (w == 0) {
                if (++wi >= nw) return -1;
                w = __shfl_sync(0xffffffffu, mine, wi * P);
            }
            const int b = __ffs(w) - 1;
            w &= w - 1;
            return wi * 32 + b;
        }
    };

    // Slots v0 .. v0 + C - 1 of this lane in row j.
    template <int C>
    __device__ __forceinline__ void load_couplings(int j, int v0, float (&c)[C]) const
    {
        if (base < N) {
            const float* p = reinterpret_cast<const float*>(W) + (size_t)j * ldw + rowoff;
#pragma unroll
            for (int q = 0; q < C / 4; ++q) {
                const float* at = p + (COAL ? 32 * v0 + 128 * q : v0 + 4 * q);
                float4 f;
                if constexpr (SW) f = *reinterpret_cast<const float4*>(at);
                else f = ldx(reinterpret_cast<const float4*>(at));
                c[4 * q] = f.x; c[4 * q + 1] = f.y; c[4 * q + 2] = f.z; c[4 * q + 3] = f.w;
            }
        } else {
#pragma unroll
            for (int v = 0; v < C; ++v) c[v] = 0.f;
        }
    }

    // acc[v] = sum over x_j = 1 of round(W_ij 2^S), C slots at a time: their three
    // accumulators and two rows (the one being added and the next) fit the registers of
    // the step.
    static constexpr int kChunk = V < 16 ? V : 16;
    __device__ __forceinline__ void sum_rows_split(int S, long long (&acc)[V]) const
    {
#pragma unroll
        for (int v0 = 0; v0 < V; v0 += kChunk) sum_chunk(S, v0, acc);
    }

    __device__ __forceinline__ void sum_chunk(int S, int v0, long long (&acc)[V]) const
    {
        constexpr int C = kChunk;
        constexpr float kMagic = 12582912.0f;       // 1.5 2^23, bits 0x4B400000
        const float2 mg = make_float2(kMagic, kMagic), nm = make_float2(-kMagic, -kMagic);
        auto pow2 = [](int x, float sign) {
            const float f = sign * __int_as_float((x + 127) << 23);
            return make_float2(f, f);
        };
        const float2 up0 = pow2(S - 40, 1.f), up1 = pow2(S - 20, 1.f), up2 = pow2(S, 1.f);
        const float2 dn0 = pow2(40 - S, -1.f), dn1 = pow2(20 - S, -1.f);
        uint32_t p0[C], p1[C], p2[C];
#pragma unroll
        for (int v = 0; v < C; ++v) p0[v] = p1[v] = p2[v] = 0;
        uint32_t rows = 0;
        auto add = [&](const float (&c)[C]) {
            ++rows;
#pragma unroll
            for (int v = 0; v < C; v += 2) {
                float2 w = make_float2(c[v], c[v + 1]);
                float2 t = __ffma2_rn(w, up0, mg);
                p0[v] += __float_as_uint(t.x);
                p0[v + 1] += __float_as_uint(t.y);
                w = __ffma2_rn(__fadd2_rn(t, nm), dn0, w);
                t = __ffma2_rn(w, up1, mg);
                p1[v] += __float_as_uint(t.x);
                p1[v + 1] += __float_as_uint(t.y);
                w = __ffma2_rn(__fadd2_rn(t, nm), dn1, w);
                t = __ffma2_rn(w, up2, mg);
                p2[v] += __float_as_uint(t.x);
                p2[v + 1] += __float_as_uint(t.y);
            }
        };
        SetBits bits{word(), 0u, -1, (N + 31) >> 5};
        float a[C], b[C];
        int j = bits.next();
        if (j >= 0) load_couplings(j, v0, a);
        while (j >= 0) {
            j = bits.next();
            if (j >= 0) load_couplings(j, v0, b);
            add(a);
            if (j < 0) break;
            j = bits.next();
            if (j >= 0) load_couplings(j, v0, a);
            add(b);
        }
        const uint32_t bias = rows * 0x4B400000u;   // of the magic's own bits, modulo 2^32
#pragma unroll
        for (int v = 0; v < C; ++v)
            acc[v0 + v] = ((long long)(int)(p0[v] - bias) << 40) + ((long long)(int)(p1[v] - bias) << 20) +
                          (long long)(int)(p2[v] - bias);
    }

    __device__ __forceinline__ void sum_rows_wide(int S, long long (&acc)[V]) const
    {
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = 0;
        SetBits bits{word(), 0u, -1, (N + 31) >> 5};
        for (int j = bits.next(); j >= 0; j = bits.next()) {
            float c[V];
            load_couplings(j, 0, c);
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] += fixed_of_f32(c[v], S);
        }
    }
};

}  // namespace step_detail
}  // namespace da
