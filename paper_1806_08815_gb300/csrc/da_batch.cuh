// da_batch.cuh -- the persistent kernels of a batched launch (da_batch.cu): one work unit's
// anneal by one warp, rows of W from global memory or from a copy staged in shared memory.
// Instantiated without traces in da_batch.cu and with them in da_batch_traced.cu: in one
// translation unit the two make a module whose first load takes 12 ms longer (the first
// server or batched launch of a process 60 instead of 48 ms).
#pragma once
#include <algorithm>
#include <type_traits>

#include "da.h"
#include "da_internal.h"
#include "da_replica.cuh"

namespace da {

struct BatchClassParams {
    const BatchItemDev* items;
    int n_items;
    long long total_units;
    unsigned long long* head;   // work counter
    long long t_limit;          // > 0: run only this many steps per unit (autotuner probes)
    const int2* groups;         // shared-memory staging: (item, first replica) of each group
    long long n_groups;
    int pitch;                  // shared-memory staging: row pitch of the staged W (32 V entries)
};

typedef void (*BatchKernel)(BatchClassParams);

namespace batch_detail {

using step_detail::WarpReplica;

// What a warp of a batched kernel keeps in shared memory: its unit's item (read outside
// the steps, so that its fields take no registers of the step) and its flip log.
template <typename Tw> struct UnitShared {
    BatchItemDev it;
    step_detail::FlipLog<typename step_detail::Arith<Tw>::E> log;
};

// One work unit: replica r of item u.it, all of its steps, by the calling warp;
// W points at the item's couplings (global memory, row pitch ldw) or at a
// copy staged in shared memory (SW, row pitch ldw = 32 V).  TRACE: the flipped index of every
// step goes to it.trace where the item has one.
template <typename Tw, int V, bool SW, bool COAL, bool TRACE>
__device__ __forceinline__ void run_unit(UnitShared<Tw>& u, int r, const Tw* W, int ldw, long long t_limit)
{
    // The precomputed Philox words and the table of round keys where there are registers for
    // them: not beside the recompute at V = 32 (1.39 instead of 1.51 ms per 1024 steps of 512
    // replicas without the words), and the table only in the staged kernels, whose bounds
    // leave it room (0.645 against 0.727 ms); the keys come from the unit's item, not from a
    // launch parameter in constant memory.
    constexpr bool kPre = V <= 16 || !std::is_same<Tw, float>::value;
    using R_ = WarpReplica<Tw, V, SW, kPre, COAL>;
    using A = step_detail::Arith<Tw>;
    using H = typename R_::H;
    constexpr bool kReal = std::is_same<Tw, float>::value;
    constexpr int nw = V;   // state words per replica (the padded width 32V / 32)
    const BatchItemDev& it = u.it;
    const int lane = threadIdx.x & 31;
    R_ rp;
    rp.init(W, it.N, ldw, (uint32_t)r, it.xs + ((size_t)it.R + r) * nw, u.log.f, &u.log.head);
#pragma unroll
    for (int v = 0; v < V; ++v) {
        if constexpr (std::is_same<Tw, step_detail::f32e>::value)   // int32 diagonal, exact in fp32
            rp.h[v] = ((rp.valid >> v) & 1u) ? __int2float_rn(static_cast<const int32_t*>(it.diag)[rp.base + v]) : 0.f;
        else
            rp.h[v] = ((rp.valid >> v) & 1u) ? static_cast<const H*>(it.diag)[rp.base + v] : H(0);
    }
    rp.xm = 0;
    rp.m = 0;
    const std::conditional_t<SW, PhiloxKeys, PhiloxSeed> keys(it.seed);
    const float inc = it.inc;
    const int* stop = it.stop;
    // a period beyond any step count never comes
    const uint32_t period = kReal && it.recompute_every <= 0xffffffffll ? (uint32_t)it.recompute_every : 0u;
    const uint32_t T = (uint32_t)(t_limit > 0 ? std::min(t_limit, it.T) : it.T);   // < 2^32
    rp.begin(0, T, it.beta, 0.f, 0, 0, 0, keys);
    // the steps up to the next point where something else is due: a recompute of the
    // fp32 fields, a look at the stop flag, the end
    uint32_t t = 0;
    while (t < T) {
        // the draws (and their step-invariant words) are made anew after a recompute: dead
        // across it, they free their registers for it
        if constexpr (kPre) {
            rp.prep_draws(keys);
            rp.draw_pre(t, keys);
        } else {
            rp.draw(t, keys);
        }
        uint32_t t1 = T;
        if (period > 0 && period - t % period < t1 - t) t1 = t + (period - t % period);
        if (stop && 1024 - t % 1024 < t1 - t) t1 = t + (1024 - t % 1024);
        int k = -1;
        for (; t < t1; ++t) {
            k = rp.template step<false>(t, true, inc, keys);
            if constexpr (TRACE) {
                if (it.trace && lane == 0) it.trace[(size_t)r * it.T + t] = k;
            }
        }
        if (stop && t % 1024 == 0 && *reinterpret_cast<const volatile int*>(stop)) break;
        if constexpr (kReal) {
            if (period > 0 && t % period == 0) {
                if (rp.n > 0) rp.settle(k >= 0);
                rp.recompute(static_cast<const float*>(it.diag), it.S);
                rp.test_current();
            }
        }
    }
    if (rp.n > 0) rp.settle();
    const uint32_t word = rp.word();
    if (lane % R_::P == 0) it.xs[(size_t)r * nw + (rp.base >> 5)] = word;
    if (lane == 0) {
        ReplicaScalars s;
        s.E = A::store_e(u.log.head.E);
        s.best = A::store_e(u.log.head.best);
        s.flips = u.log.head.flips;
        s.m = rp.m;
        s.check = 0;
        it.sc[r] = s;
    }
    __syncwarp();           // every lane is done with the item before the next one takes its place
}

// COAL: rows of W from the items' copies in the one-warp row order (it.Wc).
// Blocks per SM in the launch bounds: registers enough for the step without spills (the
// compiler's own choice leaves V = 16 with fewer: 0.77 instead of 0.69 ms per 1024 steps
// of 512 fp32 replicas).  TRACE is a kernel of its own: a test of the item's trace in every
// step costs launches without one 1 to 5 %.
template <typename Tw, int V, bool COAL, bool TRACE>
__global__ void __launch_bounds__(128, V == 4 ? 4 : V == 8 ? 3 : 2)
    batch_kernel(const __grid_constant__ BatchClassParams bp)
{
    __shared__ UnitShared<Tw> shared[4];
    UnitShared<Tw>& u = shared[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned long long unit = 0;
        if (lane == 0) unit = atomicAdd(bp.head, 1ull);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= (unsigned long long)bp.total_units) break;
        // the item holding this unit (items sorted by unit0)
        int lo = 0, hi = bp.n_items - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((unsigned long long)bp.items[mid].unit0 <= unit) lo = mid;
            else hi = mid - 1;
        }
        if (lane == 0) u.it = bp.items[lo];
        __syncwarp();
        const int r = (int)(unit - (unsigned long long)u.it.unit0);
        if constexpr (COAL) run_unit<Tw, V, false, true, TRACE>(u, r, static_cast<const Tw*>(u.it.Wc), 32 * V, bp.t_limit);
        else run_unit<Tw, V, false, false, TRACE>(u, r, static_cast<const Tw*>(u.it.W), u.it.ldw, bp.t_limit);
    }
}

// Shared-memory staging: the block takes group g = (item, r0) from the
// counter, copies rows 0..N-1 of the item's W into shared memory (row pitch
// 32 V, zeros beyond column N), and warp w runs replica r0 + w.
template <typename Tw, int V, bool TRACE>
__global__ void __launch_bounds__(512) batch_kernel_smem(const __grid_constant__ BatchClassParams bp)
{
    extern __shared__ __align__(16) unsigned char wsm_raw[];
    Tw* Ws = reinterpret_cast<Tw*>(wsm_raw);
    __shared__ long long s_group;
    __shared__ UnitShared<Tw> shared[16];
    const int warp = threadIdx.x >> 5;
    for (;;) {
        __syncthreads();   // every warp is done with the previous group's copy
        if (threadIdx.x == 0) s_group = (long long)atomicAdd(bp.head, 1ull);
        __syncthreads();
        const long long g = s_group;
        if (g >= bp.n_groups) break;
        const int2 gi = bp.groups[g];
        const BatchItemDev it = bp.items[gi.x];
        const Tw* Wg = static_cast<const Tw*>(it.W);
        const int cols = bp.pitch;
        for (int e = threadIdx.x; e < it.N * cols; e += blockDim.x) {
            const int row = e / cols, col = e - row * cols;
            Tw v{};
            if (col < it.N) v = Wg[(size_t)row * it.ldw + col];
            Ws[e] = v;
        }
        __syncthreads();
        const int r = gi.y + warp;
        if ((threadIdx.x & 31) == 0) shared[warp].it = it;
        __syncwarp();
        if (r < it.R) run_unit<Tw, V, true, false, TRACE>(shared[warp], r, Ws, cols, bp.t_limit);
    }
}

// Kernels per step coupling form wk: kWInt8AsF32 (integer instances on exact
// fp32 couplings), kWFp32, kWInt16 (16-bit couplings, int32 fields; rows from L2
// only: the staged copy holds 4-byte entries).
template <bool TRACE>
inline BatchKernel smem_kernel_for(int wk, int V)
{
    if (wk == kWInt16) return nullptr;
    if (wk == kWInt8AsF32) {
        switch (V) {
        case 4: return batch_kernel_smem<step_detail::f32e, 4, TRACE>;
        case 8: return batch_kernel_smem<step_detail::f32e, 8, TRACE>;
        }
    } else {
        switch (V) {
        case 4: return batch_kernel_smem<float, 4, TRACE>;
        case 8: return batch_kernel_smem<float, 8, TRACE>;
        }
    }
    return nullptr;
}

// The rows-from-L2 kernel of a class; coal: its items carry the row-ordered copies
// (the fp32 forms at V >= 8).
template <bool TRACE>
inline BatchKernel kernel_for(int wk, int V, bool coal)
{
    if (coal && wk == kWInt8AsF32) {
        switch (V) {
        case 8: return batch_kernel<step_detail::f32e, 8, true, TRACE>;
        case 16: return batch_kernel<step_detail::f32e, 16, true, TRACE>;
        case 32: return batch_kernel<step_detail::f32e, 32, true, TRACE>;
        }
        return nullptr;
    }
    if (coal && wk == kWFp32) {
        switch (V) {
        case 8: return batch_kernel<float, 8, true, TRACE>;
        case 16: return batch_kernel<float, 16, true, TRACE>;
        case 32: return batch_kernel<float, 32, true, TRACE>;
        }
        return nullptr;
    }
    if (wk == kWInt16) {
        switch (V) {
        case 4: return batch_kernel<int16_t, 4, false, TRACE>;
        case 8: return batch_kernel<int16_t, 8, false, TRACE>;
        case 16: return batch_kernel<int16_t, 16, false, TRACE>;
        case 32: return batch_kernel<int16_t, 32, false, TRACE>;
        }
    } else if (wk == kWInt8AsF32) {
        switch (V) {
        case 4: return batch_kernel<step_detail::f32e, 4, false, TRACE>;
        case 8: return batch_kernel<step_detail::f32e, 8, false, TRACE>;
        case 16: return batch_kernel<step_detail::f32e, 16, false, TRACE>;
        case 32: return batch_kernel<step_detail::f32e, 32, false, TRACE>;
        }
    } else {
        switch (V) {
        case 4: return batch_kernel<float, 4, false, TRACE>;
        case 8: return batch_kernel<float, 8, false, TRACE>;
        case 16: return batch_kernel<float, 16, false, TRACE>;
        case 32: return batch_kernel<float, 32, false, TRACE>;
        }
    }
    return nullptr;
}

}  // namespace batch_detail

// The kernels that store traces (da_batch_traced.cu).
BatchKernel traced_smem_kernel_for(int wk, int V);
BatchKernel traced_kernel_for(int wk, int V, bool coal);

}  // namespace da
