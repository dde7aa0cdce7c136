// da_step_common.cuh -- arithmetic and warp helpers shared by the step
// kernels (da_step.cuh, da_replica.cuh, da_batch.cu).
#pragma once
#include "da_device.cuh"
#include "da_internal.h"

namespace da {
namespace step_detail {

template <typename Tw> struct Arith;
template <> struct Arith<int8_t> {
    using H = int32_t;    // effective fields
    using E = long long;  // tracked energy
    static __device__ __forceinline__ H signed_field(H g, uint32_t x) { return x ? -g : g; }
    static __device__ __forceinline__ float to_float(H g) { return __int2float_rn(g); }
    using Sign = int32_t;
    static __device__ __forceinline__ Sign sign(uint32_t xold) { return xold ? -1 : 1; }
    static __device__ __forceinline__ H apply_signed(H h, int8_t w, Sign s) { return h + s * (H)w; }
    static __device__ __forceinline__ E load_e(long long b) { return b; }
    static __device__ __forceinline__ long long store_e(E e) { return e; }
    static constexpr bool kReal = false;
    static __device__ __forceinline__ uint32_t log_bits(H dE) { return (uint32_t)dE; }
    static __device__ __forceinline__ long long log_int(uint32_t b) { return (long long)(int)b; }
};
// 16-bit integer couplings (the DA's fixed-point precision): as int8, wider W.
template <> struct Arith<int16_t> {
    using H = int32_t;
    using E = long long;
    static __device__ __forceinline__ H signed_field(H g, uint32_t x) { return x ? -g : g; }
    static __device__ __forceinline__ float to_float(H g) { return __int2float_rn(g); }
    using Sign = int32_t;
    static __device__ __forceinline__ Sign sign(uint32_t xold) { return xold ? -1 : 1; }
    static __device__ __forceinline__ H apply_signed(H h, int16_t w, Sign s) { return h + s * (H)w; }
    static __device__ __forceinline__ E load_e(long long b) { return b; }
    static __device__ __forceinline__ long long store_e(E e) { return e; }
    static constexpr bool kReal = false;
    static __device__ __forceinline__ uint32_t log_bits(H dE) { return (uint32_t)dE; }
    static __device__ __forceinline__ long long log_int(uint32_t b) { return (long long)(int)b; }
};
template <> struct Arith<float> {
    using H = float;
    using E = double;
    static __device__ __forceinline__ H signed_field(H g, uint32_t x)
    {
        return __int_as_float(__float_as_int(g) ^ (int)(x << 31));
    }
    static __device__ __forceinline__ float to_float(H g) { return g; }
    using Sign = float;
    static __device__ __forceinline__ Sign sign(uint32_t xold) { return xold ? -1.0f : 1.0f; }
    // h + s w with s = +-1: the product is exact, so this is the same single
    // rounding as a correctly rounded addition or subtraction
    static __device__ __forceinline__ H apply_signed(H h, float w, Sign s) { return __fmaf_rn(s, w, h); }
    static __device__ __forceinline__ E load_e(long long b) { return __longlong_as_double(b); }
    static __device__ __forceinline__ long long store_e(E e) { return __double_as_longlong(e); }
    static constexpr bool kReal = true;
    static __device__ __forceinline__ uint32_t log_bits(H dE) { return __float_as_uint(dE); }
};

// Integer couplings of a DA_INT8 instance stored as fp32 (exact: |W| <= 128 and
// every |Q_ii| + sum_j |Q_ij| < 2^24, so every field and Delta E is an exact
// fp32 integer): the step runs on fp32 fields and FFMA updates, with exactly
// the values of the int8/int32 form, and books the energy in int64.
struct f32e {
    float f;
};
template <> struct Arith<f32e> {
    using H = float;
    using E = long long;
    static __device__ __forceinline__ H signed_field(H g, uint32_t x) { return Arith<float>::signed_field(g, x); }
    static __device__ __forceinline__ float to_float(H g) { return g; }
    using Sign = float;
    static __device__ __forceinline__ Sign sign(uint32_t xold) { return xold ? -1.0f : 1.0f; }
    static __device__ __forceinline__ H apply_signed(H h, f32e w, Sign s) { return __fmaf_rn(s, w.f, h); }
    static __device__ __forceinline__ E load_e(long long b) { return b; }
    static __device__ __forceinline__ long long store_e(E e) { return e; }
    static constexpr bool kReal = false;
    static __device__ __forceinline__ uint32_t log_bits(H dE) { return __float_as_uint(dE); }
    static __device__ __forceinline__ long long log_int(uint32_t b) { return (long long)__float2int_rn(__uint_as_float(b)); }
};

// Delta E_i as the acceptance test takes it: fl32((1 - 2 x) g).  Rounding is
// symmetric, so the sign is applied to the rounded field (integer fields: one
// conversion and one xor instead of a negation, a selection and a conversion).
template <typename A>
__device__ __forceinline__ float delta_of(typename A::H g, uint32_t x)
{
    return __int_as_float(__float_as_int(A::to_float(g)) ^ (int)(x << 31));
}

// ---- tracked energy and best state, 32 flips at a time ----------------------------
// The tracked energy of a replica (the in-order sum of the flips' Delta E: fp64 sum of
// fp32 values for real couplings, int64 for integer ones) and the best-state test
// after every flip are needed by nothing inside a step.  A step only appends (Delta E,
// k) to a log of 32 entries; settle_log() then forms all of the window's energies at
// once, one flip per lane, and finds the first strictly lowest one; the state it
// belongs to is the current state with the later flips undone.  Per flip this costs
// one store, where the test after every flip cost an fp64 conversion, add, compare and
// branch (64 + 64 + 110 cycles alone and one fp64 warp instruction per 19 cycles and
// SM, measured) and, at a new best state, a store of the state under the step.
struct FlipEntry {
    uint32_t dE;   // bits of Delta E (fp32 or int32)
    int k;         // flipped variable
};
template <typename EE> struct FlipHead {   // one per warp
    EE E, best;        // up to the last settled flip
    long long flips;
};
template <typename EE> struct FlipLog {
    FlipEntry f[32];
    FlipHead<EE> head;
};

__device__ __forceinline__ long long warp_min(long long v)   // over the warp
{
    const int hi = (int)(v >> 32);
    const int mh = __reduce_min_sync(0xffffffffu, hi);
    const uint32_t ml = __reduce_min_sync(0xffffffffu, hi == mh ? (uint32_t)v : 0xffffffffu);
    return (long long)mh << 32 | ml;
}

// Inclusive prefix sums of v over the lanes, and the first lane below `tested` with the
// lowest one (`low`).
__device__ __forceinline__ int first_lowest(long long v, int lane, int tested, long long& low)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    const long long w = lane < tested ? v : 0x7FFFFFFFFFFFFFFFll;
    low = warp_min(w);
    return __ffs(__ballot_sync(0xffffffffu, w == low)) - 1;
}

// Sums over the warp of values whose absolute values sum to at most 2^53.
__device__ __forceinline__ long long warp_sum53(long long v)
{
    const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)v & 0x3FFFFFFu);
    const int hi = __reduce_add_sync(0xffffffffu, (int)(v >> 26));
    return ((long long)hi << 26) + (long long)lo;
}

// The n <= 32 flips of a log added to E in order; the first `tested` resulting energies
// are tested: returns the index of the flip after which the energy was first strictly
// lowest, if that is below `best` (then best = that energy), or -1.
template <typename A>
__device__ __forceinline__ int settle_log(const FlipEntry* f, int n, int tested, int lane, typename A::E& E,
                                          typename A::E& best)
{
    const uint32_t bits = lane < n ? f[lane].dE : 0u;
    if constexpr (!A::kReal) {
        const long long v = A::log_int(bits);            // |v| < 2^31 each
        const long long neg = warp_sum53(min(v, 0ll));
        int at = -1;
        if (E + neg < best && tested > 0) {
            long long low;
            const int q = first_lowest(v, lane, tested, low);
            if (E + low < best) {
                best = E + low;
                at = q;
            }
        }
        E += warp_sum53(v);
        return at;
    } else {
        // Where E and every value are multiples of a unit 2^(k-53) and no partial sum can
        // exceed 2^k, each fp64 addition of the in-order sum is exact, and so are the
        // sums of the values as integers; otherwise the additions are made one by one.
        const uint32_t a = bits & 0x7FFFFFFFu;
        const uint32_t amax = __reduce_max_sync(0xffffffffu, a);
        const unsigned long long eb = (unsigned long long)__double_as_longlong(E);
        const int xE = (int)(eb >> 52) & 0x7FF;
        const bool zero = (eb << 1) == 0;
        const int ed = (int)(amax >> 23) - 127;          // |Delta E| < 2^(ed + 1): they sum to less than 2^(ed + 6)
        bool exact = ed <= 100 && ed >= -100 && (zero || (xE >= 600 && xE <= 1400));
        if (exact) {                                      // uniform
            const int eE = xE - 1023;                     // |E| = mE 2^(eE - 52)
            const unsigned long long mE = (eb & 0xFFFFFFFFFFFFFull) | (1ull << 52);
            int unit;                                     // k - 53
            if (zero) {
                unit = ed + 6 - 53;
            } else {
                const int s = ed + 6 - (eE - 52);
                const bool room = s <= 52 && mE + (1ull << max(s, 0)) <= (1ull << 53);
                unit = (room ? eE + 1 : max(eE + 1, ed + 6) + 1) - 53;
                const int drop = unit - (eE - 52);        // >= 0
                exact = drop < 53 && (mE & ((1ull << drop) - 1)) == 0;
            }
            const uint32_t x = a >> 23;
            const uint32_t mant = x ? (a & 0x7FFFFFu) | 0x800000u : a;
            const int sh = (int)max(x, 1u) - 150 - unit;  // Delta E = +-mant 2^(sh + unit), below 2^53 units
            long long v = 0;
            if (mant) {
                if (sh >= 0) v = (long long)mant << min(sh, 38);
                else if (sh > -24 && (mant & ((1u << -sh) - 1u)) == 0) v = mant >> -sh;
                else exact = false;
            }
            if (__all_sync(0xffffffffu, exact)) {
                if ((int)bits < 0) v = -v;
                const double scale = __longlong_as_double((long long)(unit + 1023) << 52);
                const double low_bound = __fma_rn(__ll2double_rn(warp_sum53(min(v, 0ll))), scale, E);   // exact
                int at = -1;
                if (low_bound < best && tested > 0) {
                    long long low;
                    const int q = first_lowest(v, lane, tested, low);
                    const double lowE = __fma_rn(__ll2double_rn(low), scale, E);
                    if (lowE < best) {
                        best = lowE;
                        at = q;
                    }
                }
                E = __fma_rn(__ll2double_rn(warp_sum53(v)), scale, E);
                return at;
            }
        }
        int at = -1;
        for (int q = 0; q < n; ++q) {
            E = __dadd_rn(E, (double)__uint_as_float(f[q].dE));
            if (q < tested && E < best) {
                best = E;
                at = q;
            }
        }
        return at;
    }
}

// The positions before the r-th (0-based) set bit of w, as a mask (its population count is
// the position): lane v counts the set bits up to v, and the positions with at most r of
// them precede the bit.
__device__ __forceinline__ uint32_t bits_before(uint32_t w, int r, int lane)
{
    return __ballot_sync(0xffffffffu, __popc(w & (0xffffffffu >> (31 - lane))) <= r);
}

// h[vk] for a warp-uniform vk: a tree of selections up to V = 16 (the indirect branch of
// a switch sits on the way to the row load: N = 256 0.538 -> 0.493 us per step, N = 512
// 0.652 -> 0.603, fp32 with 64 replicas), a switch for V = 32, where 31 selections cost
// more than the branch (1.274 against 1.330 us per step at N = 1024, 1024 replicas).
template <typename H, int V>
__device__ __forceinline__ H select_slot(const H (&h)[V], int vk)
{
    if constexpr (V <= 16) {
        H a[V];
#pragma unroll
        for (int v = 0; v < V; ++v) a[v] = h[v];
#pragma unroll
        for (int w = V / 2; w >= 1; w /= 2) {
#pragma unroll
            for (int v = 0; v < w; ++v) a[v] = (vk & w) ? a[v + w] : a[v];
        }
        return a[0];
    }
#define DA_SLOT(n) \
    case n:        \
        if constexpr (V > n) return h[n]; else return h[0];
    switch (vk) {
        DA_SLOT(0) DA_SLOT(1) DA_SLOT(2) DA_SLOT(3) DA_SLOT(4) DA_SLOT(5) DA_SLOT(6) DA_SLOT(7)
        DA_SLOT(8) DA_SLOT(9) DA_SLOT(10) DA_SLOT(11) DA_SLOT(12) DA_SLOT(13) DA_SLOT(14) DA_SLOT(15)
        DA_SLOT(16) DA_SLOT(17) DA_SLOT(18) DA_SLOT(19) DA_SLOT(20) DA_SLOT(21) DA_SLOT(22) DA_SLOT(23)
        DA_SLOT(24) DA_SLOT(25) DA_SLOT(26) DA_SLOT(27) DA_SLOT(28) DA_SLOT(29) DA_SLOT(30) DA_SLOT(31)
    default: return h[0];
    }
#undef DA_SLOT
}

__device__ __forceinline__ void group_barrier(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Loads of instance data through the read-only path: a kernel's inputs are
// fixed while it runs.
template <typename T>
__device__ __forceinline__ T ldx(const T* p)
{
    return __ldg(p);
}

// Row k of W at the V consecutive entries of this lane (16-byte loads where
// the lane's slice allows).  load() reads global memory through the read-only
// path; load_shared() reads a copy of W staged in shared memory (fp32 forms
// only).
template <typename Tw, int V> struct Row;
template <int V> struct Row<float, V> {
    static __device__ __forceinline__ void load(const float* p, float (&c)[V])
    {
        static_assert(V % 4 == 0, "V");
#pragma unroll
        for (int q = 0; q < V / 4; ++q) {
            const float4 f = ldx(reinterpret_cast<const float4*>(p) + q);
            c[4 * q] = f.x; c[4 * q + 1] = f.y; c[4 * q + 2] = f.z; c[4 * q + 3] = f.w;
        }
    }
};
template <int V> struct Row<f32e, V> {
    static __device__ __forceinline__ void load(const f32e* p, f32e (&c)[V])
    {
        static_assert(V % 4 == 0, "V");
#pragma unroll
        for (int q = 0; q < V / 4; ++q) {
            const float4 f = ldx(reinterpret_cast<const float4*>(p) + q);
            c[4 * q].f = f.x; c[4 * q + 1].f = f.y; c[4 * q + 2].f = f.z; c[4 * q + 3].f = f.w;
        }
    }
};

// Row k of W in the warp row order (step_uses_coal in da_internal.h): p points at
// the lane's first entry; float4 number q, at p + 128 q, holds the lane's slots
// 4 q .. 4 q + 3.
template <typename Tw, int V> struct RowCoal;
template <int V> struct RowCoal<float, V> {
    static __device__ __forceinline__ void load(const float* p, float (&c)[V])
    {
        static_assert(V % 4 == 0, "V");
#pragma unroll
        for (int q = 0; q < V / 4; ++q) {
            const float4 f = ldx(reinterpret_cast<const float4*>(p + 128 * q));
            c[4 * q] = f.x; c[4 * q + 1] = f.y; c[4 * q + 2] = f.z; c[4 * q + 3] = f.w;
        }
    }
};
template <int V> struct RowCoal<f32e, V> {
    static __device__ __forceinline__ void load(const f32e* p, f32e (&c)[V])
    {
        static_assert(V % 4 == 0, "V");
        const float* pf = reinterpret_cast<const float*>(p);
#pragma unroll
        for (int q = 0; q < V / 4; ++q) {
            const float4 f = ldx(reinterpret_cast<const float4*>(pf + 128 * q));
            c[4 * q].f = f.x; c[4 * q + 1].f = f.y; c[4 * q + 2].f = f.z; c[4 * q + 3].f = f.w;
        }
    }
};

// 16-byte loads from shared memory (p points into the block's staged copy).
template <typename Tw, int V> struct RowShared {
    static __device__ __forceinline__ void load(const Tw* p, Tw (&c)[V])
    {
        static_assert(sizeof(Tw) == 4 && V % 4 == 0, "fp32 forms only");
        const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
#pragma unroll
        for (int q = 0; q < V / 4; ++q) {
            float x, y, z, w;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(x), "=f"(y), "=f"(z), "=f"(w)
                         : "r"(a + 16u * q)
                         : "memory");
            reinterpret_cast<float*>(&c[4 * q])[0] = x;
            reinterpret_cast<float*>(&c[4 * q + 1])[0] = y;
            reinterpret_cast<float*>(&c[4 * q + 2])[0] = z;
            reinterpret_cast<float*>(&c[4 * q + 3])[0] = w;
        }
    }
};
template <int V> struct Row<int8_t, V> {
    static __device__ __forceinline__ void unpack(uint32_t u, int8_t* c)
    {
        c[0] = (int8_t)(u & 0xFFu); c[1] = (int8_t)((u >> 8) & 0xFFu);
        c[2] = (int8_t)((u >> 16) & 0xFFu); c[3] = (int8_t)(u >> 24);
    }
    static __device__ __forceinline__ void load(const int8_t* p, int8_t (&c)[V])
    {
        if constexpr (V == 4) {
            unpack(ldx(reinterpret_cast<const unsigned int*>(p)), c);
        } else if constexpr (V == 8) {
            const uint2 u = ldx(reinterpret_cast<const uint2*>(p));
            unpack(u.x, c); unpack(u.y, c + 4);
        } else {
#pragma unroll
            for (int q = 0; q < V / 16; ++q) {
                const uint4 u = ldx(reinterpret_cast<const uint4*>(p) + q);
                unpack(u.x, c + 16 * q); unpack(u.y, c + 16 * q + 4);
                unpack(u.z, c + 16 * q + 8); unpack(u.w, c + 16 * q + 12);
            }
        }
    }
};

template <int V> struct Row<int16_t, V> {
    static __device__ __forceinline__ void unpack(uint32_t u, int16_t* c)
    {
        c[0] = (int16_t)(u & 0xFFFFu);
        c[1] = (int16_t)(u >> 16);
    }
    static __device__ __forceinline__ void load(const int16_t* p, int16_t (&c)[V])
    {
        if constexpr (V == 4) {
            const uint2 u = ldx(reinterpret_cast<const uint2*>(p));
            unpack(u.x, c); unpack(u.y, c + 2);
        } else {
#pragma unroll
            for (int q = 0; q < V / 8; ++q) {
                const uint4 u = ldx(reinterpret_cast<const uint4*>(p) + q);
                unpack(u.x, c + 8 * q); unpack(u.y, c + 8 * q + 2);
                unpack(u.z, c + 8 * q + 4); unpack(u.w, c + 8 * q + 6);
            }
        }
    }
};

// Replicas per block and the blocks per SM the register budget is sized for: 8 one-warp
// replicas per SM, so that 1024 replicas fill 152 SMs in one wave; for G > 1 as many as
// fit without spills (sized for 7 blocks per SM, G = 4 with V = 8 took 0.729 instead of
// 0.596 us per step at N = 1024; sized for 2, G = 8 with V = 32 3.05 instead of 1.72 at
// N = 8192; 32 replicas).
template <int G, int V> struct OccupancyGV;
template <int V> struct OccupancyGV<1, V> { static constexpr int rpb = 4, min_blocks = 2; };
template <int V> struct OccupancyGV<2, V> { static constexpr int rpb = 2, min_blocks = V == 32 ? 3 : 4; };
template <int V> struct OccupancyGV<4, V> { static constexpr int rpb = 1, min_blocks = V == 32 ? 3 : 4; };
template <int V> struct OccupancyGV<8, V> { static constexpr int rpb = 1, min_blocks = V >= 16 ? 1 : 2; };

// The state words of a replica are standard bit-packed words (x_i is bit i%32
// of word i/32); a lane's V bits are one slice of word (w*32V + l*V) / 32.
template <int V>
__device__ __forceinline__ uint32_t gather_word(uint32_t bits, int lane)
{
    constexpr int P = 32 / V;  // lanes per word
    uint32_t m = (V == 32) ? bits : (bits << ((lane % P) * V));
#pragma unroll
    for (int o = 1; o < P; o <<= 1) m |= __shfl_xor_sync(0xffffffffu, m, o);
    return m;
}

// Trials (a)-(b) of one lane's V variables in the log domain (lg2_draw,
// kLogBand in da_device.cuh): returns the mask of surely accepted trials and
// sets `unsure` when any trial has |t| <= kLogBand and must take the exact
// test (decide_exact).  With E_off = +0 (no offset, or no step without a flip
// since the last one) the subtraction returns delta unchanged: at V = 32 a branch
// leaves it out, below that V packed additions cost less than the branch (N = 64
// 0.398 -> 0.377 us per step, N = 1024 with 1024 replicas 1.274 -> 1.286 without it).
// The test is made on t' = s - (24 - kLogBand), s = fma(delta, c, L), instead of
// t = s - 24: wherever |t| < 12, s lies in [12, 36] and both subtractions are
// exact (Sterbenz), so t' = t + kLogBand and
//   t < -kLogBand  <=>  t' < 0      (its sign bit; t' = +0 when t = -kLogBand),
//   |t| <= kLogBand <=> 0 <= t' <= 2 kLogBand (its bits as an unsigned integer
//                       at most those of 2^-14: negative t' have bit 31 set);
// elsewhere both sides agree on a sign far from the band.  The sign bits are
// shifted into the mask and the band is one unsigned minimum per trial; pairs of
// trials share one packed fma and one packed add (each lane of a packed
// operation rounds as the scalar one).
template <typename A, int V>
__device__ __forceinline__ uint32_t decide_log(const typename A::H (&h)[V], uint32_t xm, float Eoff, float c,
                                               const float (&L)[V], bool& unsure)
{
    static_assert(V % 2 == 0, "trials are decided in pairs");
    constexpr float kShift = 24.0f - kLogBand;   // 23.999969482421875, exact in fp32
    constexpr uint32_t kBandBits = 0x38800000u;  // 2^-14 = 2 kLogBand
    const float2 cc = make_float2(c, c), sh = make_float2(-kShift, -kShift);
    uint32_t acc = 0, umin = 0xffffffffu;
    auto pair = [&](int v, float d0, float d1) {
        const float2 tp = __fadd2_rn(__ffma2_rn(make_float2(d0, d1), cc, make_float2(L[v], L[v + 1])), sh);
        const uint32_t b0 = __float_as_uint(tp.x), b1 = __float_as_uint(tp.y);
        acc = __funnelshift_l(b1, acc, 1);       // bit v + 1, then bit v
        acc = __funnelshift_l(b0, acc, 1);
        umin = min(umin, min(b0, b1));
    };
    if (V > 16 && Eoff == 0.0f) {
#pragma unroll
        for (int v = V - 2; v >= 0; v -= 2)
            pair(v, delta_of<A>(h[v], (xm >> v) & 1u), delta_of<A>(h[v + 1], (xm >> (v + 1)) & 1u));
    } else {
#pragma unroll
        for (int v = V - 2; v >= 0; v -= 2)
            pair(v, __fsub_rn(delta_of<A>(h[v], (xm >> v) & 1u), Eoff),
                 __fsub_rn(delta_of<A>(h[v + 1], (xm >> (v + 1)) & 1u), Eoff));
    }
    unsure = umin <= kBandBits;
    return acc;
}

// The trials of this lane with |t| <= kLogBand, decided by the exact test
// delta <= 0 || u < exp_neg(-beta delta) with u from the trial's Philox word
// (recomputed: block (i/4, t, rep, 0), lane i%4 for variable i = base + v).
template <typename A, int V, class Keys>
__device__ __forceinline__ uint32_t decide_exact(const typename A::H (&h)[V], uint32_t xm, float Eoff, float beta,
                                                 const float (&L)[V], uint32_t acc, int base, uint32_t step,
                                                 uint32_t rep, const Keys& keys)
{
    const float c = __fmul_rn(beta, kLog2e);
    uint32_t band = 0;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const float t = __fsub_rn(__fmaf_rn(__fsub_rn(delta_of<A>(h[v], (xm >> v) & 1u), Eoff), c, L[v]), 24.0f);
        band |= (uint32_t)(fabsf(t) <= kLogBand) << v;
    }
    while (band) {
        const int v = __ffs(band) - 1;
        band &= band - 1;
        const float delta = __fsub_rn(delta_of<A>(select_slot<typename A::H, V>(h, v), (xm >> v) & 1u), Eoff);
        const float ax = -__fmul_rn(beta, delta);
        const uint32_t wd = pick(philox4x32_10((uint32_t)((base + v) >> 2), step, rep, 0u, keys), v & 3);
        acc |= (uint32_t)(delta <= 0.0f || uniform01(wd) < exp_neg(ax)) << v;
    }
    return acc;
}

// The rare parts of a step out of line, so that the code a step runs through is short and in
// one piece: with one or two warps per scheduler its instruction fetch is exposed (0.27
// stall cycles per instruction at V = 8).  Measured per V: N = 1024 with 1024 replicas
// 1.209 -> 1.182 us per step, with 128 (V = 8) 0.620 -> 0.608, N = 64 0.352 -> 0.347; but
// V = 16 keeps them inline where it is not WIDE (WarpReplica; step_kernel for the other case).

// decide_exact, where OUT out of line on copies of the lane's fields and draws made for the call.
template <typename A, int V> struct ExactArgs {
    typename A::H h[V];
    float L[V];
};
template <typename A, int V, class Keys>
__device__ __noinline__ uint32_t decide_exact_call(const ExactArgs<A, V>& a, uint32_t xm, float Eoff, float beta,
                                                   uint32_t acc, int base, uint32_t step, uint32_t rep,
                                                   const Keys& keys)
{
    return decide_exact<A, V>(a.h, xm, Eoff, beta, a.L, acc, base, step, rep, keys);
}
template <typename A, int V, bool OUT, class Keys>
__device__ __forceinline__ uint32_t decide_exact_out(const typename A::H (&h)[V], uint32_t xm, float Eoff, float beta,
                                                     const float (&L)[V], uint32_t acc, int base, uint32_t step,
                                                     uint32_t rep, const Keys& keys)
{
    if constexpr (!OUT) {
        return decide_exact<A, V>(h, xm, Eoff, beta, L, acc, base, step, rep, keys);
    } else {
        ExactArgs<A, V> a;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            a.h[v] = h[v];
            a.L[v] = L[v];
        }
        return decide_exact_call<A, V>(a, xm, Eoff, beta, acc, base, step, rep, keys);
    }
}

}  // namespace step_detail
}  // namespace da
