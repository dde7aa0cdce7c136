// da_mma.cu -- the exact field recompute on the tensor cores (tcgen05).
//
// The recompute g = diag + W x of R states is a dense contraction
// G[r][i] = sum_j X[r][j] W[j][i] with X in {0, 1}: the states are the M side
// (128 per tile, one per TMEM lane), the variables i the N side (64 per tile)
// and the couplings j the K side.  Its value is defined exactly (da_fields.cu):
// every coupling is put on the fixed-point grid, v_ij = round(W_ij 2^S) (the
// integer couplings themselves), and summed in integers.  The tensor cores reach
// the same integers: v is split into balanced digits of b bits,
//   v = sum_l d_l 2^(b l),   d_l in [-2^(b-1), 2^(b-1)),
// every digit is exact in fp16 (|d| <= 2048), and b is chosen so that no
// partial sum of digits over the K side exceeds 2^22 in magnitude, inside
// the 24-bit integer range of the fp32 accumulator.  Each digit plane is one
// accumulator in tensor memory; the epilogue combines the planes in 64-bit
// integers, adds the fixed-point diagonal and rounds once, exactly like the
// CUDA-core form.
//
// Operands use the tensor core's canonical K-major layout (8-row x 16-byte
// core matrices, [K chunk][row group][8][8] halves per tile).  The digit planes
// of the instance are built once per context in that layout in HBM, so a
// pipeline stage takes them in contiguous bulk copies; the states are not
// staged in HBM at all: eight warps of the block expand the tile's state bits
// (2 words per state and stage) to f16 {0, 1} directly into the stage.
//
// Block: 16 warps, 128 states x 64 variables.  Warp 0 allocates tensor memory and
// issues the digit planes' bulk copies (4 KB a lane) into a 3-stage ring; warps 2-9
// write the stage's state tile (half a state each, the word of the next chunk loaded
// while the current one is written); one thread of warp 1 issues the MMAs (4 K-steps of
// 16 per stage, the digit planes side by side as the columns of one MMA, up to four planes,
// or of two: one MMA of 64 columns per plane took 1.17 us a stage at 5 planes, this form
// 0.85) and
// commits the stage back to both producers; then all 16 warps read their TMEM lanes
// (warp w: states 32 (w % 4).., 16 variables from 16 (w / 4)) and write fields and
// 128-bit partial energies, and the last block of a state tile sums those.
//
// What bounds it at the sizes of an anneal (N = 1024) is the chain of a short launch:
// 16 stages of 0.5 us of MMAs each, and half the time outside them.  With the step
// launch that follows, a recompute at N = 1024 costs 30 us with 128 states (38.5 with
// the energies in a launch of their own and the form before) and 34 us with 1024 (49.4);
// at N = 8192 it streams the digit planes from HBM.  (32-variable tiles, two blocks an
// SM, measured slower: every block expands its states again, and at 6 digit planes only
// one block fits.)
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>
#include <set>
#include <utility>

#include "da_fixed.cuh"
#include "da_internal.h"
#include "da_tc.cuh"

namespace da {
namespace {

constexpr int kBM = kTcStates;   // states per tile (TMEM lanes)
constexpr int kBN = 64;    // variables per tile (TMEM columns per digit plane)
constexpr int kBK = 64;    // couplings per pipeline stage
constexpr int kStages = 3;
constexpr uint32_t kPiece = 4096;            // bytes of one bulk copy (kBTile is a multiple)
constexpr int kThreads = 128 * (kBN / 16);   // warp w reads TMEM lanes 32 (w % 4).., columns 16 (w / 4)..
constexpr int kMinBlocks = 512 / kThreads;   // blocks per SM the launch bounds plan for
constexpr int kExpanders = 2 * kBM;  // threads of warps 2-9: the state tile of each stage, half a state each
constexpr uint32_t kATile = kBM * kBK * 2;   // bytes of one state tile (16 KB)
constexpr uint32_t kBTile = kBN * kBK * 2;   // bytes of one digit-plane tile (8 KB)
constexpr uint32_t kWaitLimit = 1u << 26;    // polls of one mbarrier before giving up ...
constexpr uint64_t kWaitNs = 2000000000ull;  // ... or 2 s, whichever comes first
constexpr int kMaxLimbs = 6;                 // digit planes for any N <= 8192 (tc_digits)

// Offset (in halves) of element (row, k) inside a tile of `rows` x 64 halves
// in the canonical K-major layout without swizzling.
__device__ __forceinline__ size_t core_offset(int rows, int row, int k)
{
    return (size_t)((k >> 3) * (rows >> 3) + (row >> 3)) * 64 + (row & 7) * 8 + (k & 7);
}

template <typename Tw>
__device__ __forceinline__ long long fixed_w(const void* W, size_t idx, int S)
{
    if constexpr (sizeof(Tw) == 4) return fixed_of_f32(static_cast<const float*>(W)[idx], S);
    else return (long long)static_cast<const Tw*>(W)[idx];   // integer couplings are their own grid
}

template <bool INT8>
__device__ __forceinline__ long long fixed_d(const void* diag, int i, int S)
{
    if constexpr (INT8) return (long long)static_cast<const int32_t*>(diag)[i];
    else return fixed_of_f32(static_cast<const float*>(diag)[i], S);
}

// The diagonal on the fixed-point grid, zero-padded to n entries.
template <bool INT8>
__global__ void build_dfix_kernel(const void* __restrict__ diag, int N, int S, long long* __restrict__ dfix, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dfix[i] = i < N ? fixed_d<INT8>(diag, i, S) : 0ll;
}

// Digit planes: one thread per (tile i, chunk j, row i, group of 8 j).
template <typename Tw>
__global__ void build_digits_kernel(const void* __restrict__ W, int N, int ldw, int S, int bits, int limbs,
                                    int kchunks, __half* __restrict__ B, long long total)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int g = (int)(idx & 7);
    const int row = (int)((idx >> 3) % kBN);
    const long long tile = idx / (8 * kBN);    // itile * kchunks + kchunk
    const int kchunk = (int)(tile % kchunks);
    const int itile = (int)(tile / kchunks);
    const int i = itile * kBN + row;
    const int jb = kchunk * kBK + g * 8;
    long long v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int j = jb + e;
        v[e] = (i < N && j < N) ? fixed_w<Tw>(W, (size_t)j * ldw + i, S) : 0ll;
    }
    const long long half_range = 1ll << (bits - 1);
    const long long mask = (1ll << bits) - 1;
    for (int l = 0; l < limbs; ++l) {
        __align__(16) __half h[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            long long d = v[e] & mask;
            if (d >= half_range) d -= mask + 1;
            v[e] = (v[e] - d) >> bits;
            h[e] = __int2half_rn((int)d);
        }
        __half* dst = B + (size_t)tile * limbs * (kBN * kBK) + core_offset(kBN * limbs, l * kBN + row, g * 8);
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(h);
    }
}

// Two f16 values {0, 1} from two state bits (bit 0 -> the lower half).
__device__ __forceinline__ uint32_t half_pair(uint32_t two)
{
    return (two & 1u) * 0x3C00u + (two >> 1) * 0x3C000000u;   // f16 1.0 = 0x3C00
}

// Makes this thread's shared-memory writes visible to the asynchronous proxy
// (the tensor cores' operand reads).
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

struct I128 {
    unsigned long long lo;
    long long hi;
};

__device__ __forceinline__ void i128_add(I128& a, long long v)
{
    const unsigned long long lo = a.lo + (unsigned long long)v;
    a.hi += (v < 0 ? -1ll : 0ll) + (lo < a.lo ? 1ll : 0ll);
    a.lo = lo;
}

__device__ __forceinline__ void i128_add2(I128& a, const I128& b)
{
    const unsigned long long lo = a.lo + b.lo;
    a.hi += b.hi + (lo < a.lo ? 1ll : 0ll);
    a.lo = lo;
}

// A partial sum that another block wrote (16-byte aligned), from L2.
__device__ __forceinline__ I128 load_partial(const I128* p)
{
    const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(p));
    return I128{v.x, (long long)v.y};
}

struct TcParams {
    const __half* B;        // [ceil(N/64)][kchunks][limbs] digit-plane tiles
    const long long* dfix;  // [kchunks * 64] fixed-point diagonal, zero-padded
    const uint32_t* xs;     // [R][nw] state bits (x_i = bit i % 32 of word i / 32)
    void* hout;             // [R][npad] or null
    I128* part;             // [gridDim.x][R] or null
    unsigned* arrived;      // [gridDim.y], 0 before the launch and after it, or null: the block
                            // of a state tile that comes last sums the partial energies itself
    long long* E;           // with arrived: E[r Estride] as launch_energy_sum writes it
    int Estride;
    uint32_t* check;        // or null: check[r 2 Estride] = 1 with every E[r Estride]
    int* err;
    int N, S, bits, limbs, kchunks, nw, R, npad;
    uint32_t ncols;         // tensor-memory columns allocated
};

template <bool INT8>
__device__ __forceinline__ uint32_t field_bits(long long acc, int S)
{
    if constexpr (INT8) return (uint32_t)(int32_t)acc;
    else return __float_as_uint(scaled_f32_of(acc, S));
}

template <bool INT8>
__global__ void __launch_bounds__(kThreads, kMinBlocks) recompute_tc_kernel(const __grid_constant__ TcParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_fail;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int i0 = blockIdx.x * kBN;
    const int m = (warp & 3) * 32 + lane;           // TMEM lane = state of the tile
    const int cg = warp >> 2;                       // 16-column group of the epilogue
    const int r = blockIdx.y * kBM + m;

    if (i0 >= p.N) {   // padding beyond N (whole block): zero fields and partial sums
        if (cg == 0 && r < p.R) {
            if (p.hout)
                for (int e = 0; e < kBN; ++e)
                    if (i0 + e < p.npad) static_cast<uint32_t*>(p.hout)[(size_t)r * p.npad + i0 + e] = 0u;
            if (p.part) p.part[(size_t)blockIdx.x * p.R + r] = I128{0ull, 0ll};
        }
        return;
    }

    const uint32_t stage_bytes = kATile + (uint32_t)p.limbs * kBTile;
    uint8_t* sm = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + kStages * stage_bytes);
    uint64_t* empty = full + kStages;
    uint64_t* done = empty + kStages;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&full[s], 1 + kExpanders);   // the copier's expect_tx and every expander
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(done, 1);
        tc::mbar_init_fence();
        s_fail = 0;
    }
    if (warp == 0) {
        tc::tmem_alloc(tslot, p.ncols);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = *tslot;
    const int nk = p.kchunks;

    if (warp == 0) {
        // bulk-copy issuers: the digit planes of each stage, a piece of kPiece bytes per lane
        const __half* b_src = p.B + (size_t)blockIdx.x * nk * p.limbs * (kBN * kBK);
        const uint32_t b_bytes = (uint32_t)p.limbs * kBTile;
        for (int c = 0; c < nk; ++c) {
            const int s = c % kStages;
            const uint32_t u = (uint32_t)(c / kStages);
            bool ok = true;
            if (lane == 0) {
                ok = u == 0 || tc::mbar_wait(&empty[s], (u - 1) & 1u, kWaitLimit, kWaitNs);
                if (ok) tc::mbar_arrive_expect_tx(&full[s], b_bytes);
                else s_fail = 1;
            }
            if (!__all_sync(0xffffffffu, ok)) break;
            const uint8_t* src = reinterpret_cast<const uint8_t*>(b_src + (size_t)c * p.limbs * (kBN * kBK));
            uint8_t* st = sm + s * stage_bytes + kATile;
            for (uint32_t o = lane * kPiece; o < b_bytes; o += 32 * kPiece)
                tc::bulk_g2s(st + o, src + o, kPiece, &full[s]);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {   // MMA issuer
            // the digit planes side by side as the N side of one MMA (two halves above 256
            // columns): the accumulator of plane l starts at column 64 l
            const int parts = p.limbs > 4 ? 2 : 1;
            const int cols = kBN * p.limbs / parts;      // 64 .. 256, a multiple of 16
            const uint32_t kstride = (uint32_t)(kBN * p.limbs / 8) * 128;   // between core-matrix columns
            const uint32_t idesc = tc::idesc_f16_f32(kBM, cols);
            for (int c = 0; c < nk; ++c) {
                const int s = c % kStages;
                const uint32_t u = (uint32_t)(c / kStages);
                if (!tc::mbar_wait(&full[s], u & 1u, kWaitLimit, kWaitNs)) {
                    s_fail = 1;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t a0 = tc::smem_u32(sm + s * stage_bytes);
                const uint32_t b0 = a0 + kATile;
#pragma unroll
                for (int q = 0; q < kBK / 16; ++q) {
                    // K-step q covers core-matrix columns 2q, 2q + 1 of the stage
                    const uint64_t ad = tc::smem_desc(a0 + q * 2 * (kBM / 8) * 128, (kBM / 8) * 128, 128);
                    for (int h = 0; h < parts; ++h) {
                        const uint64_t bd = tc::smem_desc(b0 + q * 2 * kstride + (uint32_t)(h * cols / 8) * 128, kstride, 128);
                        tc::mma_f16(tbase + (uint32_t)(h * cols), ad, bd, idesc, (c > 0 || q > 0) ? 1u : 0u);
                    }
                }
                tc::mma_commit(&empty[s]);
            }
            tc::mma_commit(done);
        }
        __syncwarp();
    } else if (warp < 2 + kExpanders / 32) {
        // the stage's state tile: thread e writes half hh = e / 128 of state e % 128, 32
        // couplings (one state word) as four 16-byte rows of f16 {0, 1} in the canonical
        // K-major layout; bits beyond N and states beyond R are 0
        const int e = (int)threadIdx.x - 64;
        const int row = e & (kBM - 1), hh = e / kBM;
        const int rs = blockIdx.y * kBM + row;
        const uint32_t* xr = p.xs + (size_t)rs * p.nw;
        // the word of chunk c: loaded one chunk ahead, so that its latency overlaps the
        // wait for the stage and the writes of the chunk before
        auto load = [&](int c) {
            const int w = 2 * c + hh;
            return rs < p.R && w < p.nw ? xr[w] : 0u;
        };
        uint32_t cur = load(0), nxt = 0u;
        for (int c = 0; c < nk; ++c) {
            const int s = c % kStages;
            const uint32_t u = (uint32_t)(c / kStages);
            if (c + 1 < nk) nxt = load(c + 1);
            if (u > 0 && !tc::mbar_wait(&empty[s], (u - 1) & 1u, kWaitLimit, kWaitNs)) {
                s_fail = 1;
                break;
            }
            uint8_t* st = sm + s * stage_bytes;
            const int nvalid = p.N - c * kBK - 32 * hh;
            const uint32_t bits = nvalid >= 32 ? cur : nvalid <= 0 ? 0u : cur & ((1u << nvalid) - 1u);
#pragma unroll
            for (int kc = 0; kc < 4; ++kc) {
                const uint32_t b = (bits >> (8 * kc)) & 0xFFu;
                const uint4 v = make_uint4(half_pair(b & 3u), half_pair((b >> 2) & 3u), half_pair((b >> 4) & 3u),
                                           half_pair(b >> 6));
                *reinterpret_cast<uint4*>(st + 2 * core_offset(kBM, row, 32 * hh + 8 * kc)) = v;
            }
            cur = nxt;
            fence_proxy_async_smem();
            tc::mbar_arrive(&full[s]);
        }
    }

    // epilogue: state r = TMEM lane m, variables i0 + 16 cg .. + 15
    if (!tc::mbar_wait(done, 0, kWaitLimit, kWaitNs)) s_fail = 1;
    __syncwarp();
    tc::fence_after_sync();
    const uint32_t lane_addr = tbase + ((uint32_t)((warp & 3) * 32) << 16);
    I128 esum{0ull, 0ll};
    const bool live = r < p.R;
    const bool vec = (p.npad & 3) == 0;
    uint32_t* hrow = p.hout ? static_cast<uint32_t*>(p.hout) + (size_t)r * p.npad : nullptr;
    {
        const int ib = i0 + cg * 16;
        long long acc[16];
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
            const longlong2 d2 = *reinterpret_cast<const longlong2*>(p.dfix + ib + e);
            acc[e] = d2.x;
            acc[e + 1] = d2.y;
        }
        for (int l = 0; l < p.limbs; ++l) {
            uint32_t v[16];
            tc::tmem_ld16(lane_addr + (uint32_t)(l * kBN + cg * 16), v);
            const int sh = p.bits * l;
#pragma unroll
            for (int e = 0; e < 16; ++e)
                acc[e] = (long long)((unsigned long long)acc[e] +
                                     ((unsigned long long)(long long)small_int_of(__uint_as_float(v[e])) << sh));
        }
        if (live) {
            if (hrow) {
                uint32_t hb[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) hb[e] = field_bits<INT8>(acc[e], p.S);  // 0 for i >= N
                if (vec && ib + 16 <= p.npad) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        *reinterpret_cast<uint4*>(hrow + ib + 4 * q) =
                            make_uint4(hb[4 * q], hb[4 * q + 1], hb[4 * q + 2], hb[4 * q + 3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (ib + e < p.npad) hrow[ib + e] = hb[e];
                }
            }
            if (p.part && ib < p.N) {
                const uint32_t xw = (p.xs[(size_t)r * p.nw + (ib >> 5)] >> (ib & 31)) & 0xFFFFu;
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    if ((xw >> e) & 1u) i128_add(esum, p.dfix[ib + e] + acc[e]);
            }
        }
    }
    // partial energies of the four column groups, in the first stage's memory: every bulk
    // copy has landed and every MMA has read its operands once `done` has completed
    I128 (*s_part)[kBM] = reinterpret_cast<I128 (*)[kBM]>(sm);
    s_part[cg][m] = esum;

    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tbase, p.ncols);
    }
    if (threadIdx.x < kBM && p.part && blockIdx.y * kBM + threadIdx.x < p.R) {
        I128 t = s_part[0][threadIdx.x];
#pragma unroll
        for (int g = 1; g < kThreads / kBM; ++g) {
            i128_add2(t, s_part[g][threadIdx.x]);
        }
        p.part[(size_t)blockIdx.x * p.R + blockIdx.y * kBM + threadIdx.x] = t;
    }
    if (threadIdx.x == 0 && s_fail) atomicExch(p.err, 1);

    // The energies of the tile's states, by the last of its blocks: a launch of their own
    // takes 5 us beside the 16 us of this one (N = 1024, 128 states).
    if (p.arrived) {
        __shared__ int s_last;
        __threadfence();                                   // the partial sums, before the arrival
        __syncthreads();
        const int tiles = (p.N + kBN - 1) / kBN;           // the blocks that come here
        if (threadIdx.x == 0) s_last = atomicAdd(&p.arrived[blockIdx.y], 1u) == (unsigned)tiles - 1u;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if (threadIdx.x == 0) p.arrived[blockIdx.y] = 0u;
        I128 t{0ull, 0ll};
        if (live)
            for (int b = cg; b < tiles; b += kThreads / kBM) {
                const I128 u = load_partial(&p.part[(size_t)b * p.R + r]);
                i128_add2(t, u);
            }
        s_part[cg][m] = t;
        __syncthreads();
        if (cg == 0 && live) {
#pragma unroll
            for (int g = 1; g < kThreads / kBM; ++g) i128_add2(t, s_part[g][m]);
            p.E[(size_t)r * p.Estride] = energy_of_sum<INT8>(t.lo, t.hi, p.S);
            if (p.check) p.check[(size_t)r * p.Estride * 2] = 1u;
        }
    }
}

size_t smem_bytes(int limbs) { return 1024 + (size_t)kStages * (kATile + (size_t)limbs * kBTile) + 8 * (2 * kStages + 1) + 16; }

int ceil_log2(long long n)
{
    int L = 0;
    while ((1ll << L) < n) ++L;
    return L;
}

}  // namespace

void tc_digits(int wtype, int N, int* bits, int* limbs)
{
    if (wtype == kWInt8) {   // the couplings are balanced 8-bit digits already
        *bits = 8;
        *limbs = 1;
        return;
    }
    // -2^22 <= partial sum < 2^22 (digits -2^(b-1) .. 2^(b-1) - 1), the range of small_int_of.
    // At half of it N = 4096 and 8192 need a sixth plane: 805 instead of 671 MB to stream at
    // N = 8192.
    const int b = std::min(12, 23 - ceil_log2(std::max(N, 2)));
    *bits = b;
    if (wtype == kWInt16) {  // |v| <= 2^15 - 1 needs b * limbs >= 17
        *limbs = (17 + b - 1) / b;
        return;
    }
    // |v| <= 2^(62 - L), 2^L >= N + 1
    const int L = ceil_log2((long long)N + 1);
    *limbs = (64 - L + b - 1) / b;
}

size_t tc_partial_bytes(int rows, int R)
{
    return (size_t)16 * (size_t)((rows + kBN - 1) / kBN) * (size_t)R;
}

// Bytes of the operand's three parts: digit planes, fixed-point diagonal, error flag.
static void tc_operand_parts(int wtype, int N, size_t* b_bytes, size_t* d_bytes)
{
    int bits = 0, limbs = 0;
    tc_digits(wtype, N, &bits, &limbs);
    const size_t kchunks = (size_t)(N + kBK - 1) / kBK;
    const size_t itiles = (size_t)(N + kBN - 1) / kBN;
    *b_bytes = itiles * kchunks * (size_t)limbs * kBTile;
    *d_bytes = kchunks * kBK * sizeof(long long);
}

size_t tc_operand_bytes(int wtype, int N)
{
    size_t b = 0, d = 0;
    tc_operand_parts(wtype, N, &b, &d);
    return (b + 255) / 256 * 256 + (d + 255) / 256 * 256 + 256;
}

static cudaError_t tc_operand_fill(int wtype, const void* W, const void* diag, int N, int ldw, int S, TcOperand* op,
                                   cudaStream_t st);

cudaError_t tc_operand_build_in(int wtype, const void* W, const void* diag, int N, int ldw, int S, void* mem,
                                TcOperand* op, cudaStream_t st)
{
    size_t b = 0, d = 0;
    tc_operand_parts(wtype, N, &b, &d);
    char* m = static_cast<char*>(mem);
    op->B = m;
    op->dfix = reinterpret_cast<long long*>(m + (b + 255) / 256 * 256);
    op->err = reinterpret_cast<int*>(m + (b + 255) / 256 * 256 + (d + 255) / 256 * 256);
    return tc_operand_fill(wtype, W, diag, N, ldw, S, op, st);
}

cudaError_t tc_operand_build(int wtype, const void* W, const void* diag, int N, int ldw, int S, TcOperand* op,
                             cudaStream_t st)
{
    size_t b = 0, d = 0;
    tc_operand_parts(wtype, N, &b, &d);
    cudaError_t e = dev_malloc(&op->B, b);
    if (e == cudaSuccess) e = dev_malloc(reinterpret_cast<void**>(&op->err), sizeof(int));
    if (e == cudaSuccess) e = dev_malloc(reinterpret_cast<void**>(&op->dfix), d);
    if (e != cudaSuccess) return e;
    return tc_operand_fill(wtype, W, diag, N, ldw, S, op, st);
}

// The digit planes and diagonal of W into op's buffers, and the error flag cleared.
static cudaError_t tc_operand_fill(int wtype, const void* W, const void* diag, int N, int ldw, int S, TcOperand* op,
                                   cudaStream_t st)
{
    tc_digits(wtype, N, &op->bits, &op->limbs);
    op->kchunks = (N + kBK - 1) / kBK;
    const int itiles = (N + kBN - 1) / kBN;
    cudaError_t e;
    e = cudaMemsetAsync(op->err, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    const long long total = (long long)itiles * op->kchunks * kBN * 8;
    const int tb = 256;
    const unsigned blocks = (unsigned)((total + tb - 1) / tb);
    const int nd = op->kchunks * kBK;
    __half* B = static_cast<__half*>(op->B);
    // the request loop builds operands beside running kernels: the carveout of the rest of its kernels
    prefer_shared<build_digits_kernel<int8_t>>();
    prefer_shared<build_digits_kernel<int16_t>>();
    prefer_shared<build_digits_kernel<float>>();
    prefer_shared<build_dfix_kernel<false>>();
    prefer_shared<build_dfix_kernel<true>>();
    if (wtype == kWInt8)
        build_digits_kernel<int8_t><<<blocks, tb, 0, st>>>(W, N, ldw, S, op->bits, op->limbs, op->kchunks, B, total);
    else if (wtype == kWInt16)
        build_digits_kernel<int16_t><<<blocks, tb, 0, st>>>(W, N, ldw, S, op->bits, op->limbs, op->kchunks, B, total);
    else
        build_digits_kernel<float><<<blocks, tb, 0, st>>>(W, N, ldw, S, op->bits, op->limbs, op->kchunks, B, total);
    if (wtype == kWFp32)
        build_dfix_kernel<false><<<(nd + tb - 1) / tb, tb, 0, st>>>(diag, N, S, op->dfix, nd);
    else
        build_dfix_kernel<true><<<(nd + tb - 1) / tb, tb, 0, st>>>(diag, N, S, op->dfix, nd);
    return cudaGetLastError();
}

void tc_operand_free(TcOperand* op)
{
    if (op->B) dev_free(op->B);
    if (op->err) dev_free(op->err);
    if (op->dfix) dev_free(op->dfix);
    *op = TcOperand{};
}

cudaError_t prepare_tc_kernels()
{
    prefer_shared<build_digits_kernel<int8_t>>();
    prefer_shared<build_digits_kernel<int16_t>>();
    prefer_shared<build_digits_kernel<float>>();
    prefer_shared<build_dfix_kernel<false>>();
    prefer_shared<build_dfix_kernel<true>>();
    prefer_shared<recompute_tc_kernel<false>>();
    prefer_shared<recompute_tc_kernel<true>>();
    cudaError_t e = cudaFuncSetAttribute(recompute_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem_bytes(kMaxLimbs));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(recompute_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem_bytes(2));
    return e;
}

cudaError_t launch_recompute_tc(bool is_int8, const TcOperand& op, const void* diag, int N, int S,
                                const uint32_t* xs, int nw, int R, void* hout, int npad, long long* E, int Estride,
                                cudaStream_t st, long long* scratch, unsigned* arrived, uint32_t* check)
{
    if (R <= 0) return cudaSuccess;
    // the dynamic shared-memory limit of each kernel form, set once per device
    static std::mutex attr_mu;
    static std::set<std::pair<int, int>> attr_done;
    int dev = 0;
    cudaGetDevice(&dev);
    const size_t smem = smem_bytes(op.limbs);
    const int max_limbs = is_int8 ? 2 : kMaxLimbs;   // integer couplings: 1 (int8) or 2 (int16) planes
    if (op.limbs < 1 || op.limbs > max_limbs) return cudaErrorInvalidValue;
    {
        std::lock_guard<std::mutex> lock(attr_mu);
        if (!attr_done.count({is_int8 ? 1 : 0, dev})) {
            const int bytes = (int)smem_bytes(max_limbs);
            cudaError_t e = is_int8 ? cudaFuncSetAttribute(recompute_tc_kernel<true>,
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)
                                    : cudaFuncSetAttribute(recompute_tc_kernel<false>,
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
            if (e != cudaSuccess) return e;
            attr_done.insert({is_int8 ? 1 : 0, dev});
        }
    }

    const int rtiles = (R + kBM - 1) / kBM;
    const int rows = hout ? std::max(npad, N) : N;
    const int itiles = (rows + kBN - 1) / kBN;
    TcParams p;
    p.B = static_cast<const __half*>(op.B);
    p.dfix = op.dfix;
    p.xs = xs;
    p.hout = hout;
    p.part = E ? reinterpret_cast<I128*>(scratch) : nullptr;
    p.arrived = E ? arrived : nullptr;
    p.E = E;
    p.Estride = Estride;
    p.check = check;
    p.err = op.err;
    p.N = N;
    p.S = S;
    p.bits = op.bits;
    p.limbs = op.limbs;
    p.kchunks = op.kchunks;
    p.nw = nw;
    p.R = R;
    p.npad = npad;
    uint32_t nc = 32;
    while (nc < (uint32_t)(op.limbs * kBN)) nc <<= 1;
    p.ncols = nc;
    dim3 grid(itiles, rtiles);
    if (is_int8)
        recompute_tc_kernel<true><<<grid, kThreads, smem, st>>>(p);
    else
        recompute_tc_kernel<false><<<grid, kThreads, smem, st>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !E || arrived) return e;
    return launch_energy_sum(is_int8, scratch, itiles, R, S, E, Estride, st, check);
}

}  // namespace da
