// RIB window attention for windows of 8 x 8 tokens on B200 (sm_100a), forward and backward: tcgen05 MMAs, TMEM, TMA loads and stores.
//
// At n = 64 keys per row the passes are bound by memory traffic: per token-head the forward moves 256 bytes and computes
// 64 * (2 d + r) products, so a tile of 128 tokens has 1420 cycles at the measured copy bandwidth and needs 512 of the exp
// pipe and about 550 of the tensor pipe; the backward has 2840 cycles per tile and needs 512 and about 1400.  Hence: every
// input is read once and every output written once, nothing goes through accumulators in global memory, and several tiles are
// under way per SM.  Measured (16 x 96 x 96 tokens, 6 heads of 32 channels, rank 16, by event hooks, which include some us per
// launch): forward 45 us, backward 6 (clearing) + 83 us for 226 and 456 MB; the two calls together 141 us.  (Before: 125
// us, 56 + 311 + 80 us and 582 us; these windows ran four at a time as 16 x 16 windows of the general kernels with three quarters of
// every score tile discarded; the backward added dq in global memory and needed a preparation and a finishing kernel.)
//
// Tile = two horizontally adjacent windows of one head, 64 rows each (one 8x8-token patch, one TMA box).  A CTA keeps to one
// head: CTA c works on head c mod heads and on every (grid / heads)-th tile of it, neighbouring CTAs on the other heads of
// the same tokens (which share their 128-byte lines).  The RIB rows of a head are therefore staged once per CTA, and the
// gradients of its tables are summed in tensor memory over all tiles of the CTA.
//
// A score tile is computed 128 x 128 although only its two diagonal 64 x 64 blocks are meant (an M128 N128 MMA costs what
// two M64 N64 would); rows read their own block, and the other block of P (dS) is zero wherever it is contracted.
#include "rib_small_window.cuh"

namespace rib {
namespace {

using namespace sm100;

struct Win8Tile { int b, Y0, X0; };      // first token of the left window

__device__ __forceinline__ Win8Tile decode_tile(const SmallWindowParams& p, int tile)
{
    Win8Tile t;
    int y, x;
    p.by_nx.divmod(tile, tile, x);
    p.by_ny.divmod(tile, t.b, y);
    t.Y0 = 8 * y; t.X0 = 16 * x;
    return t;
}

constexpr uint64_t kDesc64 = smem_desc_const(16, 512, kSwizzle64B);
constexpr uint32_t kIdescS8 = idesc_bf16_f32(kTile, kTile, false);            // both operands K-major
constexpr uint32_t kIdescPV8 = idesc_bf16_f32(kTile, kD, true);               // A in TMEM, B MN-major

// ================================================================================================ forward
// Roles (640 threads): warp 0 TMA loads, warp 1 issues S, warp 2 PV (and owns the TMEM allocation), warp 3 TMA stores of the
// output; warps 4-19 are four groups of four softmax warps, one thread per row, group g on tiles g, g + 4, ....  Each group
// has 128 columns of tensor memory: S; then P over its columns 0-63 and O in columns 64-95, once the scores are in registers.
// The output rows go through the shared memory of the tile's own q rows.
namespace fwd8 {
constexpr int kThreads = 640, kGroups = 4, kStages = 8;
constexpr uint32_t kStageBytes = 3 * kContentBytes;                           // q, k, v
constexpr uint32_t kOffRib = kStages * kStageBytes;                           // query RIB rows, key RIB rows
constexpr uint32_t kOffBar = kOffRib + 2 * kContentBytes;
enum Bar { kFull = 0, kEmpty = kFull + kStages, kStore = kEmpty + kStages, kSFull = kStore + kStages, kPReady = kSFull + kGroups,
           kOFull = kPReady + kGroups, kTFree = kOFull + kGroups, kDrain = kTFree + kGroups, kNumBars = kDrain + 2 };
constexpr uint32_t kOffMisc = kOffBar + kNumBars * 8;
constexpr uint32_t kSmemBytes = kOffMisc + 16 + 1024;
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");

template <int R>
__global__ void __launch_bounds__(kThreads, 1)
rib_window8_fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                       const __grid_constant__ CUtensorMap tm_out, const __grid_constant__ SmallWindowParams p)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    auto bar = [&](int i) { return base + kOffBar + 8u * i; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + kOffMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + kOffMisc + 4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int group0, head;
    p.by_heads.divmod((int)blockIdx.x, group0, head);
    const int count = (p.tiles - group0 + p.groups - 1) / p.groups;           // tiles of this CTA: group0 + t * groups

    if (threadIdx.x == 0) {
        abort_flag[0] = 0; abort_flag[1] = 0;   // [1] stays 0: used by the drain waits
        for (int s = 0; s < kStages; ++s) { mbar_init(bar(kFull + s), 1); mbar_init(bar(kEmpty + s), 1); mbar_init(bar(kStore + s), 4); }
        for (int g = 0; g < kGroups; ++g) {
            mbar_init(bar(kSFull + g), 1); mbar_init(bar(kPReady + g), 4); mbar_init(bar(kOFull + g), 1); mbar_init(bar(kTFree + g), 4);
        }
        mbar_init(bar(kDrain), 1); mbar_init(bar(kDrain + 1), 1);
        fence_barrier_init();
        prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v); prefetch_tensormap(&tm_out);
    }
    if (warp == 2) {
        tmem_alloc(base + kOffMisc, 512);
        tmem_relinquish();
    }
    if (warp >= 4 && warp < 8) {
        const int row = (int)threadIdx.x - 128;             // the 64 rows of the tables twice
        stage_rib_row(p, head, row & 63, base_ptr + kOffRib, base_ptr + kOffRib + kContentBytes, row);
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int t = 0;
            bool ok = true;
            for (; t < count; ++t) {
                const int st = t % kStages, use = t / kStages;
                if (use > 0 && !mbar_wait(bar(kEmpty + st), (use - 1) & 1, abort_flag, p.status)) { ok = false; break; }
                const Win8Tile c = decode_tile(p, group0 + t * p.groups);
                mbar_arrive_expect_tx(bar(kFull + st), kStageBytes);
                const uint32_t dst = base + st * kStageBytes;
                for (int sub = 0; sub < 2; ++sub) {
                    tma_load_5d(dst + sub * kPatchContent, &tm_q, bar(kFull + st), 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                    tma_load_5d(dst + kContentBytes + sub * kPatchContent, &tm_k, bar(kFull + st), 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                    tma_load_5d(dst + 2 * kContentBytes + sub * kPatchContent, &tm_v, bar(kFull + st), 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                }
            }
            if (!ok)                            // gave up: let the copies already in flight land before the CTA may exit
                for (int b2 = t > kStages ? t - kStages : 0; b2 < t; ++b2)
                    mbar_wait(bar(kFull + b2 % kStages), (b2 / kStages) & 1, abort_flag + 1, p.status);
        }
    } else if (warp == 1) {
        // ---- S = Q~ K~^T; the whole warp walks the loop and waits, one elected lane issues
        const uint64_t qp = smem_desc_at(kDesc64, base + kOffRib), kp = smem_desc_at(kDesc64, base + kOffRib + kContentBytes);
        for (int t = 0; t < count; ++t) {
            const int st = t % kStages, g = t % kGroups;
            if (!mbar_wait_warp(bar(kFull + st), (t / kStages) & 1, abort_flag, p.status) ||
                !(t < kGroups || mbar_wait_warp(bar(kTFree + g), (t / kGroups - 1) & 1, abort_flag, p.status))) break;
            tc_fence_after();
            if (elect_one()) {
                const uint64_t q = smem_desc_at(kDesc64, base + st * kStageBytes), k = smem_desc_at(kDesc64, base + st * kStageBytes + kContentBytes);
                const uint32_t d = tmem + g * kTile;
                mma_ss(d, q, k, kIdescS8, 0u);
                mma_ss(d, q + 2, k + 2, kIdescS8, 1u);            // + 32 bytes: second K16 step
                mma_ss(d, qp, kp, kIdescS8, 1u);
                if (R == 32) mma_ss(d, qp + 2, kp + 2, kIdescS8, 1u);
                mma_commit(bar(kSFull + g));
            }
            __syncwarp();
        }
        if (elect_one()) mma_commit(bar(kDrain));
        __syncwarp();
        mbar_wait(bar(kDrain), 0, abort_flag + 1, p.status);
    } else if (warp == 2) {
        // ---- O = P V
        for (int t = 0; t < count; ++t) {
            const int st = t % kStages, g = t % kGroups;
            if (!mbar_wait_warp(bar(kPReady + g), (t / kGroups) & 1, abort_flag, p.status)) break;
            tc_fence_after();
            if (elect_one()) {
                const uint64_t v = smem_desc_at(kDesc64, base + st * kStageBytes + 2 * kContentBytes);
                const uint32_t a = tmem + g * kTile;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ts(a + 64, a + 8 * kk, v + 64 * kk, kIdescPV8, kk ? 1u : 0u);
                mma_commit(bar(kOFull + g));
            }
            __syncwarp();
        }
        if (elect_one()) mma_commit(bar(kDrain + 1));
        __syncwarp();
        mbar_wait(bar(kDrain + 1), 0, abort_flag + 1, p.status);
    } else if (warp == 3) {
        // ---- output rows to global memory; the stage is free once its rows have been read
        if (lane == 0) {
            for (int t = 0; t < count; ++t) {
                const int st = t % kStages;
                if (!mbar_wait(bar(kStore + st), (t / kStages) & 1, abort_flag, p.status)) break;
                const Win8Tile c = decode_tile(p, group0 + t * p.groups);
                for (int sub = 0; sub < 2; ++sub)
                    tma_store_5d(&tm_out, base + st * kStageBytes + sub * kPatchContent, 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                bulk_commit_group();
                bulk_wait_group_read<0>();
                mbar_arrive(bar(kEmpty + st));
            }
            bulk_wait_group<0>();
        }
    } else {
        const int g = (warp - 4) >> 2, quarter = warp & 3, row = quarter * 32 + lane;
        const uint32_t t0 = tmem + ((uint32_t)(quarter * 32) << 16) + g * kTile;
        const int own = row >> 6;                                 // left or right window: score columns 64 own .., P columns 32 own ..
        const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
        uint32_t zero[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) zero[e] = 0u;
        for (int t = g; t < count; t += kGroups) {
            const int st = t % kStages;
            const uint32_t phase = (t / kGroups) & 1;
            if (!mbar_wait_warp(bar(kSFull + g), phase, abort_flag, p.status)) break;
            tc_fence_after();
            uint32_t s[2][32];
            tmem_ld32(t0 + 64 * own, s[0]);
            tmem_ld32(t0 + 64 * own + 32, s[1]);
            tmem_wait_ld();
            float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
                mx0 = max3(mx0, __uint_as_float(s[0][e]), __uint_as_float(s[0][e + 1]));
                mx1 = max3(mx1, __uint_as_float(s[1][e]), __uint_as_float(s[1][e + 1]));
            }
            const float mx = fmaxf(mx0, mx1), neg = -mx * p.scale_log2;
            const float2 neg2 = make_float2(neg, neg);
            // the output is normalised by the sum of the rounded probabilities, which are what meets V; lse takes the unrounded ones
            float2 sum = make_float2(0.f, 0.f), rounded = make_float2(0.f, 0.f);
#pragma unroll
            for (int ch = 0; ch < 2; ++ch) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[ch][2 * i]), __uint_as_float(s[ch][2 * i + 1])), scale2, neg2);
                    const float2 e = make_float2(ex2_approx(x.x), ex2_approx(x.y));
                    sum = __fadd2_rn(sum, e);
                    pk[i] = pack_bf16x2(e.x, e.y);
                    rounded = __fadd2_rn(rounded, make_float2(__uint_as_float(pk[i] << 16), __uint_as_float(pk[i] & 0xffff0000u)));
                }
                tmem_st16(t0 + 32 * own + 16 * ch, pk);
            }
            tmem_st32(t0 + 32 * (own ^ 1), zero);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kPReady + g));
            const Win8Tile c = decode_tile(p, group0 + t * p.groups);
            if (p.lse) {
                const int Y = c.Y0 + ((row >> 3) & 7), X = c.X0 + 8 * own + (row & 7);
                p.lse[(((size_t)c.b * p.heads + head) * p.H + Y) * p.W + X] = mx * p.inv_sqrt_d + logf(sum.x + sum.y);
            }
            if (!mbar_wait_warp(bar(kOFull + g), phase, abort_flag, p.status)) break;
            tc_fence_after();
            tmem_ld32(t0 + 64, s[0]);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kTFree + g));
            write_row(base_ptr + st * kStageBytes, row, s[0], 1.f / (rounded.x + rounded.y));
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kStore + st));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}
}  // namespace fwd8

// ================================================================================================ backward
// Per tile (rows = queries):  S = Q~ K~^T, dP = dO V^T;  P = exp2(S log2e/sqrt(d) - lse log2e), dS = P o (dP - D), D = rowsum(dO o O)
// from the rows in shared memory;  dV = P^T dO, dK~ = dS^T Q~, dQ~ = dS K~.  P and dS go to shared memory as rows of their own
// window's 64 keys and are contracted as MN-major A operands: for the 16 queries of a step the atom of the other window's
// keys is a block of zeros (one below the two tiles and one above, the distance between the atoms being non-negative).  dS goes
// to tensor memory as well, for dQ~, where the other window's columns stay zero.  The content columns of dQ~, dK~ are
// cleared when they have been read, so that every MMA accumulates and the RIB columns (the gradients of the tables) add up
// over the tiles of the CTA.
//
// Roles (512 threads): warp 0 TMA loads; warp 1 issues S and dP, warp 3 dV, dK~ and dQ~; warp 2 owns the TMEM allocation; warps
// 4-11 P and dS (two threads per query row, 32 keys each); warps 12-15 move the gradients out (through the shared memory of
// the tile's own q, k, v rows and TMA stores) and add the table gradients to global memory at the end.
namespace bwd8 {
constexpr int kThreads = 512, kStages = 4;
constexpr uint32_t kQ = 0, kK = kContentBytes, kV = 2 * kContentBytes, kDO = 3 * kContentBytes, kO = 4 * kContentBytes, kStageBytes = 5 * kContentBytes;
constexpr uint32_t kOffRib = kStages * kStageBytes;                           // query RIB rows, key RIB rows
constexpr uint32_t kZeroBytes = 2048;                                         // 16 query rows x 64 keys
constexpr uint32_t kOffZeroLo = kOffRib + 2 * kContentBytes;
constexpr uint32_t kOffP = kOffZeroLo + kZeroBytes;                           // [128 queries][64 keys], 128-byte rows, SWIZZLE_128B
constexpr uint32_t kOffDS = kOffP + kTile * 128;
constexpr uint32_t kOffZeroHi = kOffDS + kTile * 128;
constexpr uint32_t kOffBar = kOffZeroHi + kZeroBytes;
enum Bar { kFull = 0, kEmpty = kFull + kStages, kSFull = kEmpty + kStages, kSFree, kReady, kDone, kDFree, kDrain, kNumBars = kDrain + 2 };
constexpr uint32_t kOffMisc = kOffBar + kNumBars * 8;
constexpr uint32_t kSmemBytes = kOffMisc + 16 + 1024;
static_assert(kOffZeroLo % 1024 == 0 && kOffP % 1024 == 0 && kSmemBytes <= 232448, "shared memory of one CTA");

// tensor memory
constexpr uint32_t kColS = 0, kColDP = 128, kColDS = 256, kColDV = 320, kColDK = 352;
template <int R> constexpr uint32_t kColDQ = kColDK + kD + R;

template <int R>
__global__ void __launch_bounds__(kThreads, 1)
rib_window8_bwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                       const __grid_constant__ CUtensorMap tm_do, const __grid_constant__ CUtensorMap tm_o, const __grid_constant__ CUtensorMap tm_dq,
                       const __grid_constant__ CUtensorMap tm_dk, const __grid_constant__ CUtensorMap tm_dv, const __grid_constant__ SmallWindowParams p)
{
    constexpr uint32_t kIdescGrad = idesc_bf16_f32_ab(kTile, kD + R, false, true);       // dQ~: A in TMEM
    constexpr uint32_t kIdescGradT = idesc_bf16_f32_ab(kTile, kD + R, true, true);       // dK~: A MN-major
    constexpr uint32_t kIdescDV = idesc_bf16_f32_ab(kTile, kD, true, true);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    auto bar = [&](int i) { return base + kOffBar + 8u * i; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + kOffMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + kOffMisc + 4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int group0, head;
    p.by_heads.divmod((int)blockIdx.x, group0, head);
    const int count = (p.tiles - group0 + p.groups - 1) / p.groups;

    if (threadIdx.x == 0) {
        abort_flag[0] = 0; abort_flag[1] = 0;   // [1] stays 0: used by the drain waits
        for (int s = 0; s < kStages; ++s) { mbar_init(bar(kFull + s), 1); mbar_init(bar(kEmpty + s), 1); }
        mbar_init(bar(kSFull), 1); mbar_init(bar(kSFree), 8); mbar_init(bar(kReady), 8); mbar_init(bar(kDone), 1); mbar_init(bar(kDFree), 4);
        mbar_init(bar(kDrain), 1); mbar_init(bar(kDrain + 1), 1);
        fence_barrier_init();
        prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v); prefetch_tensormap(&tm_do); prefetch_tensormap(&tm_o);
        prefetch_tensormap(&tm_dq); prefetch_tensormap(&tm_dk); prefetch_tensormap(&tm_dv);
    }
    if (warp == 2) {
        tmem_alloc(base + kOffMisc, 512);
        tmem_relinquish();
    }
    if (warp >= 4 && warp < 8) {
        const int t = (int)threadIdx.x - 128;
        stage_rib_row(p, head, t & 63, base_ptr + kOffRib, base_ptr + kOffRib + kContentBytes, t);
        *reinterpret_cast<uint4*>(base_ptr + kOffZeroLo + 16 * t) = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(base_ptr + kOffZeroHi + 16 * t) = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int t = 0;
            bool ok = true;
            for (; t < count; ++t) {
                const int st = t % kStages, use = t / kStages;
                if (use > 0 && !mbar_wait(bar(kEmpty + st), (use - 1) & 1, abort_flag, p.status)) { ok = false; break; }
                const Win8Tile c = decode_tile(p, group0 + t * p.groups);
                mbar_arrive_expect_tx(bar(kFull + st), kStageBytes);
                const uint32_t dst = base + st * kStageBytes;
                for (int sub = 0; sub < 2; ++sub) {
                    const uint32_t at = dst + sub * kPatchContent;
                    tma_load_5d(at + kQ, &tm_q, bar(kFull + st), 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                    tma_load_5d(at + kK, &tm_k, bar(kFull + st), 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                    tma_load_5d(at + kV, &tm_v, bar(kFull + st), 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                    tma_load_5d(at + kDO, &tm_do, bar(kFull + st), 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                    tma_load_5d(at + kO, &tm_o, bar(kFull + st), 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                }
            }
            if (!ok)                            // gave up: let the copies already in flight land before the CTA may exit
                for (int b2 = t > kStages ? t - kStages : 0; b2 < t; ++b2)
                    mbar_wait(bar(kFull + b2 % kStages), (b2 / kStages) & 1, abort_flag + 1, p.status);
        }
    } else if (warp == 1) {
        // ---- S and dP of tile t once the arithmetic warps hold those of tile t - 1 in registers
        const uint64_t qp = smem_desc_at(kDesc64, base + kOffRib), kp = smem_desc_at(kDesc64, base + kOffRib + kContentBytes);
        for (int t = 0; t < count; ++t) {
            const int st = t % kStages;
            if (!mbar_wait_warp(bar(kFull + st), (t / kStages) & 1, abort_flag, p.status) ||
                !(t == 0 || mbar_wait_warp(bar(kSFree), (t - 1) & 1, abort_flag, p.status))) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t at = base + st * kStageBytes;
                const uint64_t q = smem_desc_at(kDesc64, at + kQ), k = smem_desc_at(kDesc64, at + kK);
                const uint64_t v = smem_desc_at(kDesc64, at + kV), go = smem_desc_at(kDesc64, at + kDO);
                mma_ss(tmem + kColS, q, k, kIdescS8, 0u);
                mma_ss(tmem + kColS, q + 2, k + 2, kIdescS8, 1u);
                mma_ss(tmem + kColS, qp, kp, kIdescS8, 1u);
                if (R == 32) mma_ss(tmem + kColS, qp + 2, kp + 2, kIdescS8, 1u);
                mma_ss(tmem + kColDP, go, v, kIdescS8, 0u);
                mma_ss(tmem + kColDP, go + 2, v + 2, kIdescS8, 1u);
                mma_commit(bar(kSFull));
            }
            __syncwarp();
        }
        if (elect_one()) mma_commit(bar(kDrain));
        __syncwarp();
        mbar_wait(bar(kDrain), 0, abort_flag + 1, p.status);
    } else if (warp == 3) {
        // ---- dV, dK~, dQ~ of tile t once P and dS are stored and the accumulators have been read
        for (int t = 0; t < count; ++t) {
            const int st = t % kStages;
            if (!mbar_wait_warp(bar(kReady), t & 1, abort_flag, p.status) || !mbar_wait_warp(bar(kDFree), t & 1, abort_flag, p.status)) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t at = base + st * kStageBytes;
                const uint64_t go = smem_desc_at(kDesc64, at + kDO);
                const uint64_t q = smem_desc(at + kQ, kOffRib - (st * kStageBytes + kQ), 512, kSwizzle64B);                       // [Q | Pq]
                const uint64_t k = smem_desc(at + kK, kOffRib + kContentBytes - (st * kStageBytes + kK), 512, kSwizzle64B);       // [K | Pk]
                // queries 16 kk .. of the left window (kk < 4): atoms (its keys, zeros); of the right window: (zeros, its keys)
                auto a_desc = [&](uint32_t off, int kk) {
                    const uint32_t rows = off + kk * 2048;
                    return kk < 4 ? smem_desc(base + rows, kOffZeroHi - rows, 1024, kSwizzle128B) : smem_desc(base + kOffZeroLo, rows - kOffZeroLo, 1024, kSwizzle128B);
                };
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ss(tmem + kColDV, a_desc(kOffP, kk), go + 64 * kk, kIdescDV, kk ? 1u : 0u);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ss(tmem + kColDK, a_desc(kOffDS, kk), q + 64 * kk, kIdescGradT, 1u);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ts(tmem + kColDQ<R>, tmem + kColDS + 8 * kk, k + 64 * kk, kIdescGrad, 1u);
                mma_commit(bar(kDone));
            }
            __syncwarp();
        }
        if (elect_one()) mma_commit(bar(kDrain + 1));
        __syncwarp();
        mbar_wait(bar(kDrain + 1), 0, abort_flag + 1, p.status);
    } else if (warp >= 4 && warp < 12) {
        // ---- P and dS: thread = (query row, 32 of its window's 64 keys)
        const int quarter = warp & 3, half = (warp - 4) >> 2, row = quarter * 32 + lane, own = row >> 6;
        const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
        const uint32_t t_s = lanes + kColS + 64 * own + 32 * half, t_dp = lanes + kColDP + 64 * own + 32 * half;
        const uint32_t t_ds = lanes + kColDS + 32 * own + 16 * half;
        const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
        uint8_t *p_row = base_ptr + kOffP + row * 128, *ds_row = base_ptr + kOffDS + row * 128;
        {
            uint32_t zero[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) zero[e] = 0u;
            tmem_st16(lanes + kColDS + 32 * (own ^ 1) + 16 * half, zero);      // the other window's columns stay zero
            tmem_wait_st();
        }
        auto lse_at = [&](int t) {
            const Win8Tile c = decode_tile(p, group0 + t * p.groups);
            return p.lse_in[(((size_t)c.b * p.heads + head) * p.H + c.Y0 + ((row >> 3) & 7)) * p.W + c.X0 + 8 * own + (row & 7)];
        };
        float lse = lse_at(0);
        for (int t = 0; t < count; ++t) {
            const int st = t % kStages;
            const float neg_lse = -lse * 1.4426950408889634f;
            if (t + 1 < count) lse = lse_at(t + 1);                            // under way while this tile is worked on
            if (!mbar_wait_warp(bar(kFull + st), (t / kStages) & 1, abort_flag, p.status)) break;
            float neg_d = 0.f;
            {
                const uint8_t *go = base_ptr + st * kStageBytes + kDO + row * 64, *o = base_ptr + st * kStageBytes + kO + row * 64;
#pragma unroll
                for (int ck = 0; ck < 4; ++ck) {
                    const int at = (ck ^ ((row >> 1) & 3)) << 4;
                    const uint4 x = *reinterpret_cast<const uint4*>(go + at), y = *reinterpret_cast<const uint4*>(o + at);
                    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        neg_d = fmaf(-__uint_as_float(xs[e] << 16), __uint_as_float(ys[e] << 16), neg_d);
                        neg_d = fmaf(-__uint_as_float(xs[e] & 0xffff0000u), __uint_as_float(ys[e] & 0xffff0000u), neg_d);
                    }
                }
            }
            if (!mbar_wait_warp(bar(kSFull), t & 1, abort_flag, p.status)) break;
            tc_fence_after();
            uint32_t s[32], dp[32];
            tmem_ld32(t_s, s);
            tmem_ld32(t_dp, dp);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kSFree));
            uint32_t pp[16], dd[16];
            const float2 l2 = make_float2(neg_lse, neg_lse), d2 = make_float2(neg_d, neg_d);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), scale2, l2);
                const float2 e = make_float2(ex2_approx(x.x), ex2_approx(x.y));
                const float2 d = __fmul2_rn(e, __fadd2_rn(make_float2(__uint_as_float(dp[2 * i]), __uint_as_float(dp[2 * i + 1])), d2));
                pp[i] = pack_bf16x2(e.x, e.y);
                dd[i] = pack_bf16x2(d.x, d.y);
            }
            if (t > 0) {                                                       // the contractions of tile t - 1 have read P and dS
                if (!mbar_wait_warp(bar(kDone), (t - 1) & 1, abort_flag, p.status)) break;
                tc_fence_after();
            }
            tmem_st16(t_ds, dd);
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) {
                const int at = ((4 * half + q4) ^ (row & 7)) << 4;
                *reinterpret_cast<uint4*>(p_row + at) = make_uint4(pp[4 * q4], pp[4 * q4 + 1], pp[4 * q4 + 2], pp[4 * q4 + 3]);
                *reinterpret_cast<uint4*>(ds_row + at) = make_uint4(dd[4 * q4], dd[4 * q4 + 1], dd[4 * q4 + 2], dd[4 * q4 + 3]);
            }
            tmem_wait_st();
            tc_fence_before();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kReady));
        }
    } else if (warp >= 12) {
        // ---- gradients out: thread = row of the accumulators
        const int quarter = warp & 3, row = quarter * 32 + lane;
        const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
        uint32_t zero[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) zero[e] = 0u;
        auto clear = [&](uint32_t col) { tmem_st32(lanes + col, zero); };
        clear(kColDK); clear(kColDK + R); clear(kColDQ<R>); clear(kColDQ<R> + R);          // 32 + R columns each
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kDFree));
        bool ok = true;
        for (int t = 0; t < count; ++t) {
            const int st = t % kStages;
            uint8_t* const stage = base_ptr + st * kStageBytes;
            // (the vote of the named barrier below keeps the four warps together)
            ok = mbar_wait_warp(bar(kDone), t & 1, abort_flag, p.status);
            if (ok) {
                tc_fence_after();
                uint32_t a[32], b[32];
                tmem_ld32(lanes + kColDQ<R>, a);
                tmem_ld32(lanes + kColDK, b);
                tmem_wait_ld();
                if (t + 1 < count) { clear(kColDQ<R>); clear(kColDK); }
                write_row(stage + kQ, row, a, p.inv_sqrt_d);
                write_row(stage + kK, row, b, p.inv_sqrt_d);
                tmem_ld32(lanes + kColDV, a);
                tmem_wait_ld();
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kDFree));
                write_row(stage + kV, row, a, 1.f);
                fence_proxy_async();
            }
            if (!named_barrier_and(1, 128, ok)) { ok = false; break; }
            if (warp == 12 && lane == 0) {
                const Win8Tile c = decode_tile(p, group0 + t * p.groups);
                const uint32_t at = base + st * kStageBytes;
                for (int sub = 0; sub < 2; ++sub) {
                    tma_store_5d(&tm_dq, at + kQ + sub * kPatchContent, 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                    tma_store_5d(&tm_dk, at + kK + sub * kPatchContent, 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                    tma_store_5d(&tm_dv, at + kV + sub * kPatchContent, 0, head, c.X0 + 8 * sub, c.Y0, c.b);
                }
                bulk_commit_group();
                bulk_wait_group_read<0>();
                mbar_arrive(bar(kEmpty + st));
            }
            __syncwarp();
        }
        if (ok) {
            // table gradients of this CTA: row of the table = place in the window
            tc_fence_after();
            float *gq = p.dpq + (size_t)head * p.pos_head_stride + (size_t)(row & 63) * p.r, *gk = p.dpk + (size_t)head * p.pos_head_stride + (size_t)(row & 63) * p.r;
#pragma unroll
            for (int part = 0; part < R / 16; ++part) {
                uint32_t a[16], b[16];
                tmem_ld16(lanes + kColDQ<R> + kD + 16 * part, a);
                tmem_ld16(lanes + kColDK + kD + 16 * part, b);
                tmem_wait_ld();
                cudaGridDependencySynchronize();                               // dpq, dpk are cleared
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                    if (16 * part + 4 * q4 >= p.r) break;                      // ranks are multiples of 8
                    add_columns(gq + 16 * part + 4 * q4, a + 4 * q4, p.inv_sqrt_r);
                    add_columns(gk + 16 * part + 4 * q4, b + 4 * q4, p.inv_sqrt_d);      // (the query rows carried sqrt(d / r))
                }
            }
        }
        if (warp == 12 && lane == 0) bulk_wait_group<0>();
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// Clears the tables' gradients (the tables themselves only, not what lies between them); the main kernel overtakes it.
__global__ void __launch_bounds__(256) rib_window8_clear_kernel(float* dpq, float* dpk, int tables, int per_table, long long stride)
{
    cudaTriggerProgrammaticLaunchCompletion();
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < tables * per_table; e += gridDim.x * blockDim.x) {
        const size_t at = (size_t)(e / per_table) * stride + e % per_table;
        dpq[at] = 0.f;
        dpk[at] = 0.f;
    }
}
}  // namespace bwd8

template <int R>
cudaError_t launch_win8_fwd(const Problem& p, cudaStream_t stream)
{
    CUtensorMap tm_q, tm_k, tm_v, tm_out;
    if (!encode_fn()) return cudaErrorNotSupported;
    if (!encode_image_map(&tm_q, p.q, p) || !encode_image_map(&tm_k, p.k, p) || !encode_image_map(&tm_v, p.v, p) || !encode_image_map(&tm_out, p.out_w, p))
        return cudaErrorInvalidValue;
    static KernelSetup setup;       // one per instantiation of this launcher, i.e. per kernel
    int sm_count = 0;
    if (cudaError_t e = setup.prepare(fwd8::rib_window8_fwd_kernel<R>, fwd8::kSmemBytes, &sm_count)) return e;
    SmallWindowParams w{};
    const int grid = fill_small_window(p, sm_count, p.H / 8, p.W / 16, &w);
    w.lse = p.lse_w;
    ProfileScope scope(RIB_KERNEL_WINDOW8_FWD, stream);
    fwd8::rib_window8_fwd_kernel<R><<<grid, fwd8::kThreads, fwd8::kSmemBytes, stream>>>(tm_q, tm_k, tm_v, tm_out, w);
    return cudaGetLastError();
}

template <int R>
cudaError_t launch_win8_bwd(const Problem& p, cudaStream_t stream)
{
    CUtensorMap tm_q, tm_k, tm_v, tm_do, tm_o, tm_dq, tm_dk, tm_dv;
    if (!encode_fn()) return cudaErrorNotSupported;
    if (!encode_image_map(&tm_q, p.q, p) || !encode_image_map(&tm_k, p.k, p) || !encode_image_map(&tm_v, p.v, p) || !encode_image_map(&tm_do, p.dout, p) ||
        !encode_image_map(&tm_o, p.out, p) || !encode_image_map(&tm_dq, p.dq, p) || !encode_image_map(&tm_dk, p.dk, p) || !encode_image_map(&tm_dv, p.dv, p))
        return cudaErrorInvalidValue;
    static KernelSetup setup;
    int sm_count = 0;
    if (cudaError_t e = setup.prepare(bwd8::rib_window8_bwd_kernel<R>, bwd8::kSmemBytes, &sm_count)) return e;
    SmallWindowParams w{};
    const int grid = fill_small_window(p, sm_count, p.H / 8, p.W / 16, &w);
    w.lse_in = p.lse_in; w.dpq = p.dpq; w.dpk = p.dpk;
    const int tables = pos_tables(p), per_table = 64 * p.r;
    const int blocks = (tables * per_table + 255) / 256 < 64 ? (tables * per_table + 255) / 256 : 64;
    {
        ProfileScope scope(RIB_KERNEL_WINDOW8_CLEAR, stream);
        bwd8::rib_window8_clear_kernel<<<blocks, 256, 0, stream>>>(p.dpq, p.dpk, tables, per_table, p.pos_head_stride);
    }
    if (cudaError_t e = cudaGetLastError()) return e;
    ProfileScope scope(RIB_KERNEL_WINDOW8_BWD, stream);
    return launch_overtaking(bwd8::rib_window8_bwd_kernel<R>, grid, bwd8::kThreads, bwd8::kSmemBytes, stream, tm_q, tm_k, tm_v, tm_do, tm_o, tm_dq, tm_dk, tm_dv, w);
}

}  // namespace

// Windows of 8 x 8 tokens without a shift on maps of whole tiles; the widths are those of the general kernels.
bool sm100_window8(const Problem& p)
{
    return p.M == 8 && p.s == 0 && p.H % 16 == 0 && p.W % 16 == 0 && !p.masked && !p.gate;
}
cudaError_t sm100_window8_fwd(const Problem& p, cudaStream_t stream)
{
    return padded_rank(p.r) == 32 ? launch_win8_fwd<32>(p, stream) : launch_win8_fwd<16>(p, stream);
}
cudaError_t sm100_window8_bwd(const Problem& p, cudaStream_t stream)
{
    return padded_rank(p.r) == 32 ? launch_win8_bwd<32>(p, stream) : launch_win8_bwd<16>(p, stream);
}

}  // namespace rib
