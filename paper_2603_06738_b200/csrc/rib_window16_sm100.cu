// RIB window attention for windows of 16 x 16 tokens on B200 (sm_100a), forward and backward: tcgen05 MMAs, TMEM, TMA loads and stores.
//
// A window is two query tiles and two key blocks of 128 tokens.  In the general kernels a work item is then over before its
// pipeline has filled, and what an item costs (staging of RIB rows, draining of accumulators, gradients added up in global
// memory) exceeds its arithmetic.  Here a CTA keeps to one head (CTA c: head c mod heads), stages the head's RIB rows once,
// takes whole windows one after the other and lets them overlap, and no gradient but those of the tables is summed
// outside the chip.  What bounds it: the serial program of the softmax (arithmetic) warps.  A unit of the forward (128 rows x 256
// keys) takes about 3600 cycles, of which the exp pipe is busy 1540; a unit of the backward (128 x 128) 2850 at rank 16 and 32 channels:
// 200 until its scores are there, 1500 of loads and exponentials, 1000 of stores of P and dS and fences, with 1470 cycles of MMAs
// beside it.  Measured by event hooks against the general kernels (4 x 96 x 96 tokens, 12 heads of 16 channels, rank 24, shift 8,
// masked): forward 60 against 84 us, backward 13 (two clearings) + 95 against 27 + 125 + 35 us; backward on 16 x 96 x 96 tokens, 6 heads of 32
// channels: rank 16 13 + 166 against 48 + 197 + 56, rank 32 13 + 190 against 56 + 228 + 95.
//
// Windows may be shifted (multiples of 8), masked, or reach beyond the map (sides multiples of 8): a window is four 8x8-token
// patches (one TMA box each), and a query patch attends to a key patch or not.
#include "rib_small_window.cuh"

namespace rib {
namespace {

using namespace sm100;

struct Win16 { int b, wy, wx, Y, X; };      // window; first position in shifted coordinates of the extended map (not wrapped)

__device__ __forceinline__ Win16 decode_window(const SmallWindowParams& p, int tile)
{
    Win16 w;
    p.by_nx.divmod(tile, tile, w.wx);
    p.by_ny.divmod(tile, w.b, w.wy);
    w.Y = 16 * w.wy + p.s; w.X = 16 * w.wx + p.s;
    return w;
}
__device__ __forceinline__ void patch_at(const SmallWindowParams& p, const Win16& w, int patch, int& Y0, int& X0)
{
    Y0 = w.Y + 8 * (patch >> 1); if (Y0 >= p.Hp) Y0 -= p.Hp;
    X0 = w.X + 8 * (patch & 1); if (X0 >= p.Wp) X0 -= p.Wp;
}
// The key patches that query patch q attends to, bit k: those in the map and, with a mask (the shift is then 8 or 0), in the last
// window of an axis those of its own row or column of patches.
__device__ __forceinline__ uint32_t attended(const SmallWindowParams& p, const Win16& w, int q)
{
    int y1 = w.Y + 8, x1 = w.X + 8;
    if (y1 >= p.Hp) y1 -= p.Hp;
    if (x1 >= p.Wp) x1 -= p.Wp;
    uint32_t ym = (w.Y < p.H ? 1u : 0u) | (y1 < p.H ? 2u : 0u), xm = (w.X < p.W ? 1u : 0u) | (x1 < p.W ? 2u : 0u);
    if (p.masked && p.s) {
        if (w.wy == (int)p.by_ny.d - 1) ym &= 1u << (q >> 1);
        if (w.wx == (int)p.by_nx.d - 1) xm &= 1u << (q & 1);
    }
    return (ym & 1u ? xm : 0u) | (ym & 2u ? xm << 2 : 0u);
}
// Row of the tables of row `row` of a window's 256 (patch row / 64, place row % 64 in it)
__device__ __forceinline__ int table_row(int row) { return (8 * (row >> 7) + ((row >> 3) & 7)) * 16 + 8 * ((row >> 6) & 1) + (row & 7); }

constexpr uint64_t kDesc64 = smem_desc_const(16, 512, kSwizzle64B);
constexpr uint32_t kWindowBytes = 2 * kContentBytes;                          // 256 rows x 64 bytes

// ================================================================================================ forward
// Unit = (window, query tile g): S = Q~_g K~^T is M128 N256, 256 columns of tensor memory per tile, so two units are under way.
// All 16 softmax warps work on one unit after the other, a thread being (row, key patch): 64 scores in registers, the row's
// maximum exchanged among its four threads through shared memory, P written over the own columns (so that 32 .. 95 and
// 160 .. 223 of the unit hold P), then O = P [V | ones] (N = 48: 32 channels and the row sum of the rounded probabilities) in the
// columns 96 .. 143, whose scores have been read.  The output of a unit is stored before or between the exponentials of
// the next, and the scores of the unit after next are computed under (the rest of) those.
// Output rows are stored from registers (a tensor map of the output would be a new one on every call with a new buffer).
// Roles (640 threads): warp 0 TMA loads, warp 1 issues S, warp 2 PV (and owns the TMEM allocation), warp 3 idles, warps 4-19
// softmax (4-7 key patch 0, 8-11 patch 1, ...).
namespace fwd16 {
constexpr int kThreads = 640, kStages = 3;
constexpr uint32_t kStageBytes = 3 * kWindowBytes;                            // q, k, v
constexpr uint32_t kOffRib = kStages * kStageBytes;                           // query RIB rows, key RIB rows
constexpr uint32_t kOffOnes = kOffRib + 2 * kWindowBytes;                     // [128 keys][32] column 0 = 1: second atom of V
constexpr uint32_t kOffMax = kOffOnes + kContentBytes;                        // [2 tiles][4 key patches][128 rows]
constexpr uint32_t kOffBar = kOffMax + 8 * kTile * 4;
enum Bar { kFull = 0, kEmpty = kFull + kStages, kSFull = kEmpty + kStages, kPReady = kSFull + 2, kOFull = kPReady + 2,
           kTFree = kOFull + 2, kMax = kTFree + 2, kDrain = kMax + 4, kNumBars = kDrain + 2 };
constexpr uint32_t kOffMisc = kOffBar + kNumBars * 8;
constexpr uint32_t kSmemBytes = kOffMisc + 16 + 1024;
static_assert(kOffOnes % 1024 == 0 && kSmemBytes <= 232448, "shared memory of one CTA");
constexpr uint32_t kIdescS = idesc_bf16_f32(kTile, 256, false), kIdescPV = idesc_bf16_f32(kTile, kD + 16, true);
constexpr uint32_t kColO = 96;                    // of a unit's 256 columns
constexpr uint32_t kPolyMask = 0x88u;             // of every 8 score pairs: which go to the FMA pipe

// kBetween: the output of the unit before is stored between the two halves of the exponentials, where its PV has completed (16 x 96 x 96
// tokens, 6 heads, masked, rank 16 124 -> 115 us, 360 x 632 at rank 32 189 -> 175; behind both halves, where the next scores wait for it,
// 126 and 192).  Not for heads of up to 24 channels, whose output some of the warps have no part in: at 16 307 against 316 us; at 24, us per call in a
// graph, masked, 4 heads, rank 8: 4 x 96 x 96 21.5 / 21.9, 256 x 256 33.7 / 34.5, 16 x 96 x 96 71.1 / 71.7, rank 24 72.2 / 72.5.
template <int R, bool kBetween>
__global__ void __launch_bounds__(kThreads, 1)
rib_window16_fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                        __nv_bfloat16* const out, const __grid_constant__ SmallWindowParams p)
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
    const int count = (p.tiles - group0 + p.groups - 1) / p.groups;           // windows of this CTA: group0 + t * groups

    if (threadIdx.x == 0) {
        abort_flag[0] = 0; abort_flag[1] = 0;   // [1] stays 0: used by the drain waits
        for (int s = 0; s < kStages; ++s) { mbar_init(bar(kFull + s), 1); mbar_init(bar(kEmpty + s), 1); }
        for (int g = 0; g < 2; ++g) {
            mbar_init(bar(kSFull + g), 1); mbar_init(bar(kPReady + g), 16); mbar_init(bar(kOFull + g), 1); mbar_init(bar(kTFree + g), 16);
        }
        for (int q4 = 0; q4 < 4; ++q4) mbar_init(bar(kMax + q4), 4);
        mbar_init(bar(kDrain), 1); mbar_init(bar(kDrain + 1), 1);
        fence_barrier_init();
        prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v);
    }
    if (warp == 2) {
        tmem_alloc(base + kOffMisc, 512);
        tmem_relinquish();
    }
    if (warp >= 4 && warp < 12) {
        const int row = (int)threadIdx.x - 128;
        stage_rib_row(p, head, table_row(row), base_ptr + kOffRib, base_ptr + kOffRib + kWindowBytes, row);
        if (row < 128) {
            uint4* dst = reinterpret_cast<uint4*>(base_ptr + kOffOnes + row * 64);
#pragma unroll
            for (int ck = 0; ck < 4; ++ck) dst[ck] = make_uint4(ck == ((row >> 1) & 3) ? 0x00003F80u : 0u, 0u, 0u, 0u);
        }
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
                const Win16 w = decode_window(p, group0 + t * p.groups);
                mbar_arrive_expect_tx(bar(kFull + st), kStageBytes);
                for (int patch = 0; patch < 4; ++patch) {          // (a patch beyond the map arrives as zeros)
                    int Y0, X0;
                    patch_at(p, w, patch, Y0, X0);
                    const uint32_t dst = base + st * kStageBytes + patch * kPatchContent;
                    tma_load_5d(dst, &tm_q, bar(kFull + st), 0, head, X0, Y0, w.b);
                    tma_load_5d(dst + kWindowBytes, &tm_k, bar(kFull + st), 0, head, X0, Y0, w.b);
                    tma_load_5d(dst + 2 * kWindowBytes, &tm_v, bar(kFull + st), 0, head, X0, Y0, w.b);
                }
            }
            if (!ok)                            // gave up: let the copies already in flight land before the CTA may exit
                for (int b2 = t > kStages ? t - kStages : 0; b2 < t; ++b2)
                    mbar_wait(bar(kFull + b2 % kStages), (b2 / kStages) & 1, abort_flag + 1, p.status);
        }
    } else if (warp == 1) {
        // ---- S of both query tiles; the whole warp walks the loop and waits, one elected lane issues
        bool ok = true;
        for (int t = 0; t < count && ok; ++t) {
            const int st = t % kStages;
            if (!mbar_wait_warp(bar(kFull + st), (t / kStages) & 1, abort_flag, p.status)) break;
            for (int g = 0; g < 2; ++g) {
                if (t > 0 && !mbar_wait_warp(bar(kTFree + g), (t - 1) & 1, abort_flag, p.status)) { ok = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t q = smem_desc_at(kDesc64, base + st * kStageBytes + g * kContentBytes), k = smem_desc_at(kDesc64, base + st * kStageBytes + kWindowBytes);
                    const uint64_t qp = smem_desc_at(kDesc64, base + kOffRib + g * kContentBytes), kp = smem_desc_at(kDesc64, base + kOffRib + kWindowBytes);
                    const uint32_t d = tmem + g * 256;
                    mma_ss(d, q, k, kIdescS, 0u);
                    mma_ss(d, q + 2, k + 2, kIdescS, 1u);         // + 32 bytes: second K16 step
                    mma_ss(d, qp, kp, kIdescS, 1u);
                    if (R == 32) mma_ss(d, qp + 2, kp + 2, kIdescS, 1u);
                    mma_commit(bar(kSFull + g));
                }
                __syncwarp();
            }
        }
        if (elect_one()) mma_commit(bar(kDrain));
        __syncwarp();
        mbar_wait(bar(kDrain), 0, abort_flag + 1, p.status);
    } else if (warp == 2) {
        // ---- O = P [V | ones]
        bool ok = true;
        for (int t = 0; t < count && ok; ++t) {
            const uint32_t v_off = (t % kStages) * kStageBytes + 2 * kWindowBytes;
            for (int g = 0; g < 2; ++g) {
                if (!mbar_wait_warp(bar(kPReady + g), t & 1, abort_flag, p.status)) { ok = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t d = tmem + g * 256;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint64_t v = smem_desc(base + v_off + h * kContentBytes, kOffOnes - (v_off + h * kContentBytes), 512, kSwizzle64B);
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) mma_ts(d + kColO, d + 128 * h + 32 + 8 * kk, v + 64 * kk, kIdescPV, h + kk ? 1u : 0u);
                    }
                    mma_commit(bar(kOFull + g));
                    if (g == 1) mma_commit(bar(kEmpty + t % kStages));      // S of both tiles finished before their P existed
                }
                __syncwarp();
            }
        }
        if (elect_one()) mma_commit(bar(kDrain + 1));
        __syncwarp();
        mbar_wait(bar(kDrain + 1), 0, abort_flag + 1, p.status);
    } else if (warp >= 4) {
        const int kq = (warp - 4) >> 2, quarter = warp & 3, row = quarter * 32 + lane;       // key patch; row of the unit == TMEM lane
        const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
        const uint32_t p_col = 64 * kq + (kq & 1 ? 0 : 32);
        float* const maxima = reinterpret_cast<float*>(base_ptr + kOffMax);                  // [tile][key patch][row]
        const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
        Win16 w = decode_window(p, group0);
        float m_last = 0.f;                      // maximum of this row in the unit before
        // O and l of a unit are complete: normalise and store this thread's 8 channels
        auto epilogue = [&](const Win16& ew, int g, float m) {
            uint32_t o[8], lsum[1];
            tmem_ld8(lanes + g * 256 + kColO + 8 * kq, o);
            tmem_ld1(lanes + g * 256 + kColO + kD, lsum);
            int Y0, X0;
            patch_at(p, ew, 2 * g + (quarter >> 1), Y0, X0);
            const int Y = Y0 + ((row >> 3) & 7), X = X0 + (row & 7);
            const size_t tok = (((size_t)ew.b * p.H + Y) * p.W + X) * p.heads + head;
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kTFree + g));
            if (Y0 < p.H && X0 < p.W) {                           // warp-uniform
                const float l = __uint_as_float(lsum[0]), inv = 1.f / l;
                if (8 * kq < p.d) {                               // (a head narrower than 32 channels: the rest of the row is padding)
                    uint32_t v[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) v[e] = pack_bf16x2(__uint_as_float(o[2 * e]) * inv, __uint_as_float(o[2 * e + 1]) * inv);
                    *reinterpret_cast<uint4*>(out + tok * p.d + 8 * kq) = make_uint4(v[0], v[1], v[2], v[3]);
                }
                if (p.lse && kq == 0) p.lse[(((size_t)ew.b * p.heads + head) * p.H + Y) * p.W + X] = m * p.inv_sqrt_d + logf(l);
            }
        };
        bool ok = true;
        for (int u = 0; u < 2 * count && ok; ++u) {
            const int t = u >> 1, g = u & 1;
            const Win16 before = w;                               // window of the unit before
            if (g == 0 && u > 0) w = decode_window(p, group0 + t * p.groups);
            const bool on = (attended(p, w, 2 * g + (quarter >> 1)) >> kq) & 1u;             // warp-uniform
            if (!mbar_wait_warp(bar(kSFull + g), t & 1, abort_flag, p.status)) break;
            tc_fence_after();
            uint32_t s[2][32];
            tmem_ld32(lanes + g * 256 + 64 * kq, s[0]);
            tmem_ld32(lanes + g * 256 + 64 * kq + 32, s[1]);
            tmem_wait_ld();
            float mx0 = -INFINITY, mx1 = -INFINITY;
            if (on) {
#pragma unroll
                for (int e = 0; e < 32; e += 2) {
                    mx0 = max3(mx0, __uint_as_float(s[0][e]), __uint_as_float(s[0][e + 1]));
                    mx1 = max3(mx1, __uint_as_float(s[1][e]), __uint_as_float(s[1][e + 1]));
                }
            }
            // (a warp can be one unit ahead of its partners here, no more: the sets of the two tiles are enough)
            float* const mine = maxima + g * 4 * kTile;
            mine[kq * kTile + row] = fmaxf(mx0, mx1);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kMax + quarter));
            auto unit_before = [&] {
                if (!mbar_wait_warp(bar(kOFull + (g ^ 1)), ((u - 1) >> 1) & 1, abort_flag, p.status)) return false;
                tc_fence_after();
                epilogue(before, g ^ 1, m_last);
                return true;
            };
            if (!kBetween && u > 0 && !unit_before()) break;
            if (!mbar_wait_warp(bar(kMax + quarter), u & 1, abort_flag, p.status)) break;
            const float m = fmaxf(fmaxf(mine[row], mine[kTile + row]), fmaxf(mine[2 * kTile + row], mine[3 * kTile + row]));
            const float neg = -m * p.scale_log2;
            const float2 neg2 = make_float2(neg, neg);
#pragma unroll
            for (int ch = 0; ch < 2; ++ch) {
                uint32_t pk[16];
                if (on) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[ch][2 * i]), __uint_as_float(s[ch][2 * i + 1])), scale2, neg2);
                        const float2 e = ((kPolyMask >> (i & 7)) & 1u) ? ex2_poly2(x) : make_float2(ex2_approx(x.x), ex2_approx(x.y));
                        pk[i] = pack_bf16x2(e.x, e.y);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) pk[i] = 0u;
                }
                tmem_st16(lanes + g * 256 + p_col + 16 * ch, pk);
                if (kBetween && ch == 0 && u > 0 && !(ok = unit_before())) break;
            }
            if (!ok) break;
            m_last = m;
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kPReady + g));
            if (u == 2 * count - 1) {
                // the last unit
                ok = mbar_wait_warp(bar(kOFull + g), t & 1, abort_flag, p.status);
                if (ok) { tc_fence_after(); epilogue(w, g, m); }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}
}  // namespace fwd16

// ================================================================================================ backward
// Unit u = 2 J + I of a window (rows = queries of tile I, columns = keys of block J):
//     S = Q~_I K~_J^T, dP = dO_I V_J^T;   P = exp2(S log2e/sqrt(d) - lse log2e), dS = P o (dP - D);
//     dV_J += P^T dO_I, dK~_J += dS^T Q~_I (A = the stored tiles, MN-major), dQ~_I += dS K~_J (A K-major).
// dV_J and dK~_J leave the chip after their two units, dQ~ at the end of the window.  The content columns of dQ~ are cleared
// when they have been read, its RIB columns (gradients of Pq) add up over the CTA's windows; those of dK~ do so in columns of their own at
// rank 16, and are added to global memory block by block at rank 32, for which tensor memory has no room.  (All windows' adds to one table
// meet at the same addresses: where the tables lay on some of them the kernel took 215 us instead of 180 at rank 16.)
//
// Roles (896 threads): warp 0 TMA loads; warp 1 issues S and dP, warp 3 dV, dK~ and dQ~; warp 2 owns the TMEM allocation; warps
// 4-19 P and dS (four threads per query row, 32 keys each); warps 20-23 move the gradients out, dv from registers, dk and dq through the
// shared memory of the window's own rows and TMA stores; warps 24-27 write
// (-lse log2e, -D) of the windows to come to tensor memory, a row being a TMEM lane to everybody.  (One set of warps for both, and lanes
// that load whole rows: 215 us on 16 x 96 x 96 tokens, 6 heads of 32 channels, rank 16, 240 at rank 32.  dv in 32-byte stores, four lanes to a
// row of dO and O 191 / 211, warps of their own, with dO from the stage, 180 / 201: 8000 cycles of waiting for
// loads held up dV and dK~ of the next window.  That form lost up to 8 % where heads are narrow and a CTA has few windows, whose scalars then wait
// for the first window's copies.  Those are asked for before the block's first barrier, the sums of dK~'s RIB columns are kept off the
// hand-over of the accumulators, 72 registers do without spills, and the TMA stores, which warp 2 issued behind barriers of their own then, are
// warp 20's again; us per call in a graph, before the warps of their own / with them / now: 64 x 64, 4 heads of 24 channels 14.8 / 16.1 / 14.6;
// 96 x 96, 6 of 16 20.1 / 21.5 / 20.2; 16 x 96 x 96, 6 of 8 156 / 159 / 152, of 32 214 / 175 / 162; head-wise tables, 4 x 96 x 96, 6 of 8
// 43.7 / 46.9 / 44.3.)
namespace bwd16 {
constexpr int kThreads = 896, kStages = 2;
constexpr uint32_t kQ = 0, kK = kWindowBytes, kV = 2 * kWindowBytes, kDO = 3 * kWindowBytes, kStageBytes = 4 * kWindowBytes;
constexpr uint32_t kOffRib = kStages * kStageBytes;                           // query RIB rows, key RIB rows
constexpr uint32_t kHalf = kTile * 128;                                       // P, dS: [2 halves of 64 keys][128 queries][128 bytes], SWIZZLE_128B
constexpr uint32_t kOffP = kOffRib + 2 * kWindowBytes, kOffDS = kOffP + 2 * kHalf, kOffBar = kOffDS + 2 * kHalf;
enum Bar { kFull = 0, kEmpty = kFull + kStages, kSFull = kEmpty + kStages, kSFree, kPReady, kPDone, kSReady, kSDone, kAcc, kKVFree, kQFree, kLd, kLdFree = kLd + 2, kDrain, kNumBars = kDrain + 2 };
constexpr uint32_t kOffMisc = kOffBar + kNumBars * 8;
constexpr uint32_t kSmemBytes = kOffMisc + 16 + 1024;
static_assert(kOffP % 1024 == 0 && kSmemBytes <= 232448, "shared memory of one CTA");

// tensor memory: S, dP, dV, dK~, dQ~ of both tiles, (-lse2, -D) of both tiles for two windows
constexpr uint32_t kColS = 0, kColDP = 128, kColDV = 256, kColDK = 288;
template <int R> constexpr uint32_t kColDQ = kColDK + kD + R;
template <int R> constexpr uint32_t kColLd = kColDQ<R> + 2 * (kD + R);
template <int R> constexpr uint32_t kColRib = kColLd<R> + 8;       // R = 16: RIB columns of dK~ of both blocks, added up over the CTA's windows

constexpr uint32_t kIdescS = idesc_bf16_f32(kTile, kTile, false);

template <int R>
__global__ void __launch_bounds__(kThreads, 1)
rib_window16_bwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                        const __grid_constant__ CUtensorMap tm_do, const __grid_constant__ CUtensorMap tm_dq, const __grid_constant__ CUtensorMap tm_dk,
                        __nv_bfloat16* const dv, const int dv_sectors, const __grid_constant__ SmallWindowParams p)
{
    static_assert(kColRib<R> + (R == 16 ? 2 * R : 0) <= 512, "tensor memory has 512 columns");
    constexpr uint32_t kIdescDV = idesc_bf16_f32_ab(kTile, kD, true, true), kIdescDK = idesc_bf16_f32_ab(kTile, kD + R, true, true);
    constexpr uint32_t kIdescDQ = idesc_bf16_f32_ab(kTile, kD + R, false, true);
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
    const uint32_t units = 4u * (uint32_t)count;

    // (The loop is kept: unrolled, its addresses cost the arithmetic warps registers.)
    auto load_window = [&](int t) {
        const int st = t % kStages;
        const Win16 w = decode_window(p, group0 + t * p.groups);
        mbar_arrive_expect_tx(bar(kFull + st), kStageBytes);
#pragma unroll 1
        for (int patch = 0; patch < 4; ++patch) {
            int Y0, X0;
            patch_at(p, w, patch, Y0, X0);
            const uint32_t at = base + st * kStageBytes + patch * kPatchContent;
            tma_load_5d(at + kQ, &tm_q, bar(kFull + st), 0, head, X0, Y0, w.b);
            tma_load_5d(at + kK, &tm_k, bar(kFull + st), 0, head, X0, Y0, w.b);
            tma_load_5d(at + kV, &tm_v, bar(kFull + st), 0, head, X0, Y0, w.b);
            tma_load_5d(at + kDO, &tm_do, bar(kFull + st), 0, head, X0, Y0, w.b);
        }
    };
    if (threadIdx.x == 0) {
        abort_flag[0] = 0; abort_flag[1] = 0;   // [1] stays 0: used by the drain waits
        for (int s = 0; s < kStages; ++s) { mbar_init(bar(kFull + s), 1); mbar_init(bar(kEmpty + s), 1); mbar_init(bar(kLd + s), 4); }
        mbar_init(bar(kSFull), 1); mbar_init(bar(kSFree), 16); mbar_init(bar(kPReady), 16); mbar_init(bar(kPDone), 1); mbar_init(bar(kSReady), 16); mbar_init(bar(kSDone), 1);
        mbar_init(bar(kAcc), 1); mbar_init(bar(kKVFree), 4); mbar_init(bar(kQFree), 4);
        mbar_init(bar(kLdFree), 16);
        mbar_init(bar(kDrain), 1); mbar_init(bar(kDrain + 1), 1);
        fence_barrier_init();
        fence_proxy_async();
        load_window(0);                         // before the rows of the tables are staged and tensor memory is there
        prefetch_tensormap(&tm_dq); prefetch_tensormap(&tm_dk);
    }
    if (warp == 2) {
        tmem_alloc(base + kOffMisc, 512);
        tmem_relinquish();
    }
    if (warp >= 4 && warp < 12) {
        const int row = (int)threadIdx.x - 128;
        stage_rib_row(p, head, table_row(row), base_ptr + kOffRib, base_ptr + kOffRib + kWindowBytes, row);
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int t = 1;
            bool ok = true;
            for (; t < count; ++t) {
                if (t >= kStages && !mbar_wait(bar(kEmpty + t % kStages), (t / kStages - 1) & 1, abort_flag, p.status)) { ok = false; break; }
                load_window(t);
            }
            if (!ok)                            // gave up: let the copies already in flight land before the CTA may exit
                for (int b2 = t > kStages ? t - kStages : 0; b2 < t; ++b2)
                    mbar_wait(bar(kFull + b2 % kStages), (b2 / kStages) & 1, abort_flag + 1, p.status);
        }
    } else if (warp == 1) {
        // ---- S and dP of a unit once the arithmetic warps hold those of the unit before in registers
        for (uint32_t u = 0; u < units; ++u) {
            const uint32_t t = u >> 2, I = u & 1, J = (u >> 1) & 1, st = t % kStages;
            if (((u & 3) == 0 && !mbar_wait_warp(bar(kFull + st), (t / kStages) & 1, abort_flag, p.status)) ||
                (u > 0 && !mbar_wait_warp(bar(kSFree), (u - 1) & 1, abort_flag, p.status))) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t at = base + st * kStageBytes, ti = I * kContentBytes, tj = J * kContentBytes;
                const uint64_t q = smem_desc_at(kDesc64, at + kQ + ti), k = smem_desc_at(kDesc64, at + kK + tj);
                const uint64_t qp = smem_desc_at(kDesc64, base + kOffRib + ti), kp = smem_desc_at(kDesc64, base + kOffRib + kWindowBytes + tj);
                const uint64_t v = smem_desc_at(kDesc64, at + kV + tj), go = smem_desc_at(kDesc64, at + kDO + ti);
                mma_ss(tmem + kColS, q, k, kIdescS, 0u);
                mma_ss(tmem + kColS, q + 2, k + 2, kIdescS, 1u);
                mma_ss(tmem + kColS, qp, kp, kIdescS, 1u);
                if (R == 32) mma_ss(tmem + kColS, qp + 2, kp + 2, kIdescS, 1u);
                mma_ss(tmem + kColDP, go, v, kIdescS, 0u);
                mma_ss(tmem + kColDP, go + 2, v + 2, kIdescS, 1u);
                mma_commit(bar(kSFull));
            }
            __syncwarp();
        }
        if (elect_one()) mma_commit(bar(kDrain));
        __syncwarp();
        mbar_wait(bar(kDrain), 0, abort_flag + 1, p.status);
    } else if (warp == 3) {
        // ---- dV of a unit once P is stored, dK~ and dQ~ once dS is, and the accumulators that it starts have been read
        constexpr uint64_t kDescT = smem_desc_const(kHalf, 1024, kSwizzle128B);         // MN-major: the two 64-key halves one leading step apart
        constexpr uint64_t kDescN = smem_desc_const(16, 1024, kSwizzle128B);            // K-major: one half
        for (uint32_t u = 0; u < units; ++u) {
            const uint32_t t = u >> 2, I = u & 1, J = (u >> 1) & 1, st = t % kStages;
            if (!mbar_wait_warp(bar(kPReady), u & 1, abort_flag, p.status) ||
                (I == 0 && !mbar_wait_warp(bar(kKVFree), (u >> 1) & 1, abort_flag, p.status))) break;
            tc_fence_after();
            if (elect_one()) {
                const uint64_t go = smem_desc_at(kDesc64, base + st * kStageBytes + kDO + I * kContentBytes), pt = smem_desc_at(kDescT, base + kOffP);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ss(tmem + kColDV, pt + 128 * kk, go + 64 * kk, kIdescDV, (kk || I) ? 1u : 0u);
                mma_commit(bar(kPDone));
            }
            __syncwarp();
            if (!mbar_wait_warp(bar(kSReady), u & 1, abort_flag, p.status) ||
                ((u & 3) == 0 && !mbar_wait_warp(bar(kQFree), t & 1, abort_flag, p.status))) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t off = st * kStageBytes, ti = I * kContentBytes, tj = J * kContentBytes;
                const uint64_t q = smem_desc(base + off + kQ + ti, kOffRib - (off + kQ), 512, kSwizzle64B);                     // [Q | Pq] of tile I
                const uint64_t k = smem_desc(base + off + kK + tj, kOffRib + kWindowBytes - (off + kK), 512, kSwizzle64B);      // [K | Pk] of block J
                const uint64_t dst = smem_desc_at(kDescT, base + kOffDS), ds = smem_desc_at(kDescN, base + kOffDS);
                const uint32_t d_q = tmem + kColDQ<R> + I * (kD + R);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ss(tmem + kColDK, dst + 128 * kk, q + 64 * kk, kIdescDK, (kk || I) ? 1u : 0u);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) mma_ss(d_q, ds + (kk >> 2) * (kHalf >> 4) + 2 * (kk & 3), k + 64 * kk, kIdescDQ, 1u);
                mma_commit(bar(kSDone));
                if (I == 1) mma_commit(bar(kAcc));
            }
            __syncwarp();
        }
        if (elect_one()) mma_commit(bar(kDrain + 1));
        __syncwarp();
        mbar_wait(bar(kDrain + 1), 0, abort_flag + 1, p.status);
    } else if (warp >= 4 && warp < 20) {
        // ---- P and dS: thread = (query row, 32 keys of the block)
        const int quarter = warp & 3, cq = (warp - 4) >> 2, row = quarter * 32 + lane;
        const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
        const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
        uint8_t *p_row = base_ptr + kOffP + (cq >> 1) * kHalf + row * 128, *ds_row = base_ptr + kOffDS + (cq >> 1) * kHalf + row * 128;
        uint32_t seen = 0u;         // bit 4 I + 2 J + half
        for (uint32_t u = 0; u < units; ++u) {
            const uint32_t t = u >> 2, I = u & 1, J = (u >> 1) & 1;
            if ((u & 3) == 0) {
                const Win16 w = decode_window(p, group0 + (int)t * p.groups);
                seen = attended(p, w, quarter >> 1) | attended(p, w, 2 + (quarter >> 1)) << 4;
                if (!mbar_wait_warp(bar(kLd + (t & 1)), (t >> 1) & 1, abort_flag, p.status)) break;
            }
            const bool on = (seen >> (4 * I + 2 * J + (cq >> 1))) & 1u;      // warp-uniform
            if (!mbar_wait_warp(bar(kSFull), u & 1, abort_flag, p.status)) break;
            tc_fence_after();
            uint32_t pp[16], dd[16], ld[2], s[4][8], dp[4][8];
            // Four pieces of 8 keys, the loads of a piece under the arithmetic of the one before; P and dS are stored together behind one
            // fence when both buffers are free already (16 x 96 x 96 tokens, 6 heads, rank 16: two pieces of 16 and a fence each 224 us, so 214).
            auto load = [&](int c) {
                tmem_ld8(lanes + kColS + 32 * cq + 8 * c, s[c]);
                tmem_ld8(lanes + kColDP + 32 * cq + 8 * c, dp[c]);
            };
            auto work = [&](int c) {
                const float2 l2 = make_float2(__uint_as_float(ld[0]), __uint_as_float(ld[0])), d2 = make_float2(__uint_as_float(ld[1]), __uint_as_float(ld[1]));
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[c][2 * i]), __uint_as_float(s[c][2 * i + 1])), scale2, l2);
                    const float2 e = make_float2(ex2_approx(x.x), ex2_approx(x.y));
                    const float2 d = __fmul2_rn(e, __fadd2_rn(make_float2(__uint_as_float(dp[c][2 * i]), __uint_as_float(dp[c][2 * i + 1])), d2));
                    pp[4 * c + i] = pack_bf16x2(e.x, e.y);
                    dd[4 * c + i] = pack_bf16x2(d.x, d.y);
                }
            };
            tmem_ld2(lanes + kColLd<R> + 4 * (t & 1) + 2 * I, ld);
            load(0); load(1);
            tmem_wait_ld();
            load(2);
            work(0);
            tmem_wait_ld();
            load(3);
            work(1);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar(kSFree));
                if ((u & 3) == 0) mbar_arrive(bar(kLdFree));          // nobody reads (-lse2, -D) of the window before any more
            }
            // have the contractions of the unit before read P and dS?  (No phase completed answers yes to parity 1, which unit 0 asks for.)
            const bool p_free = mbar_try_wait(bar(kPDone), (u - 1) & 1), ds_free = mbar_test(bar(kSDone), (u - 1) & 1);
            work(2);
            work(3);
            if (!on) {
#pragma unroll
                for (int i = 0; i < 16; ++i) pp[i] = dd[i] = 0u;
            }
            auto put = [&](uint8_t* line, const uint32_t (&v)[16]) {
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4)
                    *reinterpret_cast<uint4*>(line + (((4 * (cq & 1) + q4) ^ (row & 7)) << 4)) = make_uint4(v[4 * q4], v[4 * q4 + 1], v[4 * q4 + 2], v[4 * q4 + 3]);
            };
            auto announce = [&](uint32_t ready) {
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(ready);
            };
            if (__all_sync(0xffffffffu, p_free & ds_free)) {
                put(p_row, pp);
                put(ds_row, dd);
                announce(bar(kPReady));
                if (lane == 0) mbar_arrive(bar(kSReady));
                continue;
            }
            // P, then dS: the contractions of the unit before that read each of them end one after the other, too
            auto store = [&](uint8_t* line, const uint32_t (&v)[16], uint32_t done, uint32_t ready) {
                if (u > 0 && !mbar_wait_warp(done, (u - 1) & 1, abort_flag, p.status)) return false;
                put(line, v);
                announce(ready);
                return true;
            };
            if (!store(p_row, pp, bar(kPDone), bar(kPReady)) || !store(ds_row, dd, bar(kSDone), bar(kSReady))) break;
        }
    } else if (warp >= 24) {
        // ---- (-lse2, -D) of every window: thread = row of a tile
        const int quarter = warp & 3;
        const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
        const uint32_t line = (uint32_t)(p.W * p.heads * p.d), in_line = (uint32_t)((lane >> 2) * p.heads * p.d + 8 * (lane & 3));
        for (int t = 0; t < count; ++t) {
            // (The columns are free by then in any case: the stage is filled again after window t - 2.  But loads of `out` that run further ahead
            // cost the kernel more than they save: without this wait 16 x 96 x 96 tokens, 6 heads of 32 channels, rank 16 180 us instead of 162.)
            if (t >= 1 && !mbar_wait_warp(bar(kLdFree), (t - 1) & 1, abort_flag, p.status)) break;
            tc_fence_after();
            // D = dO . O: four lanes take a row (8 channels each), an instruction the 8 rows of a line of tokens; dO lies in the stage.  (With a row per
            // lane every load touches 32 lines, which holds up the queue of everybody's loads and stores.)
            const Win16 w = decode_window(p, group0 + t * p.groups);
            float neg_lse[2] = {-INFINITY, -INFINITY}, neg_d[2] = {0.f, 0.f};      // a query beyond the map: probability 0
            bool exists[2];
            uint4 y[2][4];
#pragma unroll
            for (int I = 0; I < 2; ++I) {
                int Y0, X0;
                patch_at(p, w, 2 * I + (quarter >> 1), Y0, X0);
                exists[I] = Y0 < p.H && X0 < p.W;            // warp-uniform
                Y0 += 4 * (quarter & 1);                     // this warp's 4 x 8 tokens; lane = 8 * row + column
                size_t at = ((((size_t)w.b * p.H + Y0) * p.W + X0) * p.heads + head) * p.d + in_line;
#pragma unroll
                for (int j = 0; j < 4; ++j, at += line)
                    y[I][j] = exists[I] && 8 * (lane & 3) < p.d ? __ldg(reinterpret_cast<const uint4*>(p.out + at)) : make_uint4(0u, 0u, 0u, 0u);
                if (exists[I]) neg_lse[I] = p.lse_in[(((size_t)w.b * p.heads + head) * p.H + Y0 + (lane >> 3)) * p.W + X0 + (lane & 7)];
            }
            const int st = t % kStages;
            if (!mbar_wait_warp(bar(kFull + st), (t / kStages) & 1, abort_flag, p.status)) break;
#pragma unroll
            for (int I = 0; I < 2; ++I) {
                if (exists[I]) {
                    const uint8_t* const rows = base_ptr + st * kStageBytes + kDO + I * kContentBytes + (quarter * 32 + (lane >> 2)) * 64;
                    neg_lse[I] *= -1.4426950408889634f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint4 x = *reinterpret_cast<const uint4*>(rows + 512 * j + (((lane & 3) ^ ((lane >> 3) & 3)) << 4));      // SWIZZLE_64B
                        const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y[I][j].x, y[I][j].y, y[I][j].z, y[I][j].w};
                        float sum = 0.f;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            sum = fmaf(-__uint_as_float(xs[e] << 16), __uint_as_float(ys[e] << 16), sum);
                            sum = fmaf(-__uint_as_float(xs[e] & 0xffff0000u), __uint_as_float(ys[e] & 0xffff0000u), sum);
                        }
                        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
                        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                        const float mine = __shfl_sync(0xffffffffu, sum, 4 * (lane & 7));
                        if ((lane >> 3) == j) neg_d[I] = mine;
                    }
                }
                __syncwarp();
                tmem_st2(lanes + kColLd<R> + 4 * (t & 1) + 2 * I, __float_as_uint(neg_lse[I]), __float_as_uint(neg_d[I]));
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kLd + (t & 1)));
        }
    } else if (warp >= 20) {
        // ---- gradients out: thread = row of a tile
        const int quarter = warp & 3, row = quarter * 32 + lane;
        const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
        const size_t table = (size_t)head * p.pos_head_stride;
        auto clear32 = [&](uint32_t col) {
            uint32_t zero[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) zero[e] = 0u;
            tmem_st32(lanes + col, zero);
        };
        for (int I = 0; I < 2; ++I) { clear32(kColDQ<R> + I * (kD + R)); clear32(kColDQ<R> + I * (kD + R) + R); }      // 32 + R columns each
        if (R == 16) clear32(kColRib<R>);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) { mbar_arrive(bar(kKVFree)); mbar_arrive(bar(kQFree)); }
        cudaGridDependencySynchronize();                     // dpq, dpk are cleared
        bool ok = true;
        for (int t = 0; t < count && ok; ++t) {
            const int st = t % kStages;
            uint8_t* const stage = base_ptr + st * kStageBytes;
            const Win16 w = decode_window(p, group0 + t * p.groups);
            for (int J = 0; J < 2; ++J) {
                // (the vote of the named barrier below keeps the four warps together)
                ok = mbar_wait_warp(bar(kAcc), J, abort_flag, p.status);
                if (ok) {
                    tc_fence_after();
                    uint32_t a[32];
                    tmem_ld32(lanes + kColDV, a);
                    tmem_wait_ld();
                    int Y0, X0;
                    patch_at(p, w, 2 * J + (row >> 6), Y0, X0);
                    if (Y0 < p.H && X0 < p.W) {              // warp-uniform
                        uint4* const dst = reinterpret_cast<uint4*>(dv + ((((size_t)w.b * p.H + Y0 + ((row >> 3) & 7)) * p.W + X0 + (row & 7)) * p.heads + head) * p.d);
                        uint32_t v[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] = pack_bf16x2(__uint_as_float(a[2 * e]), __uint_as_float(a[2 * e + 1]));
                        if (dv_sectors) {                    // rows of whole 32-byte sectors: half the instructions, each of which touches 32 lines
                            st_global_v8(dst, v);
                            if (p.d > 16) st_global_v8(dst + 2, v + 8);
                        } else {
#pragma unroll
                            for (int q4 = 0; q4 < 4; ++q4) {
                                if (8 * q4 >= p.d) break;
                                dst[q4] = make_uint4(v[4 * q4], v[4 * q4 + 1], v[4 * q4 + 2], v[4 * q4 + 3]);
                            }
                        }
                    }
                    __syncwarp();
                    tmem_ld32(lanes + kColDK, a);
                    tmem_wait_ld();
                    write_row(stage + kK + J * kContentBytes, row, a, p.inv_sqrt_d);
                    if (R == 16) tmem_ld16(lanes + kColDK + kD, reinterpret_cast<uint32_t(&)[16]>(a));
                    else tmem_ld32(lanes + kColDK + kD, a);
                    tmem_wait_ld();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kKVFree));
                    if (R == 16) {
                        // behind the hand-over, which the next block's dV and dK~ wait for; the store is awaited with those of J = 1
                        uint32_t sums[16];
                        tmem_ld16(lanes + kColRib<R> + R * J, sums);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) sums[e] = __float_as_uint(__uint_as_float(sums[e]) + __uint_as_float(a[e]));
                        if (t + 1 < count) {
                            tmem_st16(lanes + kColRib<R> + R * J, sums);
                        } else {
                            float* const gk = p.dpk + table + (size_t)table_row(J * kTile + row) * p.r;
#pragma unroll
                            for (int c = 0; c < R; c += 4)
                                if (c < p.r) add_columns(gk + c, sums + c, p.inv_sqrt_d);       // (the query rows carried sqrt(d / r))
                        }
                    } else {
                        float* const gk = p.dpk + table + (size_t)table_row(J * kTile + row) * p.r;
#pragma unroll
                        for (int c = 0; c < R; c += 4)
                            if (c < p.r) add_columns(gk + c, a + c, p.inv_sqrt_d);       // (the query rows carried sqrt(d / r))
                    }
                    if (J == 1) {
#pragma unroll
                        for (int I = 0; I < 2; ++I) {
                            tmem_ld32(lanes + kColDQ<R> + I * (kD + R), a);
                            tmem_wait_ld();
                            clear32(kColDQ<R> + I * (kD + R));
                            write_row(stage + kQ + I * kContentBytes, row, a, p.inv_sqrt_d);
                        }
                        tmem_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar(kQFree));
                    }
                    fence_proxy_async();
                }
                if (!named_barrier_and(1, 128, ok)) { ok = false; break; }
                if (warp == 20 && lane == 0) {
                    const uint32_t at = base + st * kStageBytes;
                    for (int patch = 0; patch < 4; ++patch) {
                        int Y0, X0;
                        patch_at(p, w, patch, Y0, X0);
                        if (Y0 >= p.H || X0 >= p.W) continue;
                        if ((patch >> 1) == J) tma_store_5d(&tm_dk, at + kK + patch * kPatchContent, 0, head, X0, Y0, w.b);
                        if (J == 1) tma_store_5d(&tm_dq, at + kQ + patch * kPatchContent, 0, head, X0, Y0, w.b);
                    }
                    bulk_commit_group();
                    if (J == 1) {
                        bulk_wait_group_read<0>();
                        mbar_arrive(bar(kEmpty + st));
                    }
                }
                __syncwarp();
            }
        }
        if (ok) {
            // gradients of Pq of this CTA
            tc_fence_after();
            for (int I = 0; I < 2; ++I) {
                uint32_t a[32];
                if (R == 16) tmem_ld16(lanes + kColDQ<R> + I * (kD + R) + kD, reinterpret_cast<uint32_t(&)[16]>(a));
                else tmem_ld32(lanes + kColDQ<R> + I * (kD + R) + kD, a);
                tmem_wait_ld();
                float* const gq = p.dpq + table + (size_t)table_row(I * kTile + row) * p.r;
#pragma unroll
                for (int c = 0; c < R; c += 4)
                    if (c < p.r) add_columns(gq + c, a + c, p.inv_sqrt_r);
            }
        }
        if (warp == 20 && lane == 0) bulk_wait_group<0>();
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// Clears the gradients of one kind of table (the tables only, not what lies between them).  The kernel behind it on the stream
// overtakes it; it ends after the kernel before it, so that the last of a chain stands for all of them.
__global__ void __launch_bounds__(256) rib_window16_clear_kernel(float* grads, int tables, int per_table, long long stride)
{
    cudaTriggerProgrammaticLaunchCompletion();
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < tables * per_table; e += gridDim.x * blockDim.x)
        grads[(size_t)(e / per_table) * stride + e % per_table] = 0.f;
    cudaGridDependencySynchronize();
}
}  // namespace bwd16

template <int R, bool kBetween>
cudaError_t launch_win16_fwd(const Problem& p, cudaStream_t stream)
{
    CUtensorMap tm_q, tm_k, tm_v;
    if (!encode_fn()) return cudaErrorNotSupported;
    if (!encode_image_map(&tm_q, p.q, p) || !encode_image_map(&tm_k, p.k, p) || !encode_image_map(&tm_v, p.v, p)) return cudaErrorInvalidValue;
    static KernelSetup setup;       // one per instantiation of this launcher, i.e. per kernel
    int sm_count = 0;
    if (cudaError_t e = setup.prepare(fwd16::rib_window16_fwd_kernel<R, kBetween>, fwd16::kSmemBytes, &sm_count)) return e;
    SmallWindowParams w{};
    const int grid = fill_small_window(p, sm_count, p.nWy, p.nWx, &w);
    w.lse = p.lse_w;
    ProfileScope scope(RIB_KERNEL_WINDOW16_FWD, stream);
    fwd16::rib_window16_fwd_kernel<R, kBetween><<<grid, fwd16::kThreads, fwd16::kSmemBytes, stream>>>(tm_q, tm_k, tm_v, p.out_w, w);
    return cudaGetLastError();
}

template <int R>
cudaError_t launch_win16_bwd(const Problem& p, cudaStream_t stream)
{
    CUtensorMap tm_q, tm_k, tm_v, tm_do, tm_dq, tm_dk;
    if (!encode_fn()) return cudaErrorNotSupported;
    if (!encode_image_map(&tm_q, p.q, p) || !encode_image_map(&tm_k, p.k, p) || !encode_image_map(&tm_v, p.v, p) || !encode_image_map(&tm_do, p.dout, p) ||
        !encode_image_map(&tm_dq, p.dq, p) || !encode_image_map(&tm_dk, p.dk, p))
        return cudaErrorInvalidValue;
    static KernelSetup setup;
    int sm_count = 0;
    if (cudaError_t e = setup.prepare(bwd16::rib_window16_bwd_kernel<R>, bwd16::kSmemBytes, &sm_count)) return e;
    SmallWindowParams w{};
    const int grid = fill_small_window(p, sm_count, p.nWy, p.nWx, &w);
    w.out = p.out; w.lse_in = p.lse_in; w.dpq = p.dpq; w.dpk = p.dpk;
    const int tables = pos_tables(p), per_table = 256 * p.r, blocks = (tables * per_table + 255) / 256 < 64 ? (tables * per_table + 255) / 256 : 64;
    {
        ProfileScope scope(RIB_KERNEL_WINDOW16_CLEAR, stream);
        bwd16::rib_window16_clear_kernel<<<blocks, 256, 0, stream>>>(p.dpq, tables, per_table, p.pos_head_stride);
    }
    if (cudaError_t e = cudaGetLastError()) return e;
    {
        ProfileScope scope(RIB_KERNEL_WINDOW16_CLEAR, stream);
        if (cudaError_t e = launch_overtaking(bwd16::rib_window16_clear_kernel, blocks, 256, 0, stream, p.dpk, tables, per_table, p.pos_head_stride)) return e;
    }
    const int dv_sectors = p.d % 16 == 0 && (reinterpret_cast<uintptr_t>(p.dv) & 31u) == 0;
    ProfileScope scope(RIB_KERNEL_WINDOW16_BWD, stream);
    return launch_overtaking(bwd16::rib_window16_bwd_kernel<R>, grid, bwd16::kThreads, bwd16::kSmemBytes, stream, tm_q, tm_k, tm_v, tm_do, tm_dq, tm_dk, p.dv, dv_sectors, w);
}

}  // namespace

// (sides that are no multiples of 8 have kernels of their own)
bool sm100_window16(const Problem& p) { return p.M == 16 && p.s % 8 == 0 && p.H % 8 == 0 && p.W % 8 == 0 && !p.gate; }
// Forward, this kernel against the general one, us per call in a graph (6 heads of 32 channels unless stated; 12 x 16: 12 heads of 16):
//   whole windows          rank 16: 10 x 64 x 64 tokens 35 / 28, 256 x 256 52 / 41, 16 x 96 x 96 108 / 83; rank 32: 36 / 33, 54 / 51; 12 x 16, rank 24:
//                          4 x 96 x 96 53 / 51, 256 x 256 94 / 86;
//   with a mask            rank 16: 64 x 64 9.0 / 12.1, 10 x 64 x 64 35 / 44, 256 x 256 52.8 / 53.6, 4 x 256 x 256 190 / 195, 16 x 96 x 96 110 / 128; rank 32:
//                          10 x 64 x 64 36 / 54, 256 x 256 54 / 66; 12 x 16, rank 24: 4 x 96 x 96 53 / 79; 4 heads of 24, rank 8: 22 / 27;
//   beyond the map         rank 16: 48 x 40 8.8 / 9.2, 104 x 120 16.0 / 16.5, 120 x 200 24.4 / 24.7, 152 x 264 36.6 / 33.3, 200 x 328 55 / 52, 360 x 632
//                          168 / 161; 6 x 8, rank 8 157 / 152, 6 x 24 162 / 163; rank 32: 120 x 200 25 / 29, 360 x 632 171 / 202; 12 x 16, rank 24: 310 / 368.
// So whole windows stay with the general kernel, masks come here, and windows beyond the map come here with RIB rows of 32 elements or
// while there is little work (120 x 200 tokens are four windows per SM).
// This kernel has the fast form of the softmax only (one exponential in four on the FMA pipe, lse from rounded probabilities):
// calls that ask for the exact form take the general kernel.
bool sm100_window16_prefers(const Problem& p)
{
    if (!sm100_window16(p) || p.exact_softmax) return false;
    return p.masked || ((p.Hp != p.H || p.Wp != p.W) && (padded_rank(p.r) == 32 || p.pairs <= 4 * 148));
}
cudaError_t sm100_window16_fwd(const Problem& p, cudaStream_t stream)
{
    if (p.d > 24) return padded_rank(p.r) == 32 ? launch_win16_fwd<32, true>(p, stream) : launch_win16_fwd<16, true>(p, stream);
    return padded_rank(p.r) == 32 ? launch_win16_fwd<32, false>(p, stream) : launch_win16_fwd<16, false>(p, stream);
}
cudaError_t sm100_window16_bwd(const Problem& p, cudaStream_t stream)
{
    return padded_rank(p.r) == 32 ? launch_win16_bwd<32>(p, stream) : launch_win16_bwd<16>(p, stream);
}

}  // namespace rib
