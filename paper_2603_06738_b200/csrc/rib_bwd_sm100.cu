// Backward RIB window attention for B200 (sm_100a): the chain rule of Eq. 6 and the softmax as five
// tcgen05 contractions per (query tile, key block) with TMEM accumulators and TMA loads.
//
// Shapes: d = 32, r = 16 or 32 (template argument R), window side M a multiple of 16, shift a multiple of 8 (as
// the forward).  The text below describes R = 16.  With R = 32 the RIB rows fill their 64-byte slots, dK~ and dQ~ are
// 64 columns wide, and tensor memory has no room left for dS^T: dK~ then takes the dS tile in shared memory as a
// K-major A operand (that tile's barrier counts two readers), and dP^T has two buffers of its own.
//
// Work item = one (batch, window, head) pair x one key block J of 128 tokens.  A persistent CTA keeps
// K~_J = [k, Pk] and V_J in shared memory and dV_J, dK~_J in tensor memory, and walks the query tiles
// I of the window.  Everything is computed transposed (keys on the TMEM lanes) so that P^T and dS^T
// feed the dV and dK~ contractions straight from tensor memory.  The unit of the pipeline is a
// half-tile u = 2 I + h: the 64 queries of patch h of tile I,
//     S^T  = K~_J Q~_u^T                    (M128 N64 K48: content rows 2 x K16, RIB rows 1 x K16)
//     dP^T = V_J dO_u^T                     (M128 N64 K32)
//     P^T  = exp2(S^T * log2e/sqrt(d) - lse_i * log2e),   dS^T = P^T o (dP^T - D_i)     (ALU warps)
//     dV_J  += P^T  dO_u                    (A from TMEM, B = dO rows, MN-major, N = 32)
//     dK~_J += dS^T Q~_u                    (A from TMEM, B = [Q content | Q RIB] tiles, MN-major, N = 48)
// and once per tile, when both halves of dS are in shared memory,
//     dQ~_I  = dS K~_J                      (A = dS, MN-major, B = [K | Pk] tiles, N = 48).
// Three buffers of S^T and dP^T rotate among the units.  P^T and dS^T are written over the scores that they come from, piece by piece,
// by the warp that has read them; S^T of unit u + 3 goes there once dV and dK~ have consumed unit u.  Two groups of arithmetic
// warps take the even and the odd half-tiles: while one group evaluates exponentials the other one's scores are
// being contracted, so neither the tensor pipe nor the exp pipe waits for a whole tile of the other.
// The RIB rows are fetched as zero-padded 64-byte rows, so that a RIB tile has the layout of a content
// tile and the concatenation of Eq. 5 is, for the MN-major operands, one descriptor whose second
// 32-column atom is the RIB tile: every contraction step is a single instruction.
// dQ~_I is one key block's share of the query gradient: it is added (fp32 red) into a workspace laid
// out [pair][group of 4 columns][token in window order][4] and finished by a small kernel that converts dq to
// bf16 and sums the RIB columns over pairs into dPq.  The RIB columns of dK~ are written per pair
// and summed over pairs by the same finishing kernel into dPk.
//
// Roles (896 threads at rank 16 on full windows, else 768): warp 0 TMA producer; three MMA-issuing warps (the tensor pipe takes
// instructions from several warps at once, and one thread issuing everything was the bottleneck):
// warp 1 issues S^T and dP^T, warp 2 (also the TMEM allocator) dV and dK~, warp 3 dQ~; warps 4-11
// P/dS arithmetic of the even half-tiles, warps 12-19 of the odd ones (a warp per 32 key rows and 32
// queries, a thread 2 key rows x 4 queries of each of its four 16 x 16 pieces); warps 20-23 drain dQ~ after every tile, they or warps
// 24-27 dK~/dV after every item.  Every wait is bounded.
// What sets the pace is the loop  scores -> arithmetic -> dV and dK~ -> next scores of the buffer  (1600 cycles of issue, contraction and
// barriers and 1350 of arithmetic), divided by the three units in flight: 2180 cycles per tile of 128 x 128 at rank 16, beside 1530 of
// tensor pipe and, replays included, nine tenths of the shared-memory data pipe.  Measured on 16 x 96 x 96 tokens in windows of 32,
// us at rank 16 / 32: scores, P^T and dS^T in buffers of their own, two of each 535 / 620; in place as above 515 / 640; dV and dK out by TMEM, shared
// memory and TMA before the item's last dQ~ 488 / 618; that and dQ~ drained in pieces of 16 columns without spills 468 / 565; S^T not
// waiting for dK~ at rank 32 468 / 550.  (At rank 16 the same costs 1 to 3 %; a third group of arithmetic warps, 64 registers each: 511.)
#include "rib_sm100_common.cuh"

namespace rib {
namespace {

using namespace sm100;

constexpr int kQStages = 4;           // ring of query-side tiles (Q content, Q RIB rows, dO, lse/D)
// Drains of dV and dK~ in warps of their own (24-27) beside those of dQ~: 466 -> 456 us on 16 x 96 x 96 tokens in windows of 32, 488 -> 474 on
// 10 x 64 x 64 in windows of 64.  At rank 32 and with partial windows the 72 registers that are then left per thread cost more (548
// against 555 us, masked windows of 32 123 against 136): there warps 20-23 do both.
template <int R, bool kPartial> constexpr bool kSplitDrains = R == 16 && !kPartial;
template <int R, bool kPartial> constexpr int kThreads = kSplitDrains<R, kPartial> ? 896 : 768;
// RIB rank R = 16 or 32 is a template argument of the kernels: dQ~ / dK~ have kD + R columns

// shared-memory map (offsets from a 1024-byte aligned base)
constexpr uint32_t kOffKc = 0;                                   // [2] key content (one slot per item in flight)
constexpr uint32_t kOffKp = kOffKc + 2 * kContentBytes;          // [2] key RIB rows, padded to 64 bytes
constexpr uint32_t kOffV = kOffKp + 2 * kContentBytes;           // [2] values
constexpr uint32_t kOffRing = kOffV + 2 * kContentBytes;
constexpr uint32_t kLdBytes = kTile * 8;                         // 64 query pairs x (-lse2, -lse2', -D, -D')
constexpr uint32_t kRingQc = 0, kRingQp = kContentBytes, kRingDO = kRingQp + kContentBytes, kRingLD = kRingDO + kContentBytes;
constexpr uint32_t kRingBytes = kRingLD + kLdBytes;              // 25600
constexpr uint32_t kOffDS = kOffRing + kQStages * kRingBytes;    // dS: [2 tiles][2 halves of 64 queries][128 keys][128 B], SWIZZLE_128B
constexpr uint32_t kDSHalf = kTile * 128;
constexpr uint32_t kOffDK = kOffDS + 4 * kDSHalf;                // dK rows of an item on their way out (dV rows leave through V's slot)
constexpr uint32_t kOffBar = kOffDK + kContentBytes;
// kSFull, kPReady, kPFree: unit mod 4 (on_unit); kDPFree: per half h (R = 32); kDSFree: per dS tile buffer.  The rule behind the split: a
// barrier's next phase must not be able to complete before every waiter has seen the current one, because a parity wait
// cannot tell "two phases ahead" from "not yet".  dQ~ of tile g waits for both halves' P^T / dS^T, but nothing that the arithmetic warps
// need for tile g + 1 depends on dQ~ of tile g; on the barriers of units 2 g, 2 g + 1 the next phases belong to tile g + 2, whose dS
// buffer is only released by dQ~ of tile g.  (tests/test_bwd_barriers.py is a model of these waits.)
enum Bar { kKVFull = 0, kKVEmpty = 2, kQFull = 4, kQEmpty = kQFull + kQStages, kSFull = kQEmpty + kQStages, kPReady = kSFull + 4,
           kPFree = kPReady + 4, kDPFree = kPFree + 4, kDSFree = kDPFree + 2, kDQFull = kDSFree + 2, kDQFree, kAccFull, kAccFree, kDrain,
           kNumBars = kDrain + 3 };
constexpr uint32_t kOffMisc = kOffBar + kNumBars * 8;
constexpr uint32_t kSmemBytes = kOffMisc + 16 + 1024;
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");
static_assert(kOffRing % 1024 == 0 && kRingBytes % 1024 == 0 && kOffDS % 1024 == 0, "swizzle atoms need aligned tiles");

// tensor-memory columns: S^T of unit u in buffer u mod 3 (64 fp32 columns), dP^T beside it (R = 16) or in buffer h of its half (R = 32, for which
// three do not fit); a warp writes P^T over its own scores (and, R = 16, dS^T over its dP^T): 32 queries in the first 16 of its 32 columns.
// R = 16: 3 x (S, dP) 0, dV 384, dK~ 416 (48), dQ~ 464 (48).
// R = 32: dK~ and dQ~ need 64 columns each, so dS^T is not kept in tensor memory (dK~ reads the dS tile in shared memory,
//         K-major): 3 x S 0, 2 x dP 192, dV 320, dK~ 352 (64), dQ~ 416 (64).
constexpr uint32_t kBuffers = 3;
template <int R> struct Cols {
    static constexpr uint32_t kStep = R == 16 ? 128 : 64, kColDP = R == 16 ? 64 : 192;      // between score buffers; dP^T of buffer / half 0
    static constexpr uint32_t kColDV = R == 16 ? 384 : 320, kColDK = kColDV + kD, kColDQ = kColDK + kD + R;
    static_assert(kColDQ + kD + R <= 512, "tensor memory has 512 columns");
};
constexpr uint32_t kTmemCols = 512;

constexpr uint32_t kIdescT32 = idesc_bf16_f32(kTile, kD, true);               // A in TMEM, B MN-major, N = 32
// dK~ (A in TMEM or K-major in shared memory, B MN-major) and dQ~ (A and B MN-major), N = kD + R
template <int R> struct Idesc {
    static constexpr uint32_t kT = idesc_bf16_f32(kTile, kD + R, true);
    static constexpr uint32_t kQ = idesc_bf16_f32_ab(kTile, kD + R, true, true);
};

struct BwdParams {
    const float2* ld;          // [pairs][n / 2] window order, per query pair: (-lse2, -lse2', -D, -D') as two float2
    float* dq_acc;             // [pairs][48 / 4][n][4] fp32, zeroed by the preparation kernel
    float* dkp;                // [pairs][16 / 4][n][4] fp32, RIB columns of dK~ (already times 1/sqrt d)
    int* status;
    int H, W, heads, M, s, n, nWy, nWx, nblk, items;
    int Hp, Wp;                // sides of the map the windows are laid over (H, W rounded up to multiples of M)
    int pos_per_head;          // 1 when Pq/Pk are head-wise: table index = head
    int masked;                // kPartial: shifted windows with a mask (a query sees the keys of its own part of a border window)
    float scale_log2;          // log2(e) / sqrt(d)
    float inv_sqrt_d;
    FastDiv div_nblk, div_heads, div_nwx, div_nwy, div_per_row;   // ..., M / 8
};

struct ItemCoord { int pair, b, wy, wx, h, J; };

__device__ __forceinline__ ItemCoord decode_item(const BwdParams& p, int item)
{
    ItemCoord c;
    p.div_nblk.divmod(item, c.pair, c.J);
    p.div_heads.divmod(c.pair, item, c.h);
    p.div_nwx.divmod(item, item, c.wx);
    p.div_nwy.divmod(item, c.b, c.wy);
    return c;
}

// kPartial: H or W is not a multiple of the window (but of 8); windows are laid over the map extended to Hp x Wp and
// an 8x8 patch of the extension holds no tokens.  TMA fills such patches with zeros; what is left to do: a key row that
// is no token gets P^T = dS^T = 0 (the 32 key rows of an arithmetic warp lie in one patch of 64, whose rows share the
// answer), a query that is no token reads -inf for -lse (written by the preparation kernel), i.e. probability 0,
// and nothing is stored for either.
template <int R, bool kPartial>
__global__ void __launch_bounds__(kThreads<R, kPartial>, 1)
rib_bwd_sm100_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
                     const __grid_constant__ CUtensorMap tm_pqs, const __grid_constant__ CUtensorMap tm_pk,
                     const __grid_constant__ CUtensorMap tm_dk, const __grid_constant__ CUtensorMap tm_dv, const BwdParams p)
{
    constexpr int kDk = kD + R;
    constexpr uint32_t kStep = Cols<R>::kStep, kColDP = Cols<R>::kColDP, kColDV = Cols<R>::kColDV, kColDK = Cols<R>::kColDK, kColDQ = Cols<R>::kColDQ;
    constexpr uint32_t kIdescSS = idesc_bf16_f32(kTile, kTile / 2, false);    // both operands K-major
    constexpr uint32_t kIdescT48 = Idesc<R>::kT, kIdescQ48 = Idesc<R>::kQ;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    auto bar = [&](int i) { return base + kOffBar + 8u * i; };
    // of kSFull, kPReady, kPFree: the barrier of a unit and the parity of its phase.  (Units -1 to -3 have the parity that a barrier without a
    // completed phase answers yes to.)
    auto on_unit = [&](int which, uint32_t unit) { return bar(which + (int)(unit & 3)); };
    auto unit_parity = [](uint32_t unit) { return (unit >> 2) & 1; };
    auto buffer_after = [](uint32_t buffer, uint32_t units) { buffer += units; return buffer >= kBuffers ? buffer - kBuffers : buffer; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + kOffMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + kOffMisc + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const WindowGeom geom{p.Hp, p.Wp, p.M, p.s};

    if (threadIdx.x == 0) {
        abort_flag[0] = 0; abort_flag[1] = 0;   // [1] stays 0: used by the drain waits
        for (int s = 0; s < 2; ++s) { mbar_init(bar(kKVFull + s), 1); mbar_init(bar(kKVEmpty + s), 5); }     // empty: the item's last dQ~, and V's slot by the four warps whose dV leaves through it
        for (int s = 0; s < kQStages; ++s) { mbar_init(bar(kQFull + s), 1); mbar_init(bar(kQEmpty + s), 1); }
        for (int h = 0; h < 2; ++h) {
            mbar_init(bar(kDPFree + h), 8);
            mbar_init(bar(kDSFree + h), R == 16 ? 1 : 2);     // R = 32: dK~ reads the dS tile as well as dQ~
        }
        for (int i = 0; i < 4; ++i) { mbar_init(bar(kSFull + i), 1); mbar_init(bar(kPReady + i), 8); mbar_init(bar(kPFree + i), 1); }
        mbar_init(bar(kDQFull), 1); mbar_init(bar(kDQFree), 4);
        mbar_init(bar(kAccFull), 1); mbar_init(bar(kAccFree), 4);
        for (int i = 0; i < 3; ++i) mbar_init(bar(kDrain + i), 1);
        fence_barrier_init();
        prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v);
        prefetch_tensormap(&tm_do); prefetch_tensormap(&tm_pqs); prefetch_tensormap(&tm_pk);
        prefetch_tensormap(&tm_dk); prefetch_tensormap(&tm_dv);
    }
    if (warp == 2) {
        tmem_alloc(base + kOffMisc, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ============================================================ TMA producer (one thread)
        if (lane == 0) {
            uint32_t g = 0, nitem = 0, kv_armed = 0, q_armed = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x, ++nitem) {
                const ItemCoord c = decode_item(p, item);
                const uint32_t slot = nitem & 1;
                if (nitem >= 2 && !mbar_wait(bar(kKVEmpty + slot), ((nitem >> 1) - 1) & 1, abort_flag, p.status)) { ok = false; break; }
                mbar_arrive_expect_tx(bar(kKVFull + slot), 3 * kContentBytes);
                ++kv_armed;
                for (int sub = 0; sub < 2; ++sub) {
                    int py, px, Y0, X0;
                    patch_origin(geom, p.div_per_row, c.wy, c.wx, 2 * c.J + sub, py, px, Y0, X0);
                    tma_load_5d(base + kOffKc + slot * kContentBytes + sub * kPatchContent, &tm_k, bar(kKVFull + slot),
                                0, c.h, X0, Y0, c.b);
                    tma_load_4d(base + kOffKp + slot * kContentBytes + sub * kPatchContent, &tm_pk, bar(kKVFull + slot), 0,
                                px, py, c.h * p.pos_per_head);
                    tma_load_5d(base + kOffV + slot * kContentBytes + sub * kPatchContent, &tm_v, bar(kKVFull + slot),
                                0, c.h, X0, Y0, c.b);
                }
                for (int I = 0; I < p.nblk; ++I, ++g) {
                    const uint32_t st = g % kQStages, use = g / kQStages;
                    if (use > 0 && !mbar_wait(bar(kQEmpty + st), (use - 1) & 1, abort_flag, p.status)) { ok = false; break; }
                    mbar_arrive_expect_tx(bar(kQFull + st), kRingBytes);
                    ++q_armed;
                    const uint32_t ring = base + kOffRing + st * kRingBytes;
                    for (int sub = 0; sub < 2; ++sub) {
                        int py, px, Y0, X0;
                        patch_origin(geom, p.div_per_row, c.wy, c.wx, 2 * I + sub, py, px, Y0, X0);
                        tma_load_5d(ring + kRingQc + sub * kPatchContent, &tm_q, bar(kQFull + st), 0, c.h, X0, Y0, c.b);
                        tma_load_4d(ring + kRingQp + sub * kPatchContent, &tm_pqs, bar(kQFull + st), 0,
                                    px, py, c.h * p.pos_per_head);
                        tma_load_5d(ring + kRingDO + sub * kPatchContent, &tm_do, bar(kQFull + st), 0, c.h, X0, Y0, c.b);
                    }
                    bulk_load_1d(ring + kRingLD, p.ld + (size_t)c.pair * p.n + (size_t)I * kTile, kLdBytes, bar(kQFull + st));
                }
            }
            if (!ok) {
                // Gave up: let the copies already in flight land before the CTA may exit.
                for (uint32_t b2 = kv_armed > 2u ? kv_armed - 2 : 0; b2 < kv_armed; ++b2)
                    mbar_wait(bar(kKVFull + (b2 & 1)), (b2 >> 1) & 1, abort_flag + 1, p.status);
                for (uint32_t b2 = q_armed > (uint32_t)kQStages ? q_armed - kQStages : 0; b2 < q_armed; ++b2)
                    mbar_wait(bar(kQFull + b2 % kQStages), (b2 / kQStages) & 1, abort_flag + 1, p.status);
            }
        }
    } else if (warp < 4) {
        // ============================================ MMA issuers: warps 1-3, the whole warp walks the
        // loops and waits (warp-uniform outcomes), one elected lane issues
        constexpr uint64_t kDesc64 = smem_desc_const(16, 512, kSwizzle64B);
        // MN-major operands of 48 columns: the content tile and, one leading-dimension step further, the RIB tile
        constexpr uint64_t kDescQ48 = smem_desc_const(kRingQp - kRingQc, 512, kSwizzle64B);
        constexpr uint64_t kDescK48 = smem_desc_const(kOffKp - kOffKc, 512, kSwizzle64B);
        constexpr uint64_t kDescDS = smem_desc_const(kDSHalf, 1024, kSwizzle128B);    // MN-major: the two 64-query halves one leading step apart
        constexpr uint64_t kDescDSk = smem_desc_const(16, 1024, kSwizzle128B);        // K-major view of one half (R = 32)
        const int nblk = p.nblk;
        const uint32_t total_tiles = (((uint32_t)p.items - blockIdx.x + gridDim.x - 1) / gridDim.x) * (uint32_t)nblk;
        const uint32_t total_units = 2 * total_tiles;       // half-tiles of this CTA, in order
        auto wait_all = [&](uint32_t b, uint32_t parity) { return mbar_wait_warp(b, parity, abort_flag, p.status); };
        bool ok = true;
        if (warp == 1) {
            // ---- S^T, dP^T of unit u as soon as dV and dK~ of unit u - 3 have consumed P^T, dS^T, which lie in the same columns; the
            // groups are then busy with units u - 1 and u - 2.  (R = 32: S^T after dV alone, dP^T when unit u - 2 has been read.)
            uint32_t nitem = 0, I = 0, buf = 0;
            uint32_t slot_base = 0;
            for (uint32_t u = 0; u < total_units && ok; ++u) {
                const uint32_t h = u & 1, g = u >> 1, st = g % kQStages, slot = nitem & 1;
                if (h == 0 && I == 0) {
                    if (!wait_all(bar(kKVFull + slot), (nitem >> 1) & 1)) { ok = false; break; }
                    slot_base = base + slot * kContentBytes;
                }
                if (h == 0 && !wait_all(bar(kQFull + st), (g / kQStages) & 1)) { ok = false; break; }
                if (!wait_all(on_unit(kPFree, u - kBuffers), unit_parity(u - kBuffers))) { ok = false; break; }
                tc_fence_after();
                const uint32_t ring = base + kOffRing + st * kRingBytes + h * kPatchContent;   // rows of patch h
                const uint64_t kc = smem_desc_at(kDesc64, slot_base + kOffKc), kp = smem_desc_at(kDesc64, slot_base + kOffKp);
                const uint64_t v = smem_desc_at(kDesc64, slot_base + kOffV);
                const uint64_t qc = smem_desc_at(kDesc64, ring + kRingQc), qp = smem_desc_at(kDesc64, ring + kRingQp);
                const uint64_t go = smem_desc_at(kDesc64, ring + kRingDO);
                const uint32_t d_s = tmem + kStep * buf, d_p = R == 16 ? d_s + kColDP : tmem + kColDP + 64 * h;
                if (elect_one()) {
                    mma_ss(d_s, kc, qc, kIdescSS, 0u);
                    mma_ss(d_s, kc + 2, qc + 2, kIdescSS, 1u);     // + 32 bytes: second K16 step
                    mma_ss(d_s, kp, qp, kIdescSS, 1u);
                    if (R == 32) mma_ss(d_s, kp + 2, qp + 2, kIdescSS, 1u);
                }
                if (R == 32) {
                    __syncwarp();
                    if (!wait_all(bar(kDPFree + h), (g - 1) & 1)) { ok = false; break; }
                    tc_fence_after();
                }
                if (elect_one()) {
                    mma_ss(d_p, v, go, kIdescSS, 0u);
                    mma_ss(d_p, v + 2, go + 2, kIdescSS, 1u);
                    mma_commit(on_unit(kSFull, u));
                }
                __syncwarp();
                buf = buffer_after(buf, 1);
                if (h == 1 && ++I == (uint32_t)nblk) { I = 0; ++nitem; }
            }
        } else if (warp == 2) {
            // ---- dV_J += P^T dO_u and dK~_J += dS^T Q~_u (A from tensor memory, 16 queries per step)
            uint32_t nitem = 0, I = 0, buf = 0;
            for (uint32_t u = 0; u < total_units && ok; ++u) {
                const uint32_t h = u & 1, g = u >> 1, st = g % kQStages;
                const bool first = I == 0 && h == 0, last = I == (uint32_t)nblk - 1 && h == 1;
                if (!wait_all(on_unit(kPReady, u), unit_parity(u)) ||
                    (first && nitem > 0 && !wait_all(bar(kAccFree), (nitem - 1) & 1))) { ok = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t ring = base + kOffRing + st * kRingBytes + h * kPatchContent;
                    const uint64_t go = smem_desc_at(kDesc64, ring + kRingDO);
                    const uint64_t q48 = smem_desc_at(kDescQ48, ring + kRingQc);
                    const uint32_t a_p = tmem + kStep * buf;          // 16 queries a step: the first 16 of every 32 columns
#pragma unroll
                    for (int kk = 0; kk < kTile / 32; ++kk)
                        mma_ts(tmem + kColDV, a_p + 32 * (kk >> 1) + 8 * (kk & 1), go + 64 * kk, kIdescT32, (kk || !first) ? 1u : 0u);
                    if (R == 32) mma_commit(on_unit(kPFree, u));      // S^T of unit u + 3 need not wait for dK~ as well
                    if (R == 16) {
                        const uint32_t a_ds = a_p + kColDP;
#pragma unroll
                        for (int kk = 0; kk < kTile / 32; ++kk)
                            mma_ts(tmem + kColDK, a_ds + 32 * (kk >> 1) + 8 * (kk & 1), q48 + 64 * kk, kIdescT48, (kk || !first) ? 1u : 0u);
                    } else {
                        // A = this half of the dS tile in shared memory, read K-major: rows are keys, the 128-byte lines the
                        // unit's 64 queries (32 bytes per K16 step)
                        const uint64_t a_ds = smem_desc_at(kDescDSk, base + kOffDS + ((g & 1) * 2 + h) * kDSHalf);
#pragma unroll
                        for (int kk = 0; kk < kTile / 32; ++kk)
                            mma_ss(tmem + kColDK, a_ds + 2 * kk, q48 + 64 * kk, kIdescT48, (kk || !first) ? 1u : 0u);
                        if (h == 1) mma_commit(bar(kDSFree + (g & 1)));
                    }
                    if (R == 16) mma_commit(on_unit(kPFree, u));
                    // the tile's query-side rows may go: S^T, dP^T of both halves finished before P^T existed
                    if (h == 1) mma_commit(bar(kQEmpty + st));
                    if (last) mma_commit(bar(kAccFull));
                }
                __syncwarp();
                buf = buffer_after(buf, 1);
                if (h == 1 && ++I == (uint32_t)nblk) { I = 0; ++nitem; }
            }
        } else if (warp == 3) {
            // ---- dQ~_I = dS K~_J once both halves of dS are in shared memory (16 keys per step)
            uint32_t nitem = 0, I = 0;
            for (uint32_t g = 0; g < total_tiles && ok; ++g) {
                if (!wait_all(on_unit(kPReady, 2 * g), unit_parity(2 * g)) || !wait_all(on_unit(kPReady, 2 * g + 1), unit_parity(2 * g)) ||
                    (g > 0 && !wait_all(bar(kDQFree), (g - 1) & 1))) { ok = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t k48 = smem_desc_at(kDescK48, base + kOffKc + (nitem & 1) * kContentBytes);
                    const uint64_t ds = smem_desc_at(kDescDS, base + kOffDS + (g & 1) * 2 * kDSHalf);
#pragma unroll
                    for (int kk = 0; kk < kTile / 16; ++kk)
                        mma_ss(tmem + kColDQ, ds + 128 * kk, k48 + 64 * kk, kIdescQ48, kk ? 1u : 0u);
                    mma_commit(bar(kDSFree + (g & 1)));
                    mma_commit(bar(kDQFull));
                    // K~_J and V_J may go once the item's last dQ~ is done (S^T, dP^T finished before it)
                    if (I == (uint32_t)nblk - 1) mma_commit(bar(kKVEmpty + (nitem & 1)));
                }
                __syncwarp();
                if (++I == (uint32_t)nblk) { I = 0; ++nitem; }
            }
        }
        // everything issued by this warp must have finished before TMEM is released
        if (elect_one()) mma_commit(bar(kDrain + warp - 1));
        __syncwarp();
        mbar_wait(bar(kDrain + warp - 1), 0, abort_flag + 1, p.status);
    } else if (warp >= 4 && warp < 20) {
        // ===== P^T and dS^T: group h = warps 4 + 8h .. 11 + 8h takes half-tile (I, h), a warp 32 key rows and 32 queries
        const int h = (warp - 4) >> 3;
        const int cg = ((warp - 4) >> 2) & 1;                // queries 32 cg .. 32 cg + 31 of the half-tile
        const int quarter = warp & 3;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
        uint32_t g = 0;
        bool ok = true;
        uint32_t buf = h;
        for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
            bool key_exists = true;       // kPartial: this warp's 32 key rows lie in one 8x8 patch of the key block
            int key_part = 0, last_window = 0;   // masked shifted windows: part of the key patch; bit 1 / 0: last window row / column
            if (kPartial) {
                const ItemCoord c = decode_item(p, item);
                int py, px, Y0, X0;
                patch_origin(geom, p.div_per_row, c.wy, c.wx, 2 * c.J + (quarter >> 1), py, px, Y0, X0);
                key_exists = Y0 < p.H && X0 < p.W;
                last_window = (c.wy == p.nWy - 1 ? 2 : 0) | (c.wx == p.nWx - 1 ? 1 : 0);
                key_part = window_part(p.M, p.s, last_window & 2, last_window & 1, py, px);
            }
            for (int I = 0; I < p.nblk; ++I, ++g) {
                // the 64 queries of this half-tile are one 8x8 patch as well: with a mask, one answer per warp and half-tile
                bool key_real = key_exists;
                if (kPartial && p.masked) {
                    const int per_row = p.M >> 3, qp = 2 * I + h;
                    key_real = key_exists && key_part == window_part(p.M, p.s, last_window & 2, last_window & 1, (qp / per_row) << 3, (qp % per_row) << 3);
                }
                const uint32_t st = g % kQStages;
                const uint32_t t_s = tmem + lane_base + 32 * cg + kStep * buf, t_dp = R == 16 ? t_s + kColDP : tmem + lane_base + 32 * cg + kColDP + 64 * h;
                buf = buffer_after(buf, 2);
                // warp-uniform outcome: the TMEM accesses below are warp-collective
                if (!mbar_wait_warp(on_unit(kSFull, 2 * g + h), unit_parity(2 * g), abort_flag, p.status) ||
                    !mbar_wait_warp(bar(kQFull + st), (g / kQStages) & 1, abort_flag, p.status)) { ok = false; break; }
                tc_fence_after();
                // The warp's 32 key rows x 32 queries in four pieces of 16 x 16 (piece c: lanes 16 (c % 2) .., queries 16 (c / 2) ..), read as
                // 16-lane fragments: a thread holds 2 key rows of 4 queries of a piece, and the per-query (-lse2, -lse2', -D, -D') cost
                // it 16 words per unit instead of 64.  What these warps share with the operand fetches of the MMAs is the one shared-memory
                // data pipe (840 of its passes per tile of 128 x 128 are theirs, 410 the adds' and stores', 992 the MMAs').  With four-byte columns in planes of
                // their own these reads take as many passes and more instructions (515 against 511 us).
                const uint32_t ld = base + kOffRing + st * kRingBytes + kRingLD + (32 * h + 16 * cg + (lane & 3)) * 16;
                auto ldq = [&](int gq) { return make_float4(lds_f32(ld + 64 * gq), lds_f32(ld + 64 * gq + 4), lds_f32(ld + 64 * gq + 8), lds_f32(ld + 64 * gq + 12)); };
                const uint32_t ds_line = base + kOffDS + ((g & 1) * 2 + h) * kDSHalf + (quarter * 32 + 8 * ((lane >> 3) & 1) + (lane & 7)) * 128;
                auto load = [&](int c, uint32_t (&s)[8], uint32_t (&dp)[8]) {
                    const uint32_t at = ((uint32_t)(16 * (c & 1)) << 16) + 16 * (c >> 1);
                    tmem_ld_16x256b_x2(t_s + at, s);
                    tmem_ld_16x256b_x2(t_dp + at, dp);
                };
                auto work = [&](const uint32_t (&s)[8], const uint32_t (&dp)[8], const float4 (&t)[2], uint32_t (&pp)[4], uint32_t (&dd)[4]) {
#pragma unroll
                    for (int gq = 0; gq < 2; ++gq)
#pragma unroll
                        for (int rr = 0; rr < 2; ++rr) {                  // key rows lane / 4 and lane / 4 + 8 of the fragment
                            const int i = 4 * gq + 2 * rr;
                            const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[i]), __uint_as_float(s[i + 1])), scale2, make_float2(t[gq].x, t[gq].y));
                            const float2 e = make_float2(ex2_approx(x.x), ex2_approx(x.y));
                            const float2 d = __fmul2_rn(e, __fadd2_rn(make_float2(__uint_as_float(dp[i]), __uint_as_float(dp[i + 1])), make_float2(t[gq].z, t[gq].w)));
                            pp[2 * gq + rr] = pack_bf16x2(e.x, e.y);
                            dd[2 * gq + rr] = pack_bf16x2(d.x, d.y);
                        }
                };
                // dS tile: row = key, 128-byte line = the unit's 64 queries, 16-byte chunks swizzled by the row.  An 8 x 8 block of the
                // fragment (8 key rows, 8 queries = one chunk) is what stmatrix stores: lanes 8 m .. 8 m + 7 name the rows of block
                // m = (chunk m / 2 of the piece, rows 8 (m % 2) ..)
                auto store = [&](int c, const uint32_t (&pp)[4], const uint32_t (&dd)[4]) {
                    const uint32_t at = ((uint32_t)(16 * (c & 1)) << 16) + 8 * (c >> 1);
                    tmem_st_16x128b_x2(t_s + at, pp);
                    if (R == 16) tmem_st_16x128b_x2(t_dp + at, dd);
                    stmatrix_x4(ds_line + 16 * (c & 1) * 128 + (((cg * 4 + 2 * (c >> 1) + (lane >> 4)) ^ (lane & 7)) << 4), dd[0], dd[1], dd[2], dd[3]);
                };
                // dQ~ of the tile before the previous one still reads this dS buffer.  (A barrier that has completed no phase answers yes to
                // parity 1, which the first tiles ask for.)
                const uint32_t b_ds = bar(kDSFree + (g & 1)), ds_parity = ((g >> 1) - 1) & 1;
                // R = 32: dP^T of this half is in registers, the next unit's may overwrite it
                auto dp_free = [&] {
                    if (R == 16) return;
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kDPFree + h));
                };
                uint32_t pp[4], dd[4];
                if (kPartial && !key_real) {
                    // nothing of this warp's key rows meets this half-tile's queries (no tokens, or another part of a masked
                    // window): P^T = dS^T = 0 without reading the scores
                    dp_free();
                    if (!mbar_wait_warp(b_ds, ds_parity, abort_flag, p.status)) { ok = false; break; }
#pragma unroll
                    for (int e = 0; e < 4; ++e) pp[e] = dd[e] = 0u;
#pragma unroll
                    for (int c = 0; c < 4; ++c) store(c, pp, dd);
                } else {
                    // a piece is stored while the next but one is on its way, over scores that this warp has read (all pieces together at the
                    // end: 537 against 515 us; the next unit's scores asked for ahead, before the arrival: 517)
                    uint32_t s0[8], dp0[8], s1[8], dp1[8];
                    float4 ta[2], tb[2];
                    const bool ds_free = mbar_try_wait(b_ds, ds_parity);
                    load(0, s0, dp0);
                    load(1, s1, dp1);
                    ta[0] = ldq(0); ta[1] = ldq(1);                         // queries 8 gq + 2 (lane % 4), + 1
                    tmem_wait_ld();
                    work(s0, dp0, ta, pp, dd);
                    if (!__all_sync(0xffffffffu, ds_free) && !mbar_wait_warp(b_ds, ds_parity, abort_flag, p.status)) { ok = false; break; }
                    load(2, s0, dp0);
                    store(0, pp, dd);
                    tb[0] = ldq(2); tb[1] = ldq(3);
                    work(s1, dp1, ta, pp, dd);
                    tmem_wait_ld();
                    load(3, s1, dp1);
                    store(1, pp, dd);
                    work(s0, dp0, tb, pp, dd);
                    tmem_wait_ld();
                    dp_free();
                    store(2, pp, dd);
                    work(s1, dp1, tb, pp, dd);
                    store(3, pp, dd);
                }
                tmem_wait_st();
                tc_fence_before();
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(on_unit(kPReady, 2 * g + h));
            }
        }
    } else if (warp >= 20) {
        // ================================ drains: dQ~ after every tile, dV / dK~ after every item
        constexpr bool kSplit = kSplitDrains<R, kPartial>;
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        auto drain_item = [&](int item, uint32_t nitem) -> bool {
            // Rows of 64 bytes, one per thread, would touch 32 lines with every store instruction and hold up the queue that all warps' loads and stores go
            // through for 2000 cycles an item; so they leave by TMA, a warp's 32 rows (half a patch) at a time (510 -> 488 us
            // on 16 x 96 x 96 tokens in windows of 32).  Each tile goes to shared memory before the next load: held back until the
            // accumulators are released, its rows spill.
            const ItemCoord c = decode_item(p, item);
            int py, px, Y0, X0;
            patch_origin(geom, p.div_per_row, c.wy, c.wx, 2 * c.J + (quarter >> 1), py, px, Y0, X0);
            const bool rows_real = !kPartial || (Y0 < p.H && X0 < p.W);   // no dk / dv rows for positions beyond the image
            if (!mbar_wait_warp(bar(kAccFull), nitem & 1, abort_flag, p.status)) return false;
            tc_fence_after();
            const int sw = (row >> 1) & 3;                    // SWIZZLE_64B
#pragma unroll
            for (int which = 0; which < 2; ++which) {         // dV through V's slot, dK through a tile of its own
                uint8_t* const stage = base_ptr + (which == 0 ? kOffV + (nitem & 1) * kContentBytes : kOffDK) + row * 64;
                const float f = which == 0 ? 1.f : p.inv_sqrt_d;
                uint32_t a[32];
                tmem_ld32(tmem + lane_base + (which == 0 ? kColDV : kColDK), a);
                tmem_wait_ld();
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) w[e] = pack_bf16x2(__uint_as_float(a[8 * q + 2 * e]) * f, __uint_as_float(a[8 * q + 2 * e + 1]) * f);
                    *reinterpret_cast<uint4*>(stage + ((q ^ sw) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            uint32_t rib[R / 16][16];
#pragma unroll
            for (int part = 0; part < R / 16; ++part) tmem_ld16(tmem + lane_base + kColDK + kD + 16 * part, rib[part]);
            tmem_wait_ld();
            tc_fence_before();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar(kAccFree));
                if (rows_real) {
                    tma_store_5d(&tm_dv, base + kOffV + (nitem & 1) * kContentBytes + quarter * (kPatchContent / 2), 0, c.h, X0, Y0 + 4 * (quarter & 1), c.b);
                    tma_store_5d(&tm_dk, base + kOffDK + quarter * (kPatchContent / 2), 0, c.h, X0, Y0 + 4 * (quarter & 1), c.b);
                    bulk_commit_group();
                }
            }
            float* dst_p = p.dkp + (size_t)c.pair * R * p.n + 4 * ((size_t)c.J * kTile + row);
#pragma unroll
            for (int col = 0; col < R; col += 4) {
                const uint32_t* v = rib[col >> 4] + (col & 15);
                *reinterpret_cast<float4*>(dst_p + (size_t)col * p.n) = make_float4(__uint_as_float(v[0]) * p.inv_sqrt_d, __uint_as_float(v[1]) * p.inv_sqrt_d,
                                                                                    __uint_as_float(v[2]) * p.inv_sqrt_d, __uint_as_float(v[3]) * p.inv_sqrt_d);
            }
            return true;
        };
        auto release_slot = [&](uint32_t nitem) {         // V's slot, when its dV rows have been read
            if (lane == 0) {
                bulk_wait_group_read<0>();                // (this thread's own stores)
                mbar_arrive(bar(kKVEmpty + (nitem & 1)));
            }
            __syncwarp();
        };
        auto drain_tile = [&](int item, int I, uint32_t g) -> bool {
            if (!mbar_wait_warp(bar(kDQFull), g & 1, abort_flag, p.status)) return false;
            tc_fence_after();
            float* dst = p.dq_acc + (size_t)p.div_nblk.div(item) * kDk * p.n + 4 * ((size_t)I * kTile + row);
#pragma unroll
            for (int part = 0; part < kDk / 16; ++part) {
                uint32_t a[16];
                tmem_ld16(tmem + lane_base + kColDQ + 16 * part, a);
                tmem_wait_ld();
                if (part + 1 == kDk / 16) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kDQFree));
                }
#pragma unroll
                for (int col = 0; col < 16; col += 4) {
                    // The adds of a tile in one burst fill the queue that all warps' loads, stores and fences go through: a pause after each one, at
                    // rank 32 after every second one, spreads them over the tile's time (16 x 96 x 96 tokens in windows of 32: no pause
                    // 502 / 589 us at rank 16 / 32, 20 ns 468 / 568, 40 ns 488 / 565).
                    red_add_f32x4(dst, a + col);
                    dst += 4 * (size_t)p.n;
                    if (R == 16 || (col & 4)) __nanosleep(20);
                }
            }
            return true;
        };
        uint32_t g = 0, nitem = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x, ++nitem) {
            if (kSplit && warp >= 24) {
                ok = drain_item(item, nitem);
                if (ok) release_slot(nitem);
                continue;
            }
            for (int I = 0; I < p.nblk && ok; ++I, ++g) {
                // (dV and dK~ before the item's last dQ~: dV and dK~ of the next item wait for the accumulators)
                if (!kSplit && I == p.nblk - 1) ok = drain_item(item, nitem);
                ok = ok && drain_tile(item, I, g);
            }
            if (!kSplit && ok) release_slot(nitem);
        }
        if (lane == 0) bulk_wait_group<0>();
        __syncwarp();
    }
    // ================================================================================ common tail
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------------------------ preparation and finishing
struct AuxParams {
    const __nv_bfloat16* out;
    const __nv_bfloat16* dout;
    const __nv_bfloat16* pq;
    const float* lse;
    float2* ld;
    float* dq_acc;
    const float* dkp;
    __nv_bfloat16* pq_scaled;
    __nv_bfloat16* dq;
    float* dpq;
    float* dpk;
    int H, W, heads, M, s, n, nWy, nWx, pairs;
    int d, r;                    // head width and rank of the caller's tensors (the accumulators are 32 + R columns wide)
    int dq_sectors;              // 1: 16 channels of a row of dq are one 32-byte sector
    int narrow;                  // kNarrow: width of the rows of out and dq (even, less than d)
    int Hp, Wp;                  // sides of the extended map (equal to H, W when they are multiples of the window)
    int tables;                  // Pq/Pk tables: 1 (shared by the heads) or heads
    long long pos_head_stride;   // elements between the tables in pq, dpq, dpk (pq_scaled is packed: n * 16 apart)
    float pos_scale, inv_sqrt_d, inv_sqrt_r;
};

// Returns false for a window position beyond the image (maps that are not multiples of the window): no token there.
__device__ __forceinline__ bool decode_pair_token(const AuxParams& p, int pair, int w, int& i, size_t& tok, size_t& scalar)
{
    const int h = pair % p.heads; pair /= p.heads;
    const int wx = pair % p.nWx; pair /= p.nWx;
    const int wy = pair % p.nWy; pair /= p.nWy;
    const int b = pair;
    int Y, X;
    window_order_token(WindowGeom{p.Hp, p.Wp, p.M, p.s}, wy, wx, w, i, Y, X);
    tok = (((size_t)b * p.H + Y) * p.W + X) * p.heads + h;
    scalar = (((size_t)b * p.heads + h) * p.H + Y) * p.W + X;
    return Y < p.H && X < p.W;
}

// Four lanes per (pair, token in window order), 8 channels each (a row per lane touches 32 lines with every load: 16 x 96 x 96 tokens, rank 16,
// 56 -> 48 us = 6.2 TB/s; 10 x 64 x 64 21 -> 17): D = dO . O and lse in the layout the main kernel
// streams; the dQ~ accumulators are cleared with 16-byte stores, (d + r) / 16 per lane, as one flat array;
// the first threads also stage bf16(Pq sqrt(d/r)) and clear dPq, dPk.
// kNarrow: the rows of out are p.narrow < d elements wide and aligned to 4 bytes only.
template <int R, bool kNarrow>
__global__ void __launch_bounds__(256) rib_bwd_prepare_kernel(const AuxParams p)
{
    constexpr int kDk = kD + R;
    const size_t total = (size_t)p.pairs * p.n;
    const size_t thread = (size_t)blockIdx.x * blockDim.x + threadIdx.x, t = thread >> 2;
    const int part = (int)(thread & 3);
    const size_t nthreads = (size_t)gridDim.x * blockDim.x;
    // staged rows are R wide (zeros from column r on), the caller's tables r wide
    const size_t per_table = (size_t)p.n * R;
    for (size_t e = thread; e < per_table * p.tables; e += nthreads) {
        const size_t tbl = e / per_table, rem = e % per_table;
        const int row = (int)(rem / R), col = (int)(rem % R);
        if (col < p.r) {
            const size_t user = tbl * (size_t)p.pos_head_stride + (size_t)row * p.r + col;
            p.pq_scaled[e] = __float2bfloat16_rn(__bfloat162float(p.pq[user]) * p.pos_scale);
            p.dpq[user] = 0.f;
            p.dpk[user] = 0.f;
        } else {
            p.pq_scaled[e] = __float2bfloat16_rn(0.f);
        }
    }
    if (t >= total) return;                                // (whole warps: total is a multiple of 128)
    const int pair = (int)(t / p.n), w = (int)(t % p.n);
    int i; size_t tok, scalar;
    const bool real = decode_pair_token(p, pair, w, i, tok, scalar);
    uint4 x = make_uint4(0u, 0u, 0u, 0u), y = x;
    float lse = 0.f;
    if (real && 8 * part < p.d) {
        x = __ldg(reinterpret_cast<const uint4*>(p.dout + tok * p.d) + part);
        if (kNarrow) {
            const uint32_t* v = reinterpret_cast<const uint32_t*>(p.out + tok * p.narrow) + 4 * part;
            const int left = p.narrow - 8 * part;
            if (left > 0) y.x = __ldg(v);
            if (left > 2) y.y = __ldg(v + 1);
            if (left > 4) y.z = __ldg(v + 2);
            if (left > 6) y.w = __ldg(v + 3);
        } else {
            y = __ldg(reinterpret_cast<const uint4*>(p.out + tok * p.d) + part);
        }
        if (part == 0) lse = p.lse[scalar];
    }
    float4* z4 = reinterpret_cast<float4*>(p.dq_acc);      // pairs * (d + r) * n floats = total * kDk / 4 vectors
#pragma unroll
    for (int k = 0; k < kDk / 16; ++k) z4[(size_t)k * 4 * total + thread] = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        acc = fmaf(__uint_as_float(xs[k] << 16), __uint_as_float(ys[k] << 16), acc);
        acc = fmaf(__uint_as_float(xs[k] & 0xffff0000u), __uint_as_float(ys[k] & 0xffff0000u), acc);
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (part == 0) {
        // a position beyond the image: as a query it gets probability 0 (exp2(-inf)) and D = 0
        float* ldf = reinterpret_cast<float*>(p.ld) + ((t >> 1) << 2) + (t & 1);
        ldf[0] = real ? -lse * 1.4426950408889634f : -INFINITY;
        ldf[2] = real ? -acc : 0.f;
    }
}

// Finishing pass over the fp32 accumulators.  grid (n / 32, groups of pairs), 32 x (2 + R / 8) threads: a thread owns one token position w
// of the window and either 16 of the 32 content columns of dQ~ (one 32-byte sector of the bf16 dq row) or 8 RIB columns of dQ~ and
// of dK~, four 16-byte reads per pair in both cases, and walks the pairs of its group.  Few registers per thread keep the SM full
// of warps, which is what this kernel (a stream of 16-byte reads, 512 bytes per warp) needs to reach the memory system.  With one
// table for all heads a group is a run of consecutive pairs; with head-wise tables it is a run of windows of
// one head (pair = head + heads * window), so that its sums belong to one table.  Per pair a content thread turns its
// piece of dQ~[:, :d] / sqrt(d) into bf16; a RIB thread keeps running sums of its columns of dQ~ (-> dPq, times
// 1/sqrt(r)) and of dK~ (-> dPk), and sends the group's sums to the zeroed results with vector atomics (these
// adds all land on the same n x r addresses: a group is long enough that their number does not set the time).
template <int R, bool kNarrow>       // kNarrow: the rows of dq are p.narrow < d elements wide
__global__ void __launch_bounds__(32 * (2 + R / 8)) rib_bwd_finish_kernel(const AuxParams p, int pairs_per_group)
{
    constexpr int kDk = kD + R;
    const int tx = threadIdx.x & 31, cg = threadIdx.x >> 5;
    const int w = blockIdx.x * 32 + tx;
    int pair0, pair1, step = 1;
    size_t table = 0;
    if (p.tables == 1) {
        pair0 = blockIdx.y * pairs_per_group;
        pair1 = min(p.pairs, pair0 + pairs_per_group);
    } else {
        const int head = blockIdx.y % p.heads, first = (blockIdx.y / p.heads) * pairs_per_group;
        step = p.heads;
        pair0 = head + first * step;
        pair1 = min(p.pairs, pair0 + pairs_per_group * step);
        table = (size_t)head * (size_t)p.pos_head_stride;
    }
    int i = 0;
    size_t tok, scalar;
    if (cg < 2) {                                            // 16 content columns
        const int channels = min(16, (kNarrow ? p.narrow : p.d) - 16 * cg);
        if (channels <= 0) return;
        if (kNarrow) {
            // A warp's 32 positions are 4 x 8 tokens, all in the map or none.  Its words change lanes through shared memory, so that a store
            // covers 4 rows in runs of up to 32 bytes: one row per lane, every store touched 32 lines
            // (8 x 96 x 96 tokens, 30 channels, rank 18 55.8 -> 43.5 us; one warp for both halves of the columns, two rows to a store: 88).
            __shared__ uint32_t staged[2][32 * 9];
            uint32_t* const mine = staged[cg];
            const int words = p.narrow / 2, word = tx & 7;
            auto load = [&](int pair, float4 (&to)[4]) {
                const float4* src = reinterpret_cast<const float4*>(p.dq_acc + (size_t)pair * kDk * p.n) + (size_t)(4 * cg) * p.n + w;
#pragma unroll
                for (int q = 0; q < 4; ++q) to[q] = 4 * q < channels ? src[(size_t)q * p.n] : make_float4(0.f, 0.f, 0.f, 0.f);
            };
            float4 f[4], ahead[4];
            load(pair0, f);
            for (int pair = pair0; pair < pair1; pair += step) {
                if (pair + step < pair1) load(pair + step, ahead);
                if (decode_pair_token(p, pair, w, i, tok, scalar)) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        mine[tx * 9 + 2 * q] = pack_bf16x2(f[q].x * p.inv_sqrt_d, f[q].y * p.inv_sqrt_d);
                        mine[tx * 9 + 2 * q + 1] = pack_bf16x2(f[q].z * p.inv_sqrt_d, f[q].w * p.inv_sqrt_d);
                    }
                    __syncwarp();
                    const size_t first = tok - (size_t)((tx >> 3) * p.W + (tx & 7)) * p.heads;
                    uint32_t* const dst = reinterpret_cast<uint32_t*>(p.dq) + (first + (size_t)(tx >> 3) * p.heads) * words + 8 * cg + word;
#pragma unroll
                    for (int four = 0; four < 8; ++four)
                        if (2 * word < channels)
                            dst[(size_t)((four >> 1) * p.W + 4 * (four & 1)) * p.heads * words] = mine[(4 * four + (tx >> 3)) * 9 + word];
                    __syncwarp();
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) f[q] = ahead[q];
            }
            return;
        }
#pragma unroll 2
        for (int pair = pair0; pair < pair1; pair += step) {
            if (!decode_pair_token(p, pair, w, i, tok, scalar)) continue;
            const float4* src = reinterpret_cast<const float4*>(p.dq_acc + (size_t)pair * kDk * p.n) + (size_t)(4 * cg) * p.n + w;
            float4 f[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) f[q] = 4 * q < channels ? src[(size_t)q * p.n] : make_float4(0.f, 0.f, 0.f, 0.f);
            uint32_t v[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[2 * q] = pack_bf16x2(f[q].x * p.inv_sqrt_d, f[q].y * p.inv_sqrt_d);
                v[2 * q + 1] = pack_bf16x2(f[q].z * p.inv_sqrt_d, f[q].w * p.inv_sqrt_d);
            }
            if (p.dq_sectors) {
                st_global_v8(p.dq + tok * p.d + 16 * cg, v);
            } else {
                uint4* dst = reinterpret_cast<uint4*>(p.dq + tok * p.d) + 2 * cg;
                dst[0] = make_uint4(v[0], v[1], v[2], v[3]);
                if (channels > 8) dst[1] = make_uint4(v[4], v[5], v[6], v[7]);
            }
        }
        return;
    }
    const int col0 = 8 * (cg - 2);                           // 8 of the R RIB columns
    if (col0 >= p.r) return;                                 // columns of the padding (ranks are multiples of 8)
    float4 sq[2], sk[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) sq[q] = sk[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [](float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; };
#pragma unroll 2
    for (int pair = pair0; pair < pair1; pair += step) {     // (the sums of a position beyond the image are zero)
        const float4* src = reinterpret_cast<const float4*>(p.dq_acc + (size_t)pair * kDk * p.n) + (size_t)((kD + col0) / 4) * p.n + w;
        const float4* srk = reinterpret_cast<const float4*>(p.dkp + (size_t)pair * R * p.n) + (size_t)(col0 / 4) * p.n + w;
#pragma unroll
        for (int q = 0; q < 2; ++q) { add(sq[q], src[(size_t)q * p.n]); add(sk[q], srk[(size_t)q * p.n]); }
    }
    // (the first pair of a group always exists: the grid is sized by the groups; i is the token's row of the tables)
    decode_pair_token(p, pair0, w, i, tok, scalar);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        atomicAdd(reinterpret_cast<float4*>(p.dpq + table + (size_t)i * p.r + col0 + 4 * q),
                  make_float4(sq[q].x * p.inv_sqrt_r, sq[q].y * p.inv_sqrt_r, sq[q].z * p.inv_sqrt_r, sq[q].w * p.inv_sqrt_r));
        atomicAdd(reinterpret_cast<float4*>(p.dpk + table + (size_t)i * p.r + col0 + 4 * q), sk[q]);
    }
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct WorkspaceLayout { size_t ld, dq_acc, dkp, pq_scaled, total; };

WorkspaceLayout workspace_layout(long long pairs, int n, int tables, int r)
{
    const int kR = padded_rank(r), kDk = kD + kR;      // the accumulators carry the padded rank
    WorkspaceLayout w;
    w.ld = 0;
    w.dq_acc = w.ld + align256((size_t)pairs * n * sizeof(float2));
    w.dkp = w.dq_acc + align256((size_t)pairs * kDk * n * sizeof(float));
    w.pq_scaled = w.dkp + align256((size_t)pairs * kR * n * sizeof(float));
    w.total = w.pq_scaled + align256((size_t)tables * n * kR * sizeof(__nv_bfloat16));
    return w;
}

}  // namespace

bool sm100_bwd_supported(const Problem& p)
{
    return p.d % 8 == 0 && p.d >= 8 && p.d <= sm100::kD && p.r % 8 == 0 && p.r >= 8 && p.r <= 32 &&
           (p.M % 16 == 0 || sm100_window8(p)) && p.s % 8 == 0 && p.M <= 256 && p.H % 8 == 0 && p.W % 8 == 0;
}

// (windows of 8 x 8 tokens need none of it; they keep the size, and with it what rib_window_attn_bwd_noalloc accepts)
size_t sm100_bwd_workspace_bytes(long long pairs, int n, int tables, int r) { return workspace_layout(pairs, n, tables, r).total; }

template <int R, bool kPartial>
cudaError_t launch_bwd(const Problem& p, cudaStream_t stream)
{
    if (!encode_fn()) return cudaErrorNotSupported;
    const int tables = pos_tables(p);
    const WorkspaceLayout wl = workspace_layout(p.pairs, p.n, tables, R);
    if (p.workspace_bytes < wl.total) return cudaErrorInvalidValue;
    uint8_t* ws = static_cast<uint8_t*>(p.workspace);
    float2* ld = reinterpret_cast<float2*>(ws + wl.ld);
    float* dq_acc = reinterpret_cast<float*>(ws + wl.dq_acc);
    float* dkp = reinterpret_cast<float*>(ws + wl.dkp);
    __nv_bfloat16* pq_scaled = reinterpret_cast<__nv_bfloat16*>(ws + wl.pq_scaled);

    CUtensorMap tm_q, tm_k, tm_v, tm_do, tm_pqs, tm_pk, tm_dk, tm_dv;
    if (!encode_image_map(&tm_q, p.q, p) || !encode_image_map(&tm_k, p.k, p) || !encode_image_map(&tm_v, p.v, p) ||
        !encode_image_map(&tm_do, p.dout, p) || !encode_pos_map_padded(&tm_pqs, pq_scaled, p, tables, (long long)p.n * R, R) ||
        !encode_pos_map_padded(&tm_pk, p.pk, p, tables, p.pos_head_stride, p.r) || !encode_image_map(&tm_dk, p.dk, p, 4) || !encode_image_map(&tm_dv, p.dv, p, 4))
        return cudaErrorInvalidValue;
    static KernelSetup setup;       // one per instantiation of this launcher, i.e. per kernel
    int sm_count = 0;
    if (cudaError_t e = setup.prepare(rib_bwd_sm100_kernel<R, kPartial>, kSmemBytes, &sm_count)) return e;
    AuxParams ap{};
    ap.out = p.out; ap.dout = p.dout; ap.pq = p.pq; ap.lse = p.lse_in;
    ap.ld = ld; ap.dq_acc = dq_acc; ap.dkp = dkp; ap.pq_scaled = pq_scaled;
    ap.dq = p.dq; ap.dpq = p.dpq; ap.dpk = p.dpk;
    ap.H = p.H; ap.W = p.W; ap.heads = p.heads; ap.M = p.M; ap.s = p.s; ap.n = p.n; ap.nWy = p.nWy; ap.nWx = p.nWx;
    ap.Hp = p.Hp; ap.Wp = p.Wp;
    ap.pairs = p.pairs;
    ap.d = p.d; ap.r = p.r; ap.narrow = p.narrow;
    ap.dq_sectors = p.d % 16 == 0 && (reinterpret_cast<uintptr_t>(p.dq) & 31u) == 0;
    ap.tables = tables;
    ap.pos_head_stride = p.pos_head_stride;
    ap.pos_scale = sqrtf(scale_width_d(p) / scale_width_r(p));
    ap.inv_sqrt_d = 1.f / sqrtf(scale_width_d(p));
    ap.inv_sqrt_r = 1.f / sqrtf(scale_width_r(p));
    const size_t tokens = (size_t)p.pairs * p.n;
    const unsigned aux_blocks = (unsigned)((tokens + 63) / 64);
    { ProfileScope scope(RIB_KERNEL_BWD_PREPARE, stream); (p.narrow ? rib_bwd_prepare_kernel<R, true> : rib_bwd_prepare_kernel<R, false>)<<<aux_blocks, 256, 0, stream>>>(ap); }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;

    BwdParams bp{};
    bp.ld = ld; bp.dq_acc = dq_acc; bp.dkp = dkp; bp.status = p.status;
    bp.H = p.H; bp.W = p.W; bp.heads = p.heads; bp.M = p.M; bp.s = p.s; bp.n = p.n; bp.nWy = p.nWy; bp.nWx = p.nWx;
    bp.Hp = p.Hp; bp.Wp = p.Wp;
    bp.nblk = p.n / kTile;
    bp.items = p.pairs * bp.nblk;
    bp.pos_per_head = tables > 1 ? 1 : 0;
    bp.masked = p.masked ? 1 : 0;
    bp.scale_log2 = 1.4426950408889634f / sqrtf(scale_width_d(p));
    bp.inv_sqrt_d = ap.inv_sqrt_d;
    bp.div_nblk = make_fast_div(bp.nblk); bp.div_heads = make_fast_div(p.heads); bp.div_nwx = make_fast_div(p.nWx); bp.div_nwy = make_fast_div(p.nWy);
    bp.div_per_row = make_fast_div(p.M >> 3);
    const int grid = bp.items < sm_count ? bp.items : sm_count;
    { ProfileScope scope(RIB_KERNEL_BWD_MAIN, stream); rib_bwd_sm100_kernel<R, kPartial><<<grid, kThreads<R, kPartial>, kSmemBytes, stream>>>(tm_q, tm_k, tm_v, tm_do, tm_pqs, tm_pk, tm_dk, tm_dv, bp); }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;

    const int windows = p.pairs / p.heads;   // pairs of one head
    const int in_line = tables == 1 ? p.pairs : windows;      // pairs whose sums go to one table
    // A block takes a run of pairs (of one head, with head-wise tables): four, or one where there are fewer than sixteen.  Measured, us with
    // the launch, for runs of 2 / 4 / 8 pairs: 864 pairs of 1024 tokens at rank 16 56 / 54 / 54, at rank 32 89 / 76 / 78, 1728 pairs at rank 32 117 / 101 /
    // 99, 60 pairs of 4096 tokens at rank 16 21 / 20 / 19; with a quarter of a token's columns per thread, 16-byte stores of dq and a pass of its
    // own for RIB columns 16 to 31 58, 88, 138 and 21 at runs of four.  Runs of eight where the grid's y has no room.
    auto groups_of = [&](int run) { return (tables == 1 ? 1ll : (long long)p.heads) * ((in_line + run - 1) / run); };
    const int per_group = in_line < 16 ? 1 : groups_of(4) <= 65535 ? 4 : 8;
    const unsigned groups = (unsigned)groups_of(per_group);
    dim3 grid_fin((unsigned)(p.n / 32), groups);
    { ProfileScope scope(RIB_KERNEL_BWD_FINISH, stream); (p.narrow ? rib_bwd_finish_kernel<R, true> : rib_bwd_finish_kernel<R, false>)<<<grid_fin, 32 * (2 + R / 8), 0, stream>>>(ap, per_group); }
    return cudaGetLastError();
}

bool sm100_bwd_takes_narrow(const Problem& p) { return !sm100_window8(p) && !sm100_window16(p); }

int sm100_bwd_launches(const Problem& p) { return sm100_window8(p) ? 2 : 3; }      // clear, main; else two clears, main or prepare, main, finish

cudaError_t sm100_bwd(const Problem& p, cudaStream_t stream)
{
    if (sm100_window8(p)) return sm100_window8_bwd(p, stream);
    if (sm100_window16(p)) return sm100_window16_bwd(p, stream);
    const bool wide = padded_rank(p.r) == 32;      // accumulators with 32 RIB columns (ranks 24 and 32), else 16 (ranks 8 and 16)
    if (p.Hp != p.H || p.Wp != p.W || p.masked) return wide ? launch_bwd<32, true>(p, stream) : launch_bwd<16, true>(p, stream);
    return wide ? launch_bwd<32, false>(p, stream) : launch_bwd<16, false>(p, stream);
}

}  // namespace rib
