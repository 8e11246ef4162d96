// Forward RIB window attention for B200 (sm_100a) on frames whose sides are not multiples of 8: tcgen05 MMAs, TMEM, TMA.
//
// These shapes are defined by the fp32 any-shape kernels (rib_generic.cu), which keep the probabilities, their sums and the
// scaled positional features in fp32.  This kernel stays close to that on the bf16 tensor cores by splitting what is not
// a bf16 number to begin with into bf16 terms:
//     P            = hi + lo           two terms, 16 significant bits: the PV contraction runs twice, into one accumulator;
//     Pq sqrt(d/r) = hi + mid + lo     three terms, all 24 bits: one K16 step (two at R = 32) of the score chain per term
//                                      (one term where d / r is a power of 4 and the product is a bf16 number);
// q, k, v and Pk are bf16 as given and enter exactly, sums are fp32, every exponential is ex2.approx (2 ulp), the row sum
// adds the unrounded fp32 probabilities.  Infinities: the terms of a number times an infinity may cancel to NaN where the number
// itself times it would not, so a row that comes out as NaN is computed once more from the plain numbers (plain_row).
//
// What bounds it: the serial program of the softmax warps, 3300 cycles per block of both query tiles of which the exp unit is busy
// 2048, beside 42 MMAs (2100 cycles of issue, from three warps).  Measured (180 x 320 tokens, 32 x 32 windows, 6 heads of 32
// channels, rank 16): 163 us a pass = 332 TFLOP/s of the layer's own flops (160 us on inputs that the pass before has read, too); one
// warp issuing everything 179 us (it held a unit for 16 + 5 MMAs and the wait between them, 1600 cycles), the any-shape kernel 13 460 us.
// Asking for the next scores before P is handed over, as the general kernel does, is 13 % slower: P then waits for them.
// Error of `out` against float64 as that kernel's (1.7e-3, the rounding to bf16; 4 parts in a million more at most), of lse below it.
//
// Work item = one (batch, window, head) pair x two query tiles of 128 tokens (two 8x8-token patches each).  Only patches that
// hold tokens are walked (LiveWindows in rib_sm100_common.cuh); a patch that straddles the border of the frame is filled up
// with zeros by TMA, its keys beyond the frame get the score -inf and its queries beyond it are not stored.
//
// Tensor memory: three score buffers of 128 columns and 2 x 2 output accumulators (query tile, key half) of 32.  Unit u =
// 2 * block + query tile uses buffer u mod 3.  A softmax thread holds one row's 64 scores of its key half in registers and
// writes P over them (hi 32 columns, lo 32 columns), so a buffer is handed back with P in it; S(u + 3) goes into the same columns
// once PV(u) has completed (nothing orders an MMA that overwrites columns behind one of another shape and accumulator that reads
// them as its A operand).  The scores of one tile's next block are thus under way while the other tile's exponentials run.
//
// Roles (640 threads): warp 0 TMA producer, which also stages the scaled query RIB rows; warp 1 issues S, warps 2 and 3
// PV of query tile 0 and 1 (warp 2 owns the TMEM allocation); warps 4-11 softmax / epilogue of query tile 0 (4-7 first key half, 8-11 second half), 12-19 of tile 1.
// Every wait is bounded.
#include "rib_sm100_common.cuh"

namespace rib {
namespace {

using namespace sm100;

constexpr int kThreads = 640;
constexpr int kTerms = 3;                 // bf16 terms of a scaled query RIB row
constexpr int kBuffers = 3;               // score / P buffers in tensor memory

// shared-memory map (offsets from a 1024-byte aligned base); RIB rows of 16 elements (32 bytes, SWIZZLE_32B) or 32 (SWIZZLE_64B)
template <int R>
struct Frame {
    static constexpr int kStages = R == 16 ? 4 : 3;                              // K / V ring: what fits
    static constexpr uint32_t kPos = kTile * R * 2, kPatchP = kPos / 2;
    static constexpr uint32_t kOffQc = 0;                                        // [2 items][2 tiles] query content
    static constexpr uint32_t kOffQp = kOffQc + 4 * kContentBytes;               // [2 items][2 tiles][kTerms] query RIB rows
    static constexpr uint32_t kOffKc = kOffQp + 4 * kTerms * kPos;               // [kStages] key content, key RIB rows, values
    static constexpr uint32_t kOffKp = kOffKc + kStages * kContentBytes;
    static constexpr uint32_t kOffV = kOffKp + kStages * kPos;
    static constexpr uint32_t kOffBar = kOffV + kStages * kContentBytes;
    // barriers: query buffers, ring stages, scores there, P there and PV completed (each 2 tile + parity of the block, on_block), merge per
    // tile and quarter of the rows, drain per issuing warp.  A parity wait cannot tell "a phase ahead" or "a phase behind" from its own,
    // so every barrier is one whose next phase needs what its waiters do after this one, and whose phase before they know to have
    // arrived: scores of a tile's block b + 2 need PV of block b, PV needs P, P the scores, and scores of block b are issued after PV
    // of block b - 2 was seen.  (Per buffer neither holds: the phase before belongs to the other tile.  Nor does it follow that a
    // commit has arrived when another one behind the same contractions has.  tests/test_frame_barriers.py is a model of it.)
    enum Bar { kQFull = 0, kQEmpty = 2, kQPos = 4, kFull = 6, kEmpty = kFull + kStages, kSFull = kEmpty + kStages, kPReady = kSFull + 4,
               kPVDone = kPReady + 4, kMerge = kPVDone + 4, kDrain = kMerge + 8, kNumBars = kDrain + 3 };
    static constexpr uint32_t kOffMisc = kOffBar + kNumBars * 8;                 // tmem base, abort flags
    static constexpr uint32_t kOffMerge = (kOffMisc + 16 + 15) & ~15u;           // [2 item parities][2 tiles][2 halves][128 rows] (max, sum)
    static constexpr uint32_t kSmemBytes = kOffMerge + 8 * kTile * 8 + 1024;     // + slack for manual alignment
    static_assert(kSmemBytes <= 232448, "shared memory of one CTA");
};

constexpr uint32_t kColO = kBuffers * kTile, kTmemCols = 512;                    // O: [2 tiles][2 key halves][32]
static_assert(kColO + 4 * kD <= kTmemCols, "tensor memory has 512 columns");

constexpr uint32_t kIdescS = idesc_bf16_f32(kTile, kTile, false);
constexpr uint32_t kIdescPV = idesc_bf16_f32(kTile, kD, true);

struct FrameParams {
    const __nv_bfloat16 *q, *k, *v, *pk;       // read by plain_row only
    const __nv_bfloat16* pq;
    __nv_bfloat16* out;
    float* lse;
    int* status;
    int H, W, heads, d, r;
    WindowGeom geom;           // sides of the extended map, window, shift
    int terms;                 // terms of the scaled query RIB rows in use: 1 or kTerms
    float scale_log2;          // log2(e) / sqrt(d)
    float rescale_threshold;   // raw-logit units: probabilities stay <= 2^8 relative to the reference.  (Here and not in a register of the softmax
                               // warps, which have none to spare: 161.4 -> 159.5 us on the map above, inputs read before.)
    float inv_sqrt_d, inv_sqrt_r;
    float pos_scale;           // sqrt(d / r): folds 1/sqrt(r) into the content scale
    long long pos_head_stride;
    int pos_per_head;
    LiveWindows live;
};

// ln(2^-n l), rounded once: the logarithm of l's mantissa is small, the rest is added up in double (once per row).  With logf(l)
// and a product in fp32, and the scores' steps the other way round, lse was 1.36 times as far from float64 as the any-shape
// kernel's (180 x 320 tokens, 32 x 32 windows: 4.1e-8 against 3.0e-8); now 2.4e-8.
__device__ __forceinline__ float log_sum(float n, float l)
{
    if (!(l > 0.f && l < INFINITY)) return -n + logf(l);             // no finite logit, or one that is no number
    const int k = ((int)__float_as_uint(l) - 0x3f3504f3) >> 23;      // l = 2^k f, f in [sqrt(1/2), sqrt(2))
    return (float)(((double)k - (double)n) * 0.69314718055994531 + (double)logf(__uint_as_float(__float_as_uint(l) - ((uint32_t)k << 23))));
}

// s plus the products of two rows of bf16 (16-byte aligned, widths are multiples of 8), the first scaled, in fp32
__device__ __forceinline__ float add_products(float s, const __nv_bfloat16* a, float scale, const __nv_bfloat16* b, int width)
{
    for (int e = 0; e < width; e += 8) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(a + e)), y = __ldg(reinterpret_cast<const uint4*>(b + e));
        const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            s = fmaf(__uint_as_float(xs[w] << 16) * scale, __uint_as_float(ys[w] << 16), s);
            s = fmaf(__uint_as_float(xs[w] & 0xffff0000u) * scale, __uint_as_float(ys[w] & 0xffff0000u), s);
        }
    }
    return s;
}

// The output row (16 channels) and lse of one query, as rib_generic.cu defines them: fp32, one number per factor.  Called for
// rows with a NaN only, by one thread per half.
__device__ __noinline__ void plain_row(const FrameParams* pp, int item, int row256, int half)
{
    const FrameParams& p = *pp;
    const LiveItem c = decode_live_item(p.live, item);
    auto place = [&](int patch, int in, int& table_row, size_t& token) {      // false: no token
        int py, px, Y0, X0;
        live_patch_origin(p.live, p.geom, c, patch, py, px, Y0, X0);
        const int Y = Y0 + (in >> 3), X = X0 + (in & 7);
        table_row = (py + (in >> 3)) * p.geom.M + px + (in & 7);
        token = (((size_t)c.b * p.H + Y) * p.W + X) * p.heads + c.h;
        return Y < p.H && X < p.W;
    };
    int i;
    size_t query;
    place(4 * c.tp + (row256 >> 6), row256 & 63, i, query);
    const __nv_bfloat16 *pq = p.pq + (size_t)c.h * p.pos_head_stride + (size_t)i * p.r, *pk = p.pk + (size_t)c.h * p.pos_head_stride;
    auto logit = [&](int j, size_t key) {
        return add_products(add_products(0.f, p.q + query * p.d, p.inv_sqrt_d, p.k + key * p.d, p.d), pq, p.inv_sqrt_r, pk + (size_t)j * p.r, p.r);
    };
    float m = -INFINITY, l = 0.f, o[16];
    for (int key = 0; key < 64 * c.patches; ++key) {
        int j;
        size_t token;
        if (place(key >> 6, key & 63, j, token)) m = fmaxf(m, logit(j, token));
    }
#pragma unroll
    for (int e = 0; e < 16; ++e) o[e] = 0.f;
    for (int key = 0; key < 64 * c.patches && m > -INFINITY; ++key) {
        int j;
        size_t token;
        if (!place(key >> 6, key & 63, j, token)) continue;
        const float w = expf(logit(j, token) - m);
        l += w;
#pragma unroll
        for (int e = 0; e < 16; ++e)
            if (half * 16 + e < p.d) o[e] = fmaf(w, __bfloat162float(p.v[token * p.d + half * 16 + e]), o[e]);
    }
    const float inv = 1.f / l;
#pragma unroll
    for (int e = 0; e < 16; ++e)
        if (half * 16 + e < p.d) p.out[query * p.d + half * 16 + e] = __float2bfloat16_rn(o[e] * inv);
    if (p.lse && half == 0) p.lse[((size_t)c.b * p.heads + c.h) * p.H * p.W + (query / p.heads - (size_t)c.b * p.H * p.W)] = m + logf(l);
}

template <int R>
__global__ void __launch_bounds__(kThreads, 1)
rib_fwd_frame_sm100_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                           const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_pk, const __grid_constant__ FrameParams p)
{
    using L = Frame<R>;
    constexpr int kStages = L::kStages;
    constexpr uint32_t kPos = L::kPos;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    auto bar = [&](int i) { return base + L::kOffBar + 8u * i; };
    // of kSFull, kPReady, kPVDone: the barrier of a tile's block and the parity of its phase.  (Blocks -1 and -2 have the parity that a
    // barrier without a completed phase answers yes to.)
    auto on_block = [&](int which, int tile, uint32_t block) { return bar(which + 2 * tile + (block & 1)); };
    auto parity = [](uint32_t block) { return (block >> 1) & 1; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + L::kOffMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + L::kOffMisc + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int items = p.live.offset[9];

    if (threadIdx.x == 0) {
        abort_flag[0] = 0; abort_flag[1] = 0;   // [1] stays 0: used by the drain waits
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(L::kQFull + i), 1); mbar_init(bar(L::kQEmpty + i), 1); mbar_init(bar(L::kQPos + i), 1);
            for (int q4 = 0; q4 < 4; ++q4) mbar_init(bar(L::kMerge + 4 * i + q4), 2);
        }
        for (int i = 0; i < 4; ++i) { mbar_init(bar(L::kSFull + i), 1); mbar_init(bar(L::kPReady + i), 8); mbar_init(bar(L::kPVDone + i), 1); }
        for (int s = 0; s < kStages; ++s) { mbar_init(bar(L::kFull + s), 1); mbar_init(bar(L::kEmpty + s), 2); }     // empty: both tiles' PV
        for (int i = 0; i < 3; ++i) mbar_init(bar(L::kDrain + i), 1);
        fence_barrier_init();
        prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v); prefetch_tensormap(&tm_pk);
    }
    if (warp == 2) {
        tmem_alloc(base + L::kOffMisc, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    bool ok = true;
    if (warp == 0) {
        // ===================== TMA producer (lane 0) and the query RIB rows Pq * sqrt(d/r) of the same item, in terms (whole warp)
        uint32_t io = 0, blk = 0;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++io) {
            const LiveItem c = decode_live_item(p.live, item);
            const uint32_t buf = io & 1;
            if (io >= 2 && !mbar_wait_warp(bar(L::kQEmpty + buf), ((io >> 1) - 1) & 1, abort_flag, p.status)) { ok = false; break; }
            if (lane == 0) {
                mbar_arrive_expect_tx(bar(L::kQFull + buf), 2 * kContentBytes);
                for (int q4 = 0; q4 < 4; ++q4) {
                    int py, px, Y0, X0;
                    live_patch_origin(p.live, p.geom, c, min(4 * c.tp + q4, c.patches - 1), py, px, Y0, X0);
                    tma_load_5d(base + L::kOffQc + 2 * buf * kContentBytes + q4 * kPatchContent, &tm_q, bar(L::kQFull + buf), 0, c.h, X0, Y0, c.b);
                }
            }
            for (int k = 0; k < 8; ++k) {
                const int r256 = lane + 32 * k, qt = r256 >> 7, row = r256 & 127;
                int py, px, Y0, X0;
                live_patch_origin(p.live, p.geom, c, min(4 * c.tp + (r256 >> 6), c.patches - 1), py, px, Y0, X0);
                const int token = (py + ((row >> 3) & 7)) * p.geom.M + px + (row & 7);      // row of the table
                const uint4* src = reinterpret_cast<const uint4*>(p.pq + (size_t)c.h * p.pos_head_stride + (size_t)token * p.r);
                uint8_t* dst = base_ptr + L::kOffQp + (2 * buf + qt) * kTerms * kPos + row * (2 * R);
                const int sw = R == 16 ? (row >> 2) & 1 : (row >> 1) & 3;                   // SWIZZLE_32B / SWIZZLE_64B
#pragma unroll
                for (int ck = 0; ck < R / 8; ++ck) {                                        // 16-byte chunks of the row
                    const uint4 v = 8 * ck < p.r ? __ldg(src + ck) : make_uint4(0u, 0u, 0u, 0u);
                    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
                    uint32_t t[kTerms][4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float lo = __uint_as_float(w[e] << 16) * p.pos_scale, hi = __uint_as_float(w[e] & 0xffff0000u) * p.pos_scale;
#pragma unroll
                        for (int term = 0; term < kTerms; ++term) {
                            t[term][e] = pack_bf16x2(lo, hi);
                            lo -= __uint_as_float(t[term][e] << 16);
                            hi -= __uint_as_float(t[term][e] & 0xffff0000u);
                        }
                    }
#pragma unroll
                    for (int term = 0; term < kTerms; ++term)
                        if (term < p.terms) *reinterpret_cast<uint4*>(dst + term * kPos + ((ck ^ sw) << 4)) = make_uint4(t[term][0], t[term][1], t[term][2], t[term][3]);
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar(L::kQPos + buf));
                const int nblk = (c.patches + 1) >> 1;
                for (int j = 0; j < nblk; ++j, ++blk) {
                    const uint32_t st = blk % kStages, use = blk / kStages;
                    if (use > 0 && !mbar_wait(bar(L::kEmpty + st), (use - 1) & 1, abort_flag, p.status)) { ok = false; break; }
                    mbar_arrive_expect_tx(bar(L::kFull + st), 2 * kContentBytes + kPos);
                    for (int sub = 0; sub < 2; ++sub) {
                        int py, px, Y0, X0;
                        live_patch_origin(p.live, p.geom, c, min(2 * j + sub, c.patches - 1), py, px, Y0, X0);
                        if (2 * j + sub >= c.patches) X0 = p.geom.W;         // no such patch: beyond the map, zeros
                        tma_load_5d(base + L::kOffKc + st * kContentBytes + sub * kPatchContent, &tm_k, bar(L::kFull + st), 0, c.h, X0, Y0, c.b);
                        tma_load_4d(base + L::kOffKp + st * kPos + sub * L::kPatchP, &tm_pk, bar(L::kFull + st), 0, px, py, c.h * p.pos_per_head);
                        tma_load_5d(base + L::kOffV + st * kContentBytes + sub * kPatchContent, &tm_v, bar(L::kFull + st), 0, c.h, X0, Y0, c.b);
                    }
                }
            } else {
                blk += (uint32_t)((c.patches + 1) >> 1);
            }
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            // (giving up here: the loop counts this item, whose query tiles are armed)
        }
        if (!ok && lane == 0) {
            // Gave up: let the copies already in flight land before the CTA may exit.
            for (uint32_t b2 = io > 2u ? io - 2 : 0; b2 < io; ++b2)
                mbar_wait(bar(L::kQFull + (b2 & 1)), (b2 >> 1) & 1, abort_flag + 1, p.status);
            for (uint32_t b2 = blk > (uint32_t)kStages ? blk - kStages : 0; b2 < blk; ++b2)
                mbar_wait(bar(L::kFull + b2 % kStages), (b2 / kStages) & 1, abort_flag + 1, p.status);
        }
    } else if (warp < 4) {
        // ===================== issuers: warp 1 the scores of both query tiles, warps 2 and 3 PV of tile 0 and 1; the whole warp walks and waits
        constexpr uint64_t kDesc64 = smem_desc_const(16, 512, kSwizzle64B), kDesc32 = smem_desc_const(16, 256, kSwizzle32B);
        constexpr uint64_t kDescP = R == 16 ? kDesc32 : kDesc64;
        uint32_t io = 0, blk = 0, sb = warp == 3 ? 1 : 0;      // sb: unit mod kBuffers
        auto next_unit = [&](uint32_t by) { sb += by; if (sb >= kBuffers) sb -= kBuffers; };
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++io) {
            const int nblk = (decode_live_item(p.live, item).patches + 1) >> 1;
            const uint32_t buf = io & 1;
            if (warp == 1 && (!mbar_wait_warp(bar(L::kQFull + buf), (io >> 1) & 1, abort_flag, p.status) ||
                              !mbar_wait_warp(bar(L::kQPos + buf), (io >> 1) & 1, abort_flag, p.status))) { ok = false; break; }
            for (int j = 0; j < nblk && ok; ++j, ++blk) {
                const uint32_t st = blk % kStages;
                if (warp == 1) {
                    if (!mbar_wait_warp(bar(L::kFull + st), (blk / kStages) & 1, abort_flag, p.status)) { ok = false; break; }
                    const uint64_t kc = smem_desc_at(kDesc64, base + L::kOffKc + st * kContentBytes), kp = smem_desc_at(kDescP, base + L::kOffKp + st * kPos);
#pragma unroll
                    for (int qt = 0; qt < 2; ++qt) {
                        // The scores overwrite the columns that PV of three units before, one of the other tile, reads P from: it has completed.
                        const uint32_t before = blk - 2 + qt;
                        if (!mbar_wait_warp(on_block(L::kPVDone, qt ^ 1, before), parity(before), abort_flag, p.status)) { ok = false; break; }
                        tc_fence_after();
                        if (elect_one()) {
                            const uint64_t qc = smem_desc_at(kDesc64, base + L::kOffQc + (2 * buf + qt) * kContentBytes);
                            const uint64_t qp = smem_desc_at(kDescP, base + L::kOffQp + (2 * buf + qt) * kTerms * kPos);
                            const uint32_t d_s = tmem + sb * kTile;
                            // smallest terms first: a step drops what lies below the last place of the sum so far
                            for (int term = p.terms - 1; term >= 0; --term) {
                                mma_ss(d_s, qp + term * (kPos >> 4), kp, kIdescS, term == p.terms - 1 ? 0u : 1u);
                                if (R == 32) mma_ss(d_s, qp + term * (kPos >> 4) + 2, kp + 2, kIdescS, 1u);
                            }
                            mma_ss(d_s, qc, kc, kIdescS, 1u);
                            mma_ss(d_s, qc + 2, kc + 2, kIdescS, 1u);          // + 32 bytes: second K16 step of the content rows
                            mma_commit(on_block(L::kSFull, qt, blk));
                            if (qt == 1 && j == nblk - 1) mma_commit(bar(L::kQEmpty + buf));
                        }
                        __syncwarp();
                        next_unit(1);
                    }
                } else {
                    // P of the unit is there.  (The first block of an item overwrites O: the softmax warps have read it before they
                    // arrive here for that block.)
                    if (!mbar_wait_warp(bar(L::kFull + st), (blk / kStages) & 1, abort_flag, p.status) ||
                        !mbar_wait_warp(on_block(L::kPReady, warp - 2, blk), parity(blk), abort_flag, p.status)) { ok = false; break; }
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t vd = smem_desc_at(kDesc64, base + L::kOffV + st * kContentBytes);
                        const uint32_t a_p = tmem + sb * kTile, d_o = tmem + kColO + (warp - 2) * 2 * kD;
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) {                   // keys 16 kk ..: key half kk / 4 has its own accumulator
                            const uint32_t a = a_p + (kk >> 2) * 64 + 8 * (kk & 3), d = d_o + (kk >> 2) * kD;
                            mma_ts(d, a, vd + 64 * kk, kIdescPV, (j == 0 && (kk & 3) == 0) ? 0u : 1u);
                            mma_ts(d, a + 32, vd + 64 * kk, kIdescPV, 1u);
                        }
                        mma_commit(on_block(L::kPVDone, warp - 2, blk));
                        mma_commit(bar(L::kEmpty + st));
                    }
                    __syncwarp();
                    next_unit(2);
                }
            }
        }
        // everything issued by this warp's leader must have finished before TMEM is released
        if (elect_one()) mma_commit(bar(L::kDrain + warp - 1));
        __syncwarp();
        mbar_wait(bar(L::kDrain + warp - 1), 0, abort_flag + 1, p.status);
    } else {
        // ================ softmax + epilogue: two threads per query row, one per half of the keys
        const int qt = (warp - 4) >> 3;
        const int half = ((warp - 4) >> 2) & 1;
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;                 // row of the tile == TMEM lane
        const uint32_t t_half = tmem + ((uint32_t)(quarter * 32) << 16) + half * 64;                // + buffer: own scores, own P
        const uint32_t t_o = tmem + ((uint32_t)(quarter * 32) << 16) + kColO + qt * 2 * kD;         // both halves' accumulators
        // [half][row]; two sets, so that a warp that is an item ahead of its partner does not overwrite what that one still reads
        float2* const merge_sets = reinterpret_cast<float2*>(base_ptr + L::kOffMerge) + qt * 2 * kTile;
        const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
        uint32_t blk = 0, nmerge = 0;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++nmerge) {
            const LiveItem c = decode_live_item(p.live, item);
            const int nblk = (c.patches + 1) >> 1;
            // does the window reach beyond the frame?  (only then can a patch hold fewer than 64 tokens)
            const bool edge = c.wy * p.geom.M + p.geom.s + p.geom.M > p.H || c.wx * p.geom.M + p.geom.s + p.geom.M > p.W;
            float m_used = -INFINITY, l = 0.f;
            for (int j = 0; j < nblk; ++j, ++blk) {
                const uint32_t sb = (2 * blk + qt) % kBuffers;
                // warp-uniform outcome: the TMEM accesses below are warp-collective
                if (!mbar_wait_warp(on_block(L::kSFull, qt, blk), parity(blk), abort_flag, p.status)) { ok = false; break; }
                tc_fence_after();
                uint32_t s[2][32];
                tmem_ld32(t_half + sb * kTile, s[0]);
                tmem_ld32(t_half + sb * kTile + 32, s[1]);
                tmem_wait_ld();
                if (edge) {
                    // this thread's 64 keys are one 8x8 patch: tokens beyond the frame (or all of a missing last patch) get -inf
                    int py, px, Y0, X0, rows = 0, cols = 0;
                    if (2 * j + half < c.patches) {
                        live_patch_origin(p.live, p.geom, c, 2 * j + half, py, px, Y0, X0);
                        rows = p.H - Y0; cols = p.W - X0;
                    }
                    if (rows < 8 || cols < 8) {              // warp-uniform
#pragma unroll
                        for (int e = 0; e < 64; ++e)
                            if ((e >> 3) >= rows || (e & 7) >= cols) s[e >> 5][e & 31] = 0xff800000u;
                    }
                }
                float mxs[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int e = 0; e < 32; e += 4) {
                    mxs[0] = max3(mxs[0], __uint_as_float(s[0][e]), __uint_as_float(s[0][e + 1]));
                    mxs[1] = max3(mxs[1], __uint_as_float(s[1][e]), __uint_as_float(s[1][e + 1]));
                    mxs[2] = max3(mxs[2], __uint_as_float(s[0][e + 2]), __uint_as_float(s[0][e + 3]));
                    mxs[3] = max3(mxs[3], __uint_as_float(s[1][e + 2]), __uint_as_float(s[1][e + 3]));
                }
                const float mx = fmaxf(fmaxf(mxs[0], mxs[1]), fmaxf(mxs[2], mxs[3]));
                if (j == 0) {
                    m_used = mx;
                } else {
                    // Move the reference (and rescale O, l) only when the maximum grew by more than the threshold; the result
                    // is exact after the final normalisation because l carries the same reference.
                    const bool need = mx > m_used + p.rescale_threshold;
                    if (__any_sync(0xffffffffu, need)) {
                        if (!mbar_wait_warp(on_block(L::kPVDone, qt, blk - 1), parity(blk - 1), abort_flag, p.status)) { ok = false; break; }
                        tc_fence_after();
                        const float factor = need ? ex2_approx(__fmul_rn(m_used, p.scale_log2) - __fmul_rn(mx, p.scale_log2)) : 1.f;
                        if (need) { l *= factor; m_used = mx; }
                        for (int g = 0; g < 4; ++g) {
                            uint32_t o[8];
                            tmem_ld8(t_o + half * kD + 8 * g, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 8; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * factor);
                            tmem_st8(t_o + half * kD + 8 * g, o);
                        }
                    }
                }
                // a half that has seen no token yet has no reference: its scores are all -inf, its probabilities 0
                const float neg = m_used == -INFINITY ? 0.f : __fmul_rn(-m_used, p.scale_log2);
                const float2 neg2 = make_float2(neg, neg);
                float2 sum_a = make_float2(0.f, 0.f), sum_b = make_float2(0.f, 0.f);
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) {                  // 16 keys at a time: next to 64 scores, no more results fit the registers
                    uint32_t hi[8], lo[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int k = 16 * (ch & 1) + 2 * i;
                        const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[ch >> 1][k]), __uint_as_float(s[ch >> 1][k + 1])), scale2, neg2);
                        const float2 e = make_float2(ex2_approx(x.x), ex2_approx(x.y));
                        if (i & 1) sum_b = __fadd2_rn(sum_b, e); else sum_a = __fadd2_rn(sum_a, e);
                        hi[i] = pack_bf16x2(e.x, e.y);
                        const float2 rest = __fadd2_rn(e, make_float2(-__uint_as_float(hi[i] << 16), -__uint_as_float(hi[i] & 0xffff0000u)));
                        lo[i] = pack_bf16x2(rest.x, rest.y);
                    }
                    tmem_st8(t_half + sb * kTile + 8 * ch, hi);
                    tmem_st8(t_half + sb * kTile + 32 + 8 * ch, lo);
                }
                l += (sum_a.x + sum_a.y) + (sum_b.x + sum_b.y);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(on_block(L::kPReady, qt, blk));
            }
            if (!ok) break;
            // ---- merge the two key halves and write this thread's 16 output columns
            float2* const merge = merge_sets + (nmerge & 1) * 4 * kTile;
            merge[half * kTile + row] = make_float2(m_used, l);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(L::kMerge + 4 * qt + quarter));
            // The partner's (m, l) must be there and the item's last PV must have completed.
            if (!mbar_wait_warp(bar(L::kMerge + 4 * qt + quarter), nmerge & 1, abort_flag, p.status) ||
                !mbar_wait_warp(on_block(L::kPVDone, qt, blk - 1), parity(blk - 1), abort_flag, p.status)) { ok = false; break; }
            tc_fence_after();
            uint32_t oa[16], ob[16];
            tmem_ld16(t_o + half * 16, oa);
            tmem_ld16(t_o + kD + half * 16, ob);
            tmem_wait_ld();
            tc_fence_before();
            const float2 other = merge[(half ^ 1) * kTile + row];
            const float m_a = half ? other.x : m_used, l_a = half ? other.y : l;
            const float m_b = half ? m_used : other.x, l_b = half ? l : other.y;
            // the offsets as the exponentials took them, so that their rounding cancels
            const float n_a = __fmul_rn(-m_a, p.scale_log2), n_b = __fmul_rn(-m_b, p.scale_log2), n = fminf(n_a, n_b);
            // (a half without a finite logit, offset inf, adds nothing)
            const float f_a = n_a == INFINITY ? 0.f : ex2_approx(n - n_a), f_b = n_b == INFINITY ? 0.f : ex2_approx(n - n_b);
            const float l_all = l_a * f_a + l_b * f_b;
            const float w_a = f_a / l_all, w_b = f_b / l_all;
            const int k = 4 * c.tp + 2 * qt + (row >> 6);
            int py, px, Y0, X0;
            live_patch_origin(p.live, p.geom, c, min(k, c.patches - 1), py, px, Y0, X0);
            const int Y = Y0 + ((row >> 3) & 7), X = X0 + (row & 7);
            if (k < c.patches && Y < p.H && X < p.W) {       // (else: no token, nothing to store)
                const size_t tok = (((size_t)c.b * p.H + Y) * p.W + X) * p.heads + c.h;
                uint4* dst = reinterpret_cast<uint4*>(p.out + tok * p.d + half * 16);
                float sum = 0.f;                             // NaN if a value is NaN
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    if (half * 16 + 8 * g >= p.d) break;     // a head narrower than 32 channels: the rest of the row is padding
                    uint32_t w[4];
#pragma unroll
                    for (int k2 = 0; k2 < 4; ++k2) {
                        const int e = 8 * g + 2 * k2;
                        const float x = __uint_as_float(oa[e]) * w_a + __uint_as_float(ob[e]) * w_b, y = __uint_as_float(oa[e + 1]) * w_a + __uint_as_float(ob[e + 1]) * w_b;
                        sum += x + y;
                        w[k2] = pack_bf16x2(x, y);
                    }
                    dst[g] = make_uint4(w[0], w[1], w[2], w[3]);
                }
                if (p.lse && half == 0) p.lse[(((size_t)c.b * p.heads + c.h) * p.H + Y) * p.W + X] = log_sum(n, l_all);
                if (isnan(sum)) plain_row(&p, item, 128 * qt + row, half);
            }
            __syncwarp();
        }
    }
    // ================================================================================ common tail
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

}  // namespace

template <int R>
cudaError_t launch_fwd_frame(const Problem& p, cudaStream_t stream)
{
    if (!encode_fn()) return cudaErrorNotSupported;
    FrameParams fp{};
    if (!make_live_windows(p, &fp.live)) return cudaErrorInvalidValue;
    CUtensorMap tm_q, tm_k, tm_v, tm_pk;
    if (!encode_image_map(&tm_q, p.q, p) || !encode_image_map(&tm_k, p.k, p) || !encode_image_map(&tm_v, p.v, p) ||
        !encode_pos_map(&tm_pk, p.pk, p, pos_tables(p), p.pos_head_stride))
        return cudaErrorInvalidValue;
    static KernelSetup setup;       // one per instantiation of this launcher, i.e. per kernel
    int sm_count = 0;
    if (cudaError_t e = setup.prepare(rib_fwd_frame_sm100_kernel<R>, Frame<R>::kSmemBytes, &sm_count)) return e;
    const float d = scale_width_d(p), r = scale_width_r(p);
    fp.q = p.q; fp.k = p.k; fp.v = p.v; fp.pk = p.pk;
    fp.inv_sqrt_d = 1.f / sqrtf(d); fp.inv_sqrt_r = 1.f / sqrtf(r);
    fp.pq = p.pq; fp.out = p.out_w; fp.lse = p.lse_w; fp.status = p.status;
    fp.H = p.H; fp.W = p.W; fp.heads = p.heads; fp.d = p.d; fp.r = p.r;
    fp.geom = WindowGeom{p.Hp, p.Wp, p.M, p.s};
    fp.scale_log2 = (float)(1.4426950408889634 / sqrt((double)d));
    fp.rescale_threshold = 8.0f / fp.scale_log2;
    fp.pos_scale = sqrtf(d / r);
    fp.terms = d == r || d == 4.f * r || 4.f * d == r ? 1 : kTerms;      // sqrt(d / r) a power of two: the product is a bf16 number
    fp.pos_head_stride = p.pos_head_stride;
    fp.pos_per_head = p.pos_head_stride ? 1 : 0;
    const int items = fp.live.offset[9], grid = items < sm_count ? items : sm_count;
    { ProfileScope scope(RIB_KERNEL_FWD_FRAME, stream); rib_fwd_frame_sm100_kernel<R><<<grid, kThreads, Frame<R>::kSmemBytes, stream>>>(tm_q, tm_k, tm_v, tm_pk, fp); }
    return cudaGetLastError();
}

bool sm100_frame_supported(const Problem& p)
{
    return p.d % 8 == 0 && p.d >= 8 && p.d <= kD && p.r % 8 == 0 && p.r >= 8 && p.r <= 32 && p.M % 16 == 0 && p.M <= 256 && p.s % 8 == 0 &&
           (p.H % 8 || p.W % 8) && !p.masked && !p.gate;
}

cudaError_t sm100_fwd_frame(const Problem& p, cudaStream_t stream)
{
    return padded_rank(p.r) == 32 ? launch_fwd_frame<32>(p, stream) : launch_fwd_frame<16>(p, stream);
}

}  // namespace rib
