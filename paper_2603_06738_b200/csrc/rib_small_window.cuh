// Shared between the kernels for windows of 8 x 8 and of 16 x 16 tokens: a CTA keeps to one head, whose RIB rows it stages once,
// and works whole windows, so that every gradient but those of the tables is final when it leaves the chip.
#pragma once
#include "rib_sm100_common.cuh"

namespace rib {
namespace sm100 {

struct SmallWindowParams {
    const __nv_bfloat16* pq;
    const __nv_bfloat16* pk;
    const __nv_bfloat16* out;  // backward at 16 x 16
    const float* lse_in;       // backward
    float* lse;                // forward, may be null
    float* dpq;
    float* dpk;
    int* status;
    int H, W, heads, d, r;
    int Hp, Wp, s;             // 16 x 16: sides of the map the windows are laid over, shift
    int masked;                // 16 x 16: the wrapped parts of a border window do not attend to each other
    int tiles, groups;         // tiles (8 x 8: pairs of windows, 16 x 16: windows) of one head; CTAs of one head
    FastDiv by_heads, by_nx, by_ny;      // heads; tiles per row and column of a map
    float scale_log2;          // log2(e) / sqrt(d)
    float inv_sqrt_d, inv_sqrt_r;
    float pos_scale;           // sqrt(d / r)
    long long pos_head_stride;
};

// One CTA per SM, a whole number per head; with more heads than SMs a CTA per head.
inline int fill_small_window(const Problem& p, int sm_count, int tiles_y, int tiles_x, SmallWindowParams* w)
{
    w->pq = p.pq; w->pk = p.pk; w->status = p.status;
    w->H = p.H; w->W = p.W; w->heads = p.heads; w->d = p.d; w->r = p.r;
    w->Hp = p.Hp; w->Wp = p.Wp; w->s = p.s; w->masked = p.masked ? 1 : 0;
    w->tiles = p.B * tiles_y * tiles_x;
    w->groups = sm_count / p.heads > 1 ? sm_count / p.heads : 1;
    if (w->groups > w->tiles) w->groups = w->tiles;
    w->by_heads = make_fast_div(p.heads); w->by_nx = make_fast_div(tiles_x); w->by_ny = make_fast_div(tiles_y);
    const float d = scale_width_d(p), r = scale_width_r(p);
    w->scale_log2 = 1.4426950408889634f / sqrtf(d);
    w->inv_sqrt_d = 1.f / sqrtf(d);
    w->inv_sqrt_r = 1.f / sqrtf(r);
    w->pos_scale = sqrtf(d / r);
    w->pos_head_stride = p.pos_head_stride;
    return w->groups * p.heads;                    // CTAs
}

// One RIB row of a head as a 64-byte row (32 elements, zeros from column r on; SWIZZLE_64B like a content tile): row `table_row`
// of the tables to row `row` of the two tiles.  Query rows are scaled by sqrt(d / r) and rounded to bf16.
__device__ __forceinline__ void stage_rib_row(const SmallWindowParams& p, int head, int table_row, uint8_t* q_tile, uint8_t* k_tile, int row)
{
    const size_t at = (size_t)head * p.pos_head_stride + (size_t)table_row * p.r;
    const uint4 *q = reinterpret_cast<const uint4*>(p.pq + at), *k = reinterpret_cast<const uint4*>(p.pk + at);
    const int sw = (row >> 1) & 3;
#pragma unroll
    for (int ck = 0; ck < 4; ++ck) {
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u), a = 8 * ck < p.r ? __ldg(q + ck) : zero, b = 8 * ck < p.r ? __ldg(k + ck) : zero;
        uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            w[e] = pack_bf16x2(__uint_as_float(w[e] << 16) * p.pos_scale, __uint_as_float(w[e] & 0xffff0000u) * p.pos_scale);
        *reinterpret_cast<uint4*>(q_tile + row * 64 + ((ck ^ sw) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(k_tile + row * 64 + ((ck ^ sw) << 4)) = b;
    }
}

// 32 fp32 columns of a row (times f) as a bf16 row of a 64-byte-row tile
__device__ __forceinline__ void write_row(uint8_t* tile, int row, const uint32_t (&a)[32], float f)
{
    const int sw = (row >> 1) & 3;
#pragma unroll
    for (int ck = 0; ck < 4; ++ck)
        *reinterpret_cast<uint4*>(tile + row * 64 + ((ck ^ sw) << 4)) =
            make_uint4(pack_bf16x2(__uint_as_float(a[8 * ck]) * f, __uint_as_float(a[8 * ck + 1]) * f),
                       pack_bf16x2(__uint_as_float(a[8 * ck + 2]) * f, __uint_as_float(a[8 * ck + 3]) * f),
                       pack_bf16x2(__uint_as_float(a[8 * ck + 4]) * f, __uint_as_float(a[8 * ck + 5]) * f),
                       pack_bf16x2(__uint_as_float(a[8 * ck + 6]) * f, __uint_as_float(a[8 * ck + 7]) * f));
}


// Adds four columns of table gradients
__device__ __forceinline__ void add_columns(float* dst, const uint32_t* a, float f)
{
    atomicAdd(reinterpret_cast<float4*>(dst), make_float4(__uint_as_float(a[0]) * f, __uint_as_float(a[1]) * f, __uint_as_float(a[2]) * f, __uint_as_float(a[3]) * f));
}

}  // namespace sm100
}  // namespace rib
