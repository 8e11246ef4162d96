// Head widths and ranks whose rows TMA cannot address (a row must be a multiple of 16 bytes: d = 30 gives 60-byte rows,
// r = 18 gives 36-byte rows -- the SST rows of the paper's network table).  For even d, r <= 32 the tensors are copied
// into scratch with every row filled up with zeros to the next multiple of 8 elements, the tcgen05 kernels run on the
// copies (zero channels change no dot product; the scales of Eq. 6 keep the true d and r), and the results are copied
// back, all copies of a pass in one launch.  The scratch comes from a stream-ordered memory pool of the library's own, one per device, that keeps what is
// freed (cudaMallocFromPoolAsync / cudaFreeAsync on the caller's stream): after the first call of a shape nothing here
// talks to the driver's allocator and nothing synchronises.  The attention passes are bound by arithmetic, so the copies (a few hundred bytes per
// token-head) cost little next to them; the any-shape kernels these shapes would otherwise take are about a hundred
// times slower.
#include "rib_common.cuh"

#include <mutex>

namespace rib {
namespace {

// One pool per device, created on first use with that device current; freed blocks stay in the pool (release threshold
// at its maximum), so the steady state of a training loop reuses the same memory.
constexpr int kMaxPoolDevices = 64;
std::mutex g_pool_mutex;
cudaMemPool_t g_pool[kMaxPoolDevices] = {};

cudaError_t scratch_pool(cudaMemPool_t* pool)
{
    int dev = -1;
    if (cudaError_t e = cudaGetDevice(&dev)) return e;
    if (dev < 0 || dev >= kMaxPoolDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    if (!g_pool[dev]) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t created = nullptr;
        if (cudaError_t e = cudaMemPoolCreate(&created, &props)) return e;
        unsigned long long keep = ~0ull;
        if (cudaError_t e = cudaMemPoolSetAttribute(created, cudaMemPoolAttrReleaseThreshold, &keep)) { cudaMemPoolDestroy(created); return e; }
        g_pool[dev] = created;
    }
    *pool = g_pool[dev];
    return cudaSuccess;
}

cudaError_t scratch_alloc(uint8_t** ptr, size_t bytes, cudaStream_t stream)
{
    cudaMemPool_t pool = nullptr;
    if (cudaError_t e = scratch_pool(&pool)) return e;
    return cudaMallocFromPoolAsync(reinterpret_cast<void**>(ptr), bytes, pool, stream);
}

// dst[row][c] = src[row][c] for c < min(ws, wd), 0 for the other columns of dst; T is a pair of elements
template <typename T>
__global__ void __launch_bounds__(256) rib_copy_columns_kernel(const T* __restrict__ src, int ws, T* __restrict__ dst, int wd, size_t rows)
{
    // (32-bit index arithmetic: the launcher splits tensors of 2^32 pairs and more)
    const unsigned total = (unsigned)rows * (unsigned)wd;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const unsigned row = e / (unsigned)wd, c = e - row * (unsigned)wd;
        T v{};
        if (c < (unsigned)ws) v = src[(size_t)row * ws + c];
        dst[e] = v;
    }
}

// Ranks above 32 (d = 30 with r = 34): the kernels hold 32 RIB columns, and the zero channels of the padded head have
// room for the rest.  Column 32 + j of the tables goes into channel d + j of the q and k copies -- for q times sqrt(d / r),
// so that the content scale 1 / sqrt(d) leaves 1 / sqrt(r) on the product, exactly as for the staged RIB rows -- indexed by
// the token's place in its window; the logits are unchanged.  Geometry of the token -> window position map:
struct PlaceGeom { int H, W, Hp, Wp, heads, M, s, d, dp, r, extra; long long table_stride; float scale; };

__device__ __forceinline__ int window_place(const PlaceGeom& g, int Y, int X)
{
    int yr = Y - g.s, xr = X - g.s;                 // the rolled frame the windows are cut from
    if (yr < 0) yr += g.Hp;
    if (xr < 0) xr += g.Wp;
    return (yr % g.M) * g.M + xr % g.M;
}

// dst[row][c]: c < d from src, d <= c < d + extra from table[place][32 + c - d] * scale, zero beyond; pairs of elements
__global__ void __launch_bounds__(256) rib_pack_with_rank_tail_kernel(const uint32_t* __restrict__ src, uint32_t* __restrict__ dst,
                                                                     const __nv_bfloat16* __restrict__ table, PlaceGeom g, unsigned rows)
{
    const unsigned wd = g.dp / 2, ws = g.d / 2, total = rows * wd;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const unsigned row = e / wd, c = e - row * wd;
        uint32_t v = 0u;
        if (c < ws) {
            v = src[(size_t)row * ws + c];
        } else if (2 * (int)(c - ws) < g.extra) {
            const unsigned h = row % (unsigned)g.heads, pixel = row / (unsigned)g.heads;
            const int X = (int)(pixel % (unsigned)g.W), Y = (int)((pixel / (unsigned)g.W) % (unsigned)g.H);
            const __nv_bfloat16* t = table + (size_t)h * g.table_stride + (size_t)window_place(g, Y, X) * g.r + 32 + 2 * (c - ws);
            const __nv_bfloat162 two = __floats2bfloat162_rn(__bfloat162float(t[0]) * g.scale, __bfloat162float(t[1]) * g.scale);
            v = *reinterpret_cast<const uint32_t*>(&two);
        }
        dst[e] = v;
    }
}

// the gradient of those table columns: channel d + j of dq and dk of every token, summed over the tokens of a place
__global__ void __launch_bounds__(256) rib_rank_tail_grads_kernel(const __nv_bfloat16* __restrict__ dq, const __nv_bfloat16* __restrict__ dk,
                                                                 float* __restrict__ dpq, float* __restrict__ dpk, PlaceGeom g, unsigned rows)
{
    const unsigned total = rows * (unsigned)g.extra;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const unsigned row = e / (unsigned)g.extra, j = e - row * (unsigned)g.extra;
        const unsigned h = row % (unsigned)g.heads, pixel = row / (unsigned)g.heads;
        const int X = (int)(pixel % (unsigned)g.W), Y = (int)((pixel / (unsigned)g.W) % (unsigned)g.H);
        const size_t at = (size_t)h * g.table_stride + (size_t)window_place(g, Y, X) * g.r + 32 + j;
        atomicAdd(dpq + at, __bfloat162float(dq[(size_t)row * g.dp + g.d + j]) * g.scale);
        atomicAdd(dpk + at, __bfloat162float(dk[(size_t)row * g.dp + g.d + j]));
    }
}

// All copies of a pass in one launch.  A copy: rows of 4-byte words, one side `wide` words a row (a multiple of 4, 16-byte aligned),
// the other `narrow`; widen: narrow to wide with zeros behind, else wide to narrow.  A thread moves 16-byte pieces of the wide side,
// which is one vector access there and up to four word accesses on the narrow side; a block as many whole rows as make up 1024 of them
// (the widest rows are 24 pieces), all loads of a thread before its stores.
struct RowCopy { const uint32_t* src; uint32_t* dst; size_t rows; unsigned first_block, rows_per_block; int narrow, wide, widen; };
constexpr int kMostCopies = 8, kCopyPieces = 4;
template <int kMost>
struct RowCopyList {
    RowCopy copy[kMost];
    int count;
    unsigned blocks;
    // src rows of ws words -> dst rows of wd words
    void add(const void* src, int ws, void* dst, int wd, size_t rows)
    {
        RowCopy& c = copy[count++];
        c.src = static_cast<const uint32_t*>(src); c.dst = static_cast<uint32_t*>(dst); c.rows = rows;
        c.widen = wd >= ws; c.wide = c.widen ? wd : ws; c.narrow = c.widen ? ws : wd;
        c.first_block = blocks;
        c.rows_per_block = 256u * kCopyPieces / (unsigned)(c.wide / 4);
        blocks += (unsigned)((rows + c.rows_per_block - 1) / c.rows_per_block);
    }
};
using RowCopies = RowCopyList<kMostCopies>;

// A copy on its own has an instantiation of its own, and a block begins with a row: with the parameters of eight copies, a search among
// them and a 64-bit division for the first row the gate's backward with 96 channels on 2 x 64 x 64 pixels took 69.1 us, so 67.0 (three
// such copies among its 14 launches; one copy kernel per tensor with scalar parameters 67.3).
template <int kMost>
__global__ void __launch_bounds__(256) rib_copy_rows_kernel(const __grid_constant__ RowCopyList<kMost> all)
{
    int which = 0;
    if (kMost > 1)
        while (which + 1 < all.count && blockIdx.x >= all.copy[which + 1].first_block) ++which;
    const RowCopy& c = all.copy[which];
    const unsigned per_row = (unsigned)c.wide / 4u;
    const size_t row0 = (size_t)(blockIdx.x - c.first_block) * c.rows_per_block;
    uint4 v[kCopyPieces];
    auto place = [&](int k, size_t& row, int& w0) {
        const unsigned at = threadIdx.x + 256u * k, r = at / per_row;
        row = row0 + r;
        w0 = 4 * (int)(at - r * per_row);
        return r < c.rows_per_block && row < c.rows;
    };
#pragma unroll
    for (int k = 0; k < kCopyPieces; ++k) {
        size_t row;
        int w0;
        v[k] = make_uint4(0u, 0u, 0u, 0u);
        if (!place(k, row, w0)) continue;
        if (!c.widen) { v[k] = *reinterpret_cast<const uint4*>(c.src + row * c.wide + w0); continue; }
        const uint32_t* in = c.src + row * c.narrow + w0;
        if (w0 < c.narrow) v[k].x = in[0];
        if (w0 + 1 < c.narrow) v[k].y = in[1];
        if (w0 + 2 < c.narrow) v[k].z = in[2];
        if (w0 + 3 < c.narrow) v[k].w = in[3];
    }
#pragma unroll
    for (int k = 0; k < kCopyPieces; ++k) {
        size_t row;
        int w0;
        if (!place(k, row, w0)) continue;
        if (c.widen) { *reinterpret_cast<uint4*>(c.dst + row * c.wide + w0) = v[k]; continue; }
        uint32_t* out = c.dst + row * c.narrow + w0;
        if (w0 < c.narrow) out[0] = v[k].x;
        if (w0 + 1 < c.narrow) out[1] = v[k].y;
        if (w0 + 2 < c.narrow) out[2] = v[k].z;
        if (w0 + 3 < c.narrow) out[3] = v[k].w;
    }
}

template <int kMost>
cudaError_t run_copies(const RowCopyList<kMost>& all, cudaStream_t stream, int* launches)
{
    if (!all.blocks) return cudaSuccess;
    if (kMost > 1 && all.count == 1) return run_copies(RowCopyList<1>{{all.copy[0]}, 1, all.blocks}, stream, launches);
    rib_copy_rows_kernel<kMost><<<all.blocks, 256, 0, stream>>>(all);
    ++*launches;
    return cudaGetLastError();
}

// bf16 image rows of `ws` elements -> rows of `wd` elements (one of the two a multiple of 8, the other smaller or equal)
cudaError_t resize_rows(const void* src, int ws, void* dst, int wd, size_t rows, cudaStream_t stream, int* launches)
{
    RowCopyList<1> one{};
    one.add(src, ws / 2, dst, wd / 2, rows);
    return run_copies(one, stream, launches);
}

template <typename T>
cudaError_t copy_columns(const void* src, int ws_elems, void* dst, int wd_elems, size_t rows, cudaStream_t stream, int* launches)
{
    const int ws = ws_elems / 2, wd = wd_elems / 2;
    const size_t chunk = (size_t)0x7fffffff / (size_t)wd;          // rows per launch: their pairs fit 31 bits
    for (size_t r0 = 0; r0 < rows; r0 += chunk) {
        const size_t nrows = rows - r0 < chunk ? rows - r0 : chunk, total = nrows * (size_t)wd;
        const unsigned blocks = (unsigned)((total + 255) / 256 < 148 * 16 ? (total + 255) / 256 : 148 * 16);
        rib_copy_columns_kernel<T><<<blocks, 256, 0, stream>>>(static_cast<const T*>(src) + r0 * ws, ws, static_cast<T*>(dst) + r0 * wd, wd, nrows);
        ++*launches;
        if (cudaError_t e = cudaGetLastError()) return e;
    }
    return cudaSuccess;
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// a table per head `stride` elements apart (or one table): rows of ws elements -> packed tables of rows of wd elements
template <typename T, typename Elem>
cudaError_t copy_tables(const Elem* src, long long src_stride, int ws, Elem* dst, long long dst_stride, int wd, int tables, int n,
                        cudaStream_t stream, int* launches)
{
    for (int t = 0; t < tables; ++t)
        if (cudaError_t e = copy_columns<T>(src + (size_t)t * src_stride, ws, dst + (size_t)t * dst_stride, wd, (size_t)n, stream, launches)) return e;
    return cudaSuccess;
}

// columns of the tables that travel in the zero channels of the padded head (ranks above 32)
int rank_tail(const Problem& p) { return p.r > 32 ? p.r - 32 : 0; }

PlaceGeom place_geom(const Problem& p)
{
    PlaceGeom g{};
    g.H = p.H; g.W = p.W; g.Hp = p.Hp; g.Wp = p.Wp; g.heads = p.heads; g.M = p.M; g.s = p.s;
    g.d = p.d; g.dp = repacked_width(p.d); g.r = p.r; g.extra = rank_tail(p);
    g.table_stride = p.pos_head_stride;
    g.scale = sqrtf((float)p.d / (float)p.r);
    return g;
}

Problem padded_shape(const Problem& p)
{
    Problem pp = p;
    pp.d = repacked_width(p.d);
    pp.r = p.r > 32 ? 32 : repacked_width(p.r);
    pp.d_true = p.d;
    pp.r_true = p.r;
    if (p.pos_head_stride) pp.pos_head_stride = (long long)p.n * pp.r;
    return pp;
}

// the tables lie behind one another, their rows no wider than the copies': they are one copy
bool tables_in_a_row(const Problem& p) { return !rank_tail(p) && (!p.pos_head_stride || p.pos_head_stride == (long long)p.n * p.r); }

// q, k and the tables into their padded copies: what is a plain copy is added to `copies`; with a rank above 32 the tail of the tables
// rides in the spare channels
cudaError_t pack(const Problem& p, __nv_bfloat16* q2, __nv_bfloat16* k2, __nv_bfloat16* pq2, __nv_bfloat16* pk2, int rp, size_t rows, RowCopies* copies,
                 cudaStream_t stream, int* launches)
{
    const int dp = repacked_width(p.d), tables = pos_tables(p);
    if (tables_in_a_row(p)) {
        copies->add(p.pq, p.r / 2, pq2, rp / 2, (size_t)tables * p.n);
        copies->add(p.pk, p.r / 2, pk2, rp / 2, (size_t)tables * p.n);
    } else {
        const long long stride = (long long)p.n * rp;
        if (cudaError_t e = copy_tables<uint32_t>(p.pq, p.pos_head_stride, p.r, pq2, stride, rp, tables, p.n, stream, launches)) return e;
        if (cudaError_t e = copy_tables<uint32_t>(p.pk, p.pos_head_stride, p.r, pk2, stride, rp, tables, p.n, stream, launches)) return e;
    }
    if (!rank_tail(p)) {
        copies->add(p.q, p.d / 2, q2, dp / 2, rows);
        copies->add(p.k, p.d / 2, k2, dp / 2, rows);
        return cudaSuccess;
    }
    PlaceGeom g = place_geom(p);
    const size_t total = rows * (size_t)(dp / 2);
    const unsigned blocks = (unsigned)((total + 255) / 256 < 148 * 16 ? (total + 255) / 256 : 148 * 16);
    rib_pack_with_rank_tail_kernel<<<blocks, 256, 0, stream>>>(reinterpret_cast<const uint32_t*>(p.q), reinterpret_cast<uint32_t*>(q2), p.pq, g, (unsigned)rows);
    g.scale = 1.f;
    rib_pack_with_rank_tail_kernel<<<blocks, 256, 0, stream>>>(reinterpret_cast<const uint32_t*>(p.k), reinterpret_cast<uint32_t*>(k2), p.pk, g, (unsigned)rows);
    *launches += 2;
    return cudaGetLastError();
}

}  // namespace

int repacked_width(int w) { return (w + 7) & ~7; }

static bool repack_supported(const Problem& p)
{
    if (p.d < 2 || p.d > 32 || p.r < 2 || (p.d & 1) || (p.r & 1) || p.d_true || p.r_true) return false;
    if (p.r > 32 && p.r - 32 > repacked_width(p.d) - p.d) return false;      // no room for the columns above 32
    if (p.d % 8 == 0 && p.r % 8 == 0) return false;          // these run on the kernels as they are
    if ((long long)p.B * p.H * p.W * p.heads * 16 > 0x7fffffffLL && p.r > 32) return false;   // 32-bit indices of the tail kernels
    return true;
}

bool sm100_repack_bwd_supported(const Problem& p) { return repack_supported(p) && sm100_bwd_supported(padded_shape(p)); }

bool sm100_repack_fwd_supported(const Problem& p)
{
    if (!repack_supported(p)) return false;
    const Problem pp = padded_shape(p);
    // (frames keep the precision of the any-shape kernel, which the rank tail in bf16 channels would not)
    return sm100_fwd_supported(pp) || (sm100_frame_supported(pp) && !rank_tail(p));
}

cudaError_t sm100_fwd_repacked(const Problem& p, cudaStream_t stream, int* launches)
{
    *launches = 0;
    Problem pp = padded_shape(p);
    const int tables = pos_tables(p);
    const size_t rows = (size_t)p.B * p.H * p.W * p.heads;
    const size_t img = up256(rows * pp.d * sizeof(__nv_bfloat16)), tab = up256((size_t)tables * p.n * pp.r * sizeof(__nv_bfloat16));
    uint8_t* buf = nullptr;
    if (cudaError_t e = scratch_alloc(&buf, 5 * img + 2 * tab, stream)) return e;
    __nv_bfloat16* q2 = reinterpret_cast<__nv_bfloat16*>(buf);
    __nv_bfloat16* k2 = reinterpret_cast<__nv_bfloat16*>(buf + img);
    __nv_bfloat16* v2 = reinterpret_cast<__nv_bfloat16*>(buf + 2 * img);
    __nv_bfloat16* o2 = reinterpret_cast<__nv_bfloat16*>(buf + 3 * img);
    __nv_bfloat16* g2 = reinterpret_cast<__nv_bfloat16*>(buf + 4 * img);          // the CLA gate, if any (layout of out)
    __nv_bfloat16* pq2 = reinterpret_cast<__nv_bfloat16*>(buf + 5 * img);
    __nv_bfloat16* pk2 = reinterpret_cast<__nv_bfloat16*>(buf + 5 * img + tab);
    RowCopies in{};
    cudaError_t e = pack(p, q2, k2, pq2, pk2, pp.r, rows, &in, stream, launches);
    in.add(p.v, p.d / 2, v2, pp.d / 2, rows);
    if (p.gate) { in.add(p.gate, p.d / 2, g2, pp.d / 2, rows); pp.gate = g2; }
    if (!e) e = run_copies(in, stream, launches);
    if (!e) {
        pp.q = q2; pp.k = k2; pp.v = v2; pp.pq = pq2; pp.pk = pk2; pp.out_w = o2;
        e = sm100_frame_supported(pp) ? sm100_fwd_frame(pp, stream) : sm100_fwd(pp, stream);
        ++*launches;
    }
    if (!e) e = resize_rows(o2, pp.d, p.out_w, p.d, rows, stream, launches);
    const cudaError_t f = cudaFreeAsync(buf, stream);
    return e ? e : f;
}

cudaError_t sm100_bwd_repacked(const Problem& p, cudaStream_t stream, int* launches)
{
    *launches = 0;
    Problem pp = padded_shape(p);
    const int tables = pos_tables(p);
    const size_t rows = (size_t)p.B * p.H * p.W * p.heads;
    const size_t img = up256(rows * pp.d * sizeof(__nv_bfloat16));
    const size_t tab = up256((size_t)tables * p.n * pp.r * sizeof(__nv_bfloat16)), gtab = up256((size_t)tables * p.n * pp.r * sizeof(float));
    uint8_t* buf = nullptr;
    if (cudaError_t e = scratch_alloc(&buf, 8 * img + 2 * tab + 2 * gtab, stream)) return e;
    auto image = [&](int i) { return reinterpret_cast<__nv_bfloat16*>(buf + (size_t)i * img); };
    __nv_bfloat16* pq2 = reinterpret_cast<__nv_bfloat16*>(buf + 8 * img);
    __nv_bfloat16* pk2 = reinterpret_cast<__nv_bfloat16*>(buf + 8 * img + tab);
    float* dpq2 = reinterpret_cast<float*>(buf + 8 * img + 2 * tab);
    float* dpk2 = reinterpret_cast<float*>(buf + 8 * img + 2 * tab + gtab);
    const long long tstride = (long long)p.n * pp.r;
    // The preparation kernel reads out, and the finishing kernel writes dq, in rows of the caller's width (those of the general kernel,
    // where no columns of the tables travel in the spare channels): two copies less.  (8 x 96 x 96 tokens, 30 channels, rank 18, windows
    // of 32: all copies of both passes 160 -> 80 us with one launch per pass, the two kernels 87 -> 105 us, both passes 721 -> 660 us; the two
    // kernels take 74 us now.  dk and dv leave the main kernel by TMA, which has no rows of 60 bytes: its strides are multiples of 16 bytes.)
    const bool direct = sm100_bwd_takes_narrow(pp) && !rank_tail(p);
    pp.narrow = direct && p.d % 8 ? p.d : 0;
    RowCopies in{};
    cudaError_t e = pack(p, image(0), image(1), pq2, pk2, pp.r, rows, &in, stream, launches);
    in.add(p.v, p.d / 2, image(2), pp.d / 2, rows);
    in.add(p.dout, p.d / 2, image(4), pp.d / 2, rows);
    if (!direct) in.add(p.out, p.d / 2, image(3), pp.d / 2, rows);
    if (!e) e = run_copies(in, stream, launches);
    if (!e) {
        pp.q = image(0); pp.k = image(1); pp.v = image(2); pp.out = direct ? p.out : image(3); pp.dout = image(4);
        pp.dq = direct ? p.dq : image(5); pp.dk = image(6); pp.dv = image(7);
        pp.pq = pq2; pp.pk = pk2; pp.dpq = dpq2; pp.dpk = dpk2;
        e = sm100_bwd(pp, stream);
        *launches += sm100_bwd_launches(pp);
    }
    RowCopies back{};
    if (!direct) back.add(image(5), pp.d / 2, p.dq, p.d / 2, rows);
    back.add(image(6), pp.d / 2, p.dk, p.d / 2, rows);
    back.add(image(7), pp.d / 2, p.dv, p.d / 2, rows);
    if (tables_in_a_row(p)) {
        back.add(dpq2, pp.r, p.dpq, p.r, (size_t)tables * p.n);
        back.add(dpk2, pp.r, p.dpk, p.r, (size_t)tables * p.n);
    } else {
        if (!e) e = copy_tables<float2>(dpq2, tstride, pp.r, p.dpq, p.pos_head_stride, p.r, tables, p.n, stream, launches);
        if (!e) e = copy_tables<float2>(dpk2, tstride, pp.r, p.dpk, p.pos_head_stride, p.r, tables, p.n, stream, launches);
    }
    if (!e) e = run_copies(back, stream, launches);
    if (!e && rank_tail(p)) {
        // (the copies above have cleared the columns from 32 on: the tail's gradients are summed into them)
        const PlaceGeom g = place_geom(p);
        const size_t total = rows * (size_t)g.extra;
        const unsigned blocks = (unsigned)((total + 255) / 256 < 148 * 16 ? (total + 255) / 256 : 148 * 16);
        rib_rank_tail_grads_kernel<<<blocks, 256, 0, stream>>>(image(5), image(6), p.dpq, p.dpk, g, (unsigned)rows);
        ++*launches;
        e = cudaGetLastError();
    }
    const cudaError_t f = cudaFreeAsync(buf, stream);
    return e ? e : f;
}

// ------------------------------------------------------------------------------------------------------------------
// The CLA gate kernels take D = 64, 128 or 192 channels.  Other even D up to 192 (6 heads of 30 or of 16 channels: 180,
// 96) run on them through copies with the channel dimension filled up with zeros: zero weights keep the added channels
// out of every real one (their own gate is sigmoid(0), which is dropped), and their gradients are zero.
// ------------------------------------------------------------------------------------------------------------------
namespace {

// dst[r][c] = src[r][c] where both have the entry, 0 elsewhere (fp32 matrices: weights in, gradients out)
__global__ void __launch_bounds__(256) rib_fit_matrix_kernel(const float* __restrict__ src, int rs, int cs, float* __restrict__ dst, int rd, int cd)
{
    const int total = rd * cd;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int r = e / cd, c = e - r * cd;
        dst[e] = r < rs && c < cs ? src[r * cs + c] : 0.f;
    }
}

cudaError_t fit_matrix(const float* src, int rs, int cs, float* dst, int rd, int cd, cudaStream_t stream, int* launches)
{
    rib_fit_matrix_kernel<<<(rd * cd + 255) / 256, 256, 0, stream>>>(src, rs, cs, dst, rd, cd);
    ++*launches;
    return cudaGetLastError();
}

struct PaddedWeights { float *w_dw, *b_dw, *w_pw, *b_pw; size_t bytes; };

size_t weight_bytes(int Dp) { return up256((size_t)Dp * 9 * 4) + 2 * up256((size_t)Dp * 4) + up256((size_t)Dp * Dp * 4); }

PaddedWeights weight_layout(uint8_t* base, int Dp)
{
    PaddedWeights w;
    size_t off = 0;
    w.w_dw = reinterpret_cast<float*>(base + off); off += up256((size_t)Dp * 9 * 4);
    w.b_dw = reinterpret_cast<float*>(base + off); off += up256((size_t)Dp * 4);
    w.w_pw = reinterpret_cast<float*>(base + off); off += up256((size_t)Dp * Dp * 4);
    w.b_pw = reinterpret_cast<float*>(base + off); off += up256((size_t)Dp * 4);
    w.bytes = off;
    return w;
}

}  // namespace

int cla_padded_channels(int D)
{
    if (D <= 0 || D > 192 || (D & 1)) return 0;
    return D <= 64 ? 64 : D <= 128 ? 128 : 192;
}

cudaError_t cla_gate_padded(const __nv_bfloat16* x, const float* w_dw, const float* b_dw, const float* w_pw, const float* b_pw, int B, int H,
                            int W, int D, __nv_bfloat16* gate, int* status, cudaStream_t stream, int* launches)
{
    *launches = 0;
    const int Dp = cla_padded_channels(D);
    const size_t pixels = (size_t)B * H * W, img = up256(pixels * Dp * 2);
    const size_t wbytes = weight_bytes(Dp);
    uint8_t* buf = nullptr;
    if (cudaError_t e = scratch_alloc(&buf, 2 * img + wbytes, stream)) return e;
    __nv_bfloat16* x2 = reinterpret_cast<__nv_bfloat16*>(buf);
    __nv_bfloat16* g2 = reinterpret_cast<__nv_bfloat16*>(buf + img);
    const PaddedWeights w = weight_layout(buf + 2 * img, Dp);
    cudaError_t e = resize_rows(x, D, x2, Dp, pixels, stream, launches);
    if (!e) e = fit_matrix(w_dw, D, 9, w.w_dw, Dp, 9, stream, launches);
    if (!e) e = fit_matrix(b_dw, 1, D, w.b_dw, 1, Dp, stream, launches);
    if (!e) e = fit_matrix(w_pw, D, D, w.w_pw, Dp, Dp, stream, launches);
    if (!e) e = fit_matrix(b_pw, 1, D, w.b_pw, 1, Dp, stream, launches);
    if (!e) { e = cla_gate(x2, w.w_dw, w.b_dw, w.w_pw, w.b_pw, B, H, W, Dp, g2, status, stream); ++*launches; }
    if (!e) e = resize_rows(g2, Dp, gate, D, pixels, stream, launches);
    const cudaError_t f = cudaFreeAsync(buf, stream);
    return e ? e : f;
}

cudaError_t cla_gate_bwd_padded(const __nv_bfloat16* x, const float* w_dw, const float* b_dw, const float* w_pw, const float* b_pw,
                                const __nv_bfloat16* dgate, int B, int H, int W, int D, __nv_bfloat16* dx, float* dw_dw, float* db_dw,
                                float* dw_pw, float* db_pw, void* workspace, bool tensor_cores, int* status, cudaStream_t stream, int* launches)
{
    *launches = 0;
    const int Dp = cla_padded_channels(D);
    const size_t pixels = (size_t)B * H * W, img = up256(pixels * Dp * 2);
    const size_t wbytes = weight_bytes(Dp);
    uint8_t* buf = nullptr;
    if (cudaError_t e = scratch_alloc(&buf, 3 * img + 2 * wbytes, stream)) return e;
    __nv_bfloat16* x2 = reinterpret_cast<__nv_bfloat16*>(buf);
    __nv_bfloat16* dg2 = reinterpret_cast<__nv_bfloat16*>(buf + img);
    __nv_bfloat16* dx2 = reinterpret_cast<__nv_bfloat16*>(buf + 2 * img);
    const PaddedWeights w = weight_layout(buf + 3 * img, Dp), g = weight_layout(buf + 3 * img + wbytes, Dp);
    cudaError_t e = resize_rows(x, D, x2, Dp, pixels, stream, launches);
    if (!e) e = resize_rows(dgate, D, dg2, Dp, pixels, stream, launches);
    if (!e) e = fit_matrix(w_dw, D, 9, w.w_dw, Dp, 9, stream, launches);
    if (!e) e = fit_matrix(b_dw, 1, D, w.b_dw, 1, Dp, stream, launches);
    if (!e) e = fit_matrix(w_pw, D, D, w.w_pw, Dp, Dp, stream, launches);
    if (!e) e = fit_matrix(b_pw, 1, D, w.b_pw, 1, Dp, stream, launches);
    if (!e) {
        e = cla_gate_bwd(x2, w.w_dw, w.b_dw, w.w_pw, w.b_pw, dg2, B, H, W, Dp, dx2, g.w_dw, g.b_dw, g.w_pw, g.b_pw, workspace, tensor_cores, status, stream);
        *launches += tensor_cores ? 3 : 4;
    }
    if (!e) e = resize_rows(dx2, Dp, dx, D, pixels, stream, launches);
    if (!e) e = fit_matrix(g.w_dw, Dp, 9, dw_dw, D, 9, stream, launches);
    if (!e) e = fit_matrix(g.b_dw, 1, Dp, db_dw, 1, D, stream, launches);
    if (!e) e = fit_matrix(g.w_pw, Dp, Dp, dw_pw, D, D, stream, launches);
    if (!e) e = fit_matrix(g.b_pw, 1, Dp, db_pw, 1, D, stream, launches);
    const cudaError_t f = cudaFreeAsync(buf, stream);
    return e ? e : f;
}

}  // namespace rib
