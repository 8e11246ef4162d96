// Shared between the tcgen05 forward and backward kernels: the tile geometry (tiles of two 8x8-token
// patches), the work-item decoding and the host-side TMA tensor-map encoders.
#pragma once
#include "rib_common.cuh"
#include "sm100_primitives.cuh"

#include <string.h>
#include <mutex>

namespace rib {
namespace sm100 {

constexpr int kD = 32, kR = 16;
constexpr int kTile = 128;                             // tokens of a query tile / key block
constexpr uint32_t kContentBytes = kTile * kD * 2;     // 8192: 128 rows x 64 B, SWIZZLE_64B
constexpr uint32_t kPosBytes = kTile * kR * 2;         // 4096: 128 rows x 32 B, SWIZZLE_32B
constexpr uint32_t kPatchContent = kContentBytes / 2, kPatchPos = kPosBytes / 2;

// A tile is not 128 consecutive tokens of the window but two 8x8-token patches: attention is
// equivariant to the order of tokens inside a window, so any enumeration works as long as the
// Pq/Pk rows and the output rows follow it.  An 8x8 patch never straddles the image border when
// the shift is a multiple of 8, so one TMA box per patch does partition and shift.
// "Window order" below means this enumeration: token w of a window lies in patch w / 64 (patches
// row-major over the window), at row (w / 8) % 8 and column w % 8 of the patch.
struct WindowGeom { int H, W, M, s; };

// Division of a non-negative int below 2^31 by a constant set on the host: q = (n * mul) >> shr, exact for every
// such n (mul = floor(2^shr / d) + 1 with shr = 31 + ceil(log2 d), so the error term n * (mul * d - 2^shr) stays
// below 2^shr).  The kernels decode work items with it instead of the emulated 32-bit division.
struct FastDiv {
    uint32_t mul, shr, d;
    __host__ __device__ __forceinline__ int div(int n) const { return (int)(((unsigned long long)(uint32_t)n * mul) >> shr); }
    __host__ __device__ __forceinline__ void divmod(int n, int& q, int& r) const { q = div(n); r = n - q * (int)d; }
};
inline FastDiv make_fast_div(int d)
{
    uint32_t l = 0;
    while ((1u << l) < (uint32_t)d) ++l;
    FastDiv f;
    f.shr = 31 + l;
    f.mul = (uint32_t)(((1ull << f.shr) / (uint32_t)d) + 1ull);
    f.d = (uint32_t)d;
    return f;
}

// Patch `sp` of window (wy, wx): top-left token in window coordinates (py, px) and in shifted,
// wrapped image coordinates (Y0, X0).
__host__ __device__ __forceinline__ void patch_origin(const WindowGeom& g, int wy, int wx, int sp, int& py, int& px,
                                                      int& Y0, int& X0)
{
    const int per_row = g.M >> 3;
    py = (sp / per_row) << 3;
    px = (sp % per_row) << 3;
    Y0 = wy * g.M + py + g.s; if (Y0 >= g.H) Y0 -= g.H;
    X0 = wx * g.M + px + g.s; if (X0 >= g.W) X0 -= g.W;
}

// The same with the division by the patches per window row prepared on the host.
__device__ __forceinline__ void patch_origin(const WindowGeom& g, const FastDiv& per_row, int wy, int wx, int sp, int& py, int& px,
                                             int& Y0, int& X0)
{
    int q, r;
    per_row.divmod(sp, q, r);
    py = q << 3;
    px = r << 3;
    Y0 = wy * g.M + py + g.s; if (Y0 >= g.H) Y0 -= g.H;
    X0 = wx * g.M + px + g.s; if (X0 >= g.W) X0 -= g.W;
}

// Window-order index w -> row of Pq/Pk (i = y * M + x) and image pixel of window (wy, wx).
__host__ __device__ __forceinline__ void window_order_token(const WindowGeom& g, int wy, int wx, int w, int& i,
                                                            int& Y, int& X)
{
    int py, px, Y0, X0;
    patch_origin(g, wy, wx, w >> 6, py, px, Y0, X0);
    const int ty = (w >> 3) & 7, tx = w & 7;
    i = (py + ty) * g.M + px + tx;
    Y = Y0 + ty;
    X = X0 + tx;
}

// ------------------------------------------------------------------------- windows of a map that they do not divide
// Windows are laid over the map extended to Hp x Wp; positions beyond H x W are no tokens.  Attention does not depend on
// the order of a window's tokens, so a kernel may walk only the patches that hold some: along each axis a window has a list
// of such patch rows (columns), which is one or two runs, and patch k of the window is (row k / cols, column k % cols) of
// the two lists.  Along an axis every window but the last one or two is full (the positions beyond the map are fewer than
// a window, and the shift is smaller than one), which gives at most three kinds of window per axis and nine in the map;
// the work items (two query tiles = four patches each) are numbered kind by kind, full windows first, so that the items
// dealt out last are the short ones.
struct AxisKind { int count, start0, len0, start1, first; FastDiv by_count, by_windows; };      // patches; first window and number of windows of the kind
struct LiveWindows {
    AxisKind y[3], x[3];
    int offset[10];                  // first item of kind 3 * ky + kx; offset[9]: all items
    FastDiv items_per_window[9];
    FastDiv by_heads;
};
struct LiveItem { int b, h, wy, wx, tp, ky, kx, patches; };

__host__ __device__ __forceinline__ LiveItem decode_live_item(const LiveWindows& g, int item)
{
    LiveItem c;
    int kind = 0;
#pragma unroll
    for (int k = 1; k < 9; ++k) kind += item >= g.offset[k] ? 1 : 0;
    c.ky = kind / 3; c.kx = kind - 3 * c.ky;
    int rest = item - g.offset[kind], i;
    g.items_per_window[kind].divmod(rest, rest, c.tp);
    g.by_heads.divmod(rest, rest, c.h);
    g.x[c.kx].by_windows.divmod(rest, rest, i);
    c.wx = g.x[c.kx].first + i;
    g.y[c.ky].by_windows.divmod(rest, c.b, i);
    c.wy = g.y[c.ky].first + i;
    c.patches = g.y[c.ky].count * g.x[c.kx].count;
    return c;
}
// Patch k of the item's window: top-left token in window coordinates and in shifted, wrapped coordinates of the extended map.
__host__ __device__ __forceinline__ void live_patch_origin(const LiveWindows& g, const WindowGeom& w, const LiveItem& c, int k, int& py, int& px,
                                                           int& Y0, int& X0)
{
    const AxisKind &ay = g.y[c.ky], &ax = g.x[c.kx];
    int r, l;
    ax.by_count.divmod(k, r, l);
    py = (r < ay.len0 ? ay.start0 + r : ay.start1 + r - ay.len0) << 3;
    px = (l < ax.len0 ? ax.start0 + l : ax.start1 + l - ax.len0) << 3;
    Y0 = c.wy * w.M + py + w.s; if (Y0 >= w.H) Y0 -= w.H;
    X0 = c.wx * w.M + px + w.s; if (X0 >= w.W) X0 -= w.W;
}

// With a mask between the wrapped parts of shifted windows the parts of the last window are windows of their own: two kinds,
// the patch rows (columns) before position M - s and those from it on.
inline int masked_axis_kinds(int size, int M, int s, AxisKind (&kinds)[3], int (&windows)[3])
{
    const int n = size / M, per_row = M / 8, cut = (M - s) / 8;
    int used = 0;
    auto add = [&](int first, int count, int start, int len) {
        kinds[used] = AxisKind{len, start, len, 0, first, make_fast_div(len), make_fast_div(count)};
        windows[used++] = count;
    };
    if (n - (s ? 1 : 0) > 0) add(0, n - (s ? 1 : 0), 0, per_row);
    if (s) { add(n - 1, 1, 0, cut); add(n - 1, 1, cut, per_row - cut); }
    return used;
}

// The kinds of window along an axis of `size` positions; returns their number, 0 if the axis is not of the form above.
inline int axis_kinds(int size, int M, int s, AxisKind (&kinds)[3], int (&windows)[3])
{
    const int n = (size + M - 1) / M, extended = n * M, per_row = M / 8;
    int used = 0;
    for (int w = 0; w < n; ++w) {
        AxisKind k{};
        int runs = 0, last = -2;
        for (int l = 0; l < per_row; ++l) {
            if ((w * M + 8 * l + s) % extended >= size) continue;
            if (last != l - 1) {
                if (runs == 0) k.start0 = l; else k.start1 = l;
                ++runs;
            }
            if (runs == 1) ++k.len0;
            last = l;
            ++k.count;
        }
        if (k.count == 0 || runs > 2) return 0;
        k.first = w;
        const bool full = k.count == per_row;
        if (full && used == 1 && kinds[0].count == per_row) { ++windows[0]; continue; }
        if (used == 3 || (full && used > 0)) return 0;
        kinds[used] = k;
        windows[used++] = 1;
    }
    for (int i = 0; i < used; ++i) { kinds[i].by_count = make_fast_div(kinds[i].count); kinds[i].by_windows = make_fast_div(windows[i]); }
    return used;
}

inline bool make_live_windows(const Problem& p, LiveWindows* g)
{
    int ny_windows[3] = {0, 0, 0}, nx_windows[3] = {0, 0, 0};
    *g = LiveWindows{};
    const int ny = p.masked ? masked_axis_kinds(p.H, p.M, p.s, g->y, ny_windows) : axis_kinds(p.H, p.M, p.s, g->y, ny_windows);
    const int nx = p.masked ? masked_axis_kinds(p.W, p.M, p.s, g->x, nx_windows) : axis_kinds(p.W, p.M, p.s, g->x, nx_windows);
    if (!ny || !nx) return false;
    long long at = 0;
    for (int k = 0; k < 9; ++k) {
        g->offset[k] = (int)at;
        const int ky = k / 3, kx = k % 3;
        if (ky >= ny || kx >= nx) { g->items_per_window[k] = make_fast_div(1); continue; }
        const int per_window = (g->y[ky].count * g->x[kx].count + 3) / 4;
        g->items_per_window[k] = make_fast_div(per_window);
        at += (long long)p.B * p.heads * ny_windows[ky] * nx_windows[kx] * per_window;
        if (at > 0x7fffffffLL) return false;
    }
    g->offset[9] = (int)at;
    g->by_heads = make_fast_div(p.heads);
    return true;
}

// ---------------------------------------------------------------------------------- host side
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    });
    return fn;
}

// Tensor maps depend on the base pointer and the shape only, and a training loop calls with the same few buffers
// over and over: the maps of the process are kept in 256 sets of 8, the one that was not asked for longest giving way (one mutex), so
// a repeated call encodes nothing.  A layer's two passes need up to 9 maps of their own (general kernels: q, k, v and Pk of the forward, dout, Pk as
// 64-byte rows, dk and dv in boxes of 4 rows, Pq in the workspace), so the 64 layers that the cycle entry points take need 576.  The key holds
// every argument of the encoding.
struct MapKey {
    const void* ptr; long long a, b; int kind, c, d, e, f, g;
    bool operator==(const MapKey& o) const
    {
        return ptr == o.ptr && a == o.a && b == o.b && kind == o.kind && c == o.c && d == o.d && e == o.e && f == o.f && g == o.g;
    }
    unsigned hash() const
    {
        unsigned long long h = 0;
        for (unsigned long long x : {(unsigned long long)(uintptr_t)ptr, (unsigned long long)a, (unsigned long long)b, (unsigned long long)(uint32_t)kind << 32 | (uint32_t)c,
                                     (unsigned long long)(uint32_t)d << 32 | (uint32_t)e, (unsigned long long)(uint32_t)f << 32 | (uint32_t)g}) {
            h = (h ^ x) * 0x9e3779b97f4a7c15ull;
            h ^= h >> 32;
        }
        return (unsigned)h;
    }
};
constexpr int kMapSets = 256, kMapWays = 8;
struct MapCache {
    struct Entry { CUtensorMap map; MapKey key; unsigned long long asked; };      // asked: when last (0: empty)
    std::mutex mutex;
    Entry entries[kMapSets][kMapWays];
    long long hits = 0, misses = 0;
    MapCache() { memset(static_cast<void*>(entries), 0, sizeof entries); }      // its 512 KB of pages once, not one by one in later calls
};
inline MapCache& map_cache()
{
    static MapCache cache;
    return cache;
}
template <typename Encode>
inline bool cached_map(CUtensorMap* map, const MapKey& key, Encode encode)
{
    MapCache& c = map_cache();
    std::lock_guard<std::mutex> lock(c.mutex);
    MapCache::Entry *const set = c.entries[key.hash() % kMapSets], *slot = set;
    const unsigned long long now = (unsigned long long)(c.hits + c.misses) + 1;
    for (int i = 0; i < kMapWays; ++i) {
        if (set[i].asked && set[i].key == key) { *map = set[i].map; set[i].asked = now; ++c.hits; return true; }
        if (set[i].asked < slot->asked) slot = set + i;
    }
    if (!encode(map)) return false;
    ++c.misses;
    *slot = MapCache::Entry{*map, key, now};
    return true;
}
inline void map_cache_counts(long long* hits, long long* misses)
{
    MapCache& c = map_cache();
    std::lock_guard<std::mutex> lock(c.mutex);
    *hits = c.hits; *misses = c.misses;
}

// bf16 [B][H][W][heads][d] image tensor (d = 8, 16, 24 or 32), box = one 8x8-token patch of one head, always 32 channels
// wide: on a narrower head the channels from d on lie beyond the tensor and arrive as zeros, so a tile has one layout
// for every head width and the zero channels change no dot product.
inline bool encode_image_map_now(CUtensorMap* map, const void* ptr, const Problem& p, int rows)
{
    const cuuint64_t dims[5] = {(cuuint64_t)p.d, (cuuint64_t)p.heads, (cuuint64_t)p.W, (cuuint64_t)p.H, (cuuint64_t)p.B};
    const cuuint64_t row = (cuuint64_t)p.d * 2;
    const cuuint64_t strides[4] = {row, row * p.heads, row * p.heads * p.W, row * p.heads * p.W * p.H};
    const cuuint32_t box[5] = {(cuuint32_t)kD, 1, 8, (cuuint32_t)rows, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(ptr), dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 [tables][M][M][r] positional features (one table shared by all heads, or one per head; r = p.r), box = one
// 8x8-token patch of one table.  `tables` = 1 or heads, `table_stride` elements apart (a multiple of 8,
// at least M * M * 16); a kernel addresses table h * (tables > 1).
// (`rows`: token rows of a box; 4 for the half patch that one warp holds)
inline bool encode_image_map(CUtensorMap* map, const void* ptr, const Problem& p, int rows = 8)
{
    const MapKey key{ptr, rows, 0, 1, p.B, p.H, p.W, p.heads, p.d};
    return cached_map(map, key, [&](CUtensorMap* m) { return encode_image_map_now(m, ptr, p, rows); });
}

inline bool encode_pos_map_now(CUtensorMap* map, const void* ptr, const Problem& p, int tables, long long table_stride,
                               cuuint32_t box_inner, CUtensorMapSwizzle swz, int cols)
{
    const cuuint64_t side = p.M;
    const cuuint64_t dims[4] = {(cuuint64_t)cols, side, side, (cuuint64_t)tables};
    const cuuint64_t one_table = (cuuint64_t)cols * 2 * side * side;
    const cuuint64_t strides[3] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * 2 * side,
                                   tables > 1 ? (cuuint64_t)table_stride * 2 : one_table};
    const cuuint32_t box[4] = {box_inner, 8, 8, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr), dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// `cols`: elements per row of the table in memory (the rank, or the padded rank of a table staged by the library)
inline bool encode_pos_map_impl(CUtensorMap* map, const void* ptr, const Problem& p, int tables, long long table_stride,
                                cuuint32_t box_inner, CUtensorMapSwizzle swz, int cols)
{
    const MapKey key{ptr, table_stride, 0, 2, cols, p.M, tables, (int)box_inner, (int)swz};
    return cached_map(map, key, [&](CUtensorMap* m) { return encode_pos_map_now(m, ptr, p, tables, table_stride, box_inner, swz, cols); });
}
// Rows of 16 (r <= 16) or 32 (r <= 32) elements: a rank below the row width is filled up with zeros by TMA.
inline int padded_rank(int r) { return r > 16 ? 32 : 16; }

inline bool encode_pos_map(CUtensorMap* map, const void* ptr, const Problem& p, int tables, long long table_stride)
{
    const bool wide = padded_rank(p.r) == 32;
    return encode_pos_map_impl(map, ptr, p, tables, table_stride, wide ? 32u : 16u, wide ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B, p.r);
}
// The same features fetched as 64-byte rows: the box is 32 elements wide on a 16-element dimension, so
// TMA fills the upper half of every row with zeros.  A 64-byte-row RIB tile has the layout of a content
// tile (SWIZZLE_64B) and can sit behind it as the second 32-column atom of one MN-major operand.
inline bool encode_pos_map_padded(CUtensorMap* map, const void* ptr, const Problem& p, int tables, long long table_stride, int cols)
{
    return encode_pos_map_impl(map, ptr, p, tables, table_stride, kD, CU_TENSOR_MAP_SWIZZLE_64B, cols);
}

inline cudaError_t sm_count_of_current_device(int* count)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(count, cudaDevAttrMultiProcessorCount, dev);
    return e;
}

// Per-kernel, per-device launch set-up: the dynamic shared-memory limit of a kernel is an attribute of the kernel on
// ONE device, so a process that drives several GPUs has to raise it on each of them.  One instance of this struct per
// kernel (a function-local static); prepare() raises the limit on the current device the first time it is seen there
// and returns that device's SM count.
struct KernelSetup {
    static constexpr int kMaxDevices = 64;
    std::mutex mutex;
    int sm_count[kMaxDevices] = {};
    template <typename Kernel>
    cudaError_t prepare(Kernel kernel, uint32_t smem_bytes, int* sms)
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(mutex);
        if (!sm_count[dev]) {
            int count = 0;
            e = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
            if (e != cudaSuccess) return e;
            sm_count[dev] = count;
        }
        *sms = sm_count[dev];
        return cudaSuccess;
    }
};

}  // namespace sm100
}  // namespace rib
