// RIB feature generator (Eq. 1-3 of the paper): window coordinates -> Fourier features -> one ReLU
// layer shared by all heads -> two linear projections to the rank-r positional features Pq, Pk that
// the attention entry points take, and the chain rule of those steps.
//
// The problem is tiny (n = window^2 <= 4096 tokens, a 42 x 32 and two 32 x 16 matrices at the paper's sizes: a few MFLOP and
// well under a megabyte), so what bounds it is the serial chain inside one block and the launches.  A block therefore takes
// only kTokens tokens and spreads every step over all of its threads: a thread evaluates single Fourier features and then
// 4-column pieces of the hidden rows, of the projections and, in the backward pass, of the weight gradients, which are
// summed over the block's tokens and added to global memory with one atomic per piece.  The gradients are cleared by one
// small kernel that the main kernel overtakes (programmatic dependent launch) up to its first atomic.  The weights reach shared
// memory by asynchronous copies while the features are computed.  Measured by event hooks (which include about 7 us per call) at window
// 32, L = 10, dh = 32, r = 16: forward 10.4 us, backward 12.8 us (staged by loads and stores, 128 threads a block: 10.8 and 14.9; a
// thread owning a whole token of a block of 128: 39.5 and 119.8); both calls at window 64, L = 12, dh = 48, r = 32: 41.4 -> 31.3 us.
//
// Coordinates: window points run from -1 to 1 inclusive on both axes (a single point sits at 0); token
// i = y * window + x has the coordinate (row, column); Eq. 1 literally, frequencies 2^l without pi.
#include "rib_common.cuh"

namespace rib {
namespace {

constexpr int kThreads = 256;
constexpr int kTokens = 16;      // tokens of a block: 64 blocks at window 32; the gradients' atomics grow with the number of blocks

struct GenParams {
    const float* w_h;      // [2 + 4 L][dh]
    const float* b_h;      // [dh]
    const float* w_pq;     // [dh][r]
    const float* w_pk;     // [dh][r]
    const float* dpq;      // [n][r]  (backward)
    const float* dpk;
    __nv_bfloat16* pq;     // [n][r]  (forward)
    __nv_bfloat16* pk;
    float* dw_h; float* db_h; float* dw_pq; float* dw_pk;
    int M, n, L, in, dh, r;
};

__device__ __forceinline__ double coordinate(int idx, int M) { return M == 1 ? 0.0 : -1.0 + 2.0 * (double)idx / (double)(M - 1); }

// The argument 2^l x of a sine and a cosine of Eq. 1, reduced to [-pi, pi].  It reaches thousands of radians at the upper
// bands, where a coordinate rounded to fp32 would be off by a visible fraction of a radian: the coordinate and the reduction
// are done in double (a handful of operations per argument), the sine itself in fp32.
// Feature order: [x, sin(2^0 x), cos(2^0 x), ...], every block 2 wide.
__device__ __forceinline__ float band_argument(double c, int l)
{
    double arg = ldexp(c, l);
    arg -= 6.283185307179586476925 * rint(arg * 0.15915494309189533577);
    return (float)arg;
}

// Shared memory: every row is padded with zeros to a multiple of 4 floats, so that a thread can take 4 columns at a time.
struct GenSmem {
    int dhp, rp;                        // padded widths
    float *w_h, *b_h, *w_pq, *w_pk;     // [in][dhp], [dhp], [dh][rp], [dh][rp]
    float *feat, *h;                    // [kTokens][in], [kTokens][dhp]
    float *da, *dq, *dk;                // backward: [kTokens][dhp], [kTokens][rp], [kTokens][rp]
};
__host__ __device__ inline int pad4(int w) { return (w + 3) & ~3; }
__host__ __device__ inline size_t smem_floats(int in, int dh, int r, bool backward)
{
    const size_t dhp = pad4(dh), rp = pad4(r), inp = pad4(in);
    return in * dhp + dhp + 2 * dh * rp + kTokens * (inp + dhp) + (backward ? kTokens * (dhp + 2 * rp) : 0);
}
__device__ __forceinline__ GenSmem carve(const GenParams& p, float* sm)
{
    GenSmem s;
    s.dhp = pad4(p.dh); s.rp = pad4(p.r);
    s.w_h = sm; s.b_h = s.w_h + p.in * s.dhp; s.w_pq = s.b_h + s.dhp; s.w_pk = s.w_pq + p.dh * s.rp;
    s.h = s.w_pk + p.dh * s.rp; s.da = s.h + kTokens * s.dhp; s.dq = s.da + kTokens * s.dhp; s.dk = s.dq + kTokens * s.rp;
    s.feat = s.h + kTokens * s.dhp;     // forward: behind h; the backward kernel moves it behind dk
    return s;
}

// A matrix into shared memory, rows of ws floats to rows of wd (zeros behind, and beyond real_rows).  Rows that are whole 16-byte
// pieces travel asynchronously: the copies of all matrices are in flight while the Fourier features are computed
// (staged_arrived before the first use).
__device__ __forceinline__ void stage(float* dst, int wd, const float* src, int ws, int rows, int real_rows)
{
    const int pieces = wd / 4;
    for (int i = threadIdx.x; i < rows * pieces; i += kThreads) {
        const int row = i / pieces, c = 4 * (i - row * pieces);
        const float* from = src + (size_t)row * ws + c;
        if (ws == wd && row < real_rows) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + 4 * i)), "l"(from) : "memory");
        } else {
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = row < real_rows && c + k < ws ? from[k] : 0.f;
            *reinterpret_cast<float4*>(dst + 4 * i) = make_float4(v[0], v[1], v[2], v[3]);
        }
    }
}
__device__ __forceinline__ void staged_arrived()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

__device__ __forceinline__ void fma4(float4& a, float x, const float4& w)
{
    a.x = fmaf(x, w.x, a.x); a.y = fmaf(x, w.y, a.y); a.z = fmaf(x, w.z, a.z); a.w = fmaf(x, w.w, a.w);
}

// Features of the block's tokens, then h = ReLU(r_in W_h + b_h) (Eq. 1, Eq. 2); rows beyond the last token are zero.
__device__ __forceinline__ void features_and_hidden(const GenParams& p, const GenSmem& s, int token0)
{
    const int items = kTokens * (1 + 2 * p.L);         // per token the coordinates and, per band and axis, a sine and a cosine
    for (int e = threadIdx.x; e < items; e += kThreads) {
        const int t = e % kTokens, k = e / kTokens, token = token0 + t;
        float* row = s.feat + t * p.in;
        const int y = token / p.M, x = token - y * p.M;
        const double cy = coordinate(y, p.M), cx = coordinate(x, p.M);
        const bool live = token < p.n;
        if (k == 0) {
            row[0] = live ? (float)cy : 0.f;
            row[1] = live ? (float)cx : 0.f;
        } else {
            const int axis = (k - 1) & 1, l = (k - 1) >> 1;
            const float arg = band_argument(axis ? cx : cy, l);
            row[2 + 4 * l + axis] = live ? sinf(arg) : 0.f;
            row[4 + 4 * l + axis] = live ? cosf(arg) : 0.f;
        }
    }
    staged_arrived();
    const int pieces = s.dhp / 4;
    for (int e = threadIdx.x; e < kTokens * pieces; e += kThreads) {
        const int t = e / pieces, j = 4 * (e - t * pieces);
        float4 a = *reinterpret_cast<const float4*>(s.b_h + j);
        const float* f = s.feat + t * p.in;
#pragma unroll 4
        for (int i = 0; i < p.in; ++i) fma4(a, f[i], *reinterpret_cast<const float4*>(s.w_h + i * s.dhp + j));
        const bool live = token0 + t < p.n;
        *reinterpret_cast<float4*>(s.h + t * s.dhp + j) =
            live ? make_float4(fmaxf(a.x, 0.f), fmaxf(a.y, 0.f), fmaxf(a.z, 0.f), fmaxf(a.w, 0.f)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------------- forward
__global__ void __launch_bounds__(kThreads) rib_generator_fwd_kernel(const GenParams p)
{
    extern __shared__ __align__(16) float sm[];
    const GenSmem s = carve(p, sm);
    stage(s.w_h, s.dhp, p.w_h, p.dh, p.in, p.in); stage(s.b_h, s.dhp, p.b_h, p.dh, 1, 1);
    stage(s.w_pq, s.rp, p.w_pq, p.r, p.dh, p.dh); stage(s.w_pk, s.rp, p.w_pk, p.r, p.dh, p.dh);
    const int token0 = blockIdx.x * kTokens;
    features_and_hidden(p, s, token0);
    const int pieces = s.rp / 4;
    for (int e = threadIdx.x; e < 2 * kTokens * pieces; e += kThreads) {                   // Eq. 3
        const bool is_k = e >= kTokens * pieces;
        const int e2 = is_k ? e - kTokens * pieces : e, t = e2 / pieces, c = 4 * (e2 - t * pieces);
        if (token0 + t >= p.n) continue;
        const float* w = (is_k ? s.w_pk : s.w_pq) + c;
        const float* h = s.h + t * s.dhp;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int j = 0; j < p.dh; ++j) fma4(a, h[j], *reinterpret_cast<const float4*>(w + j * s.rp));
        __nv_bfloat16* dst = (is_k ? p.pk : p.pq) + (size_t)(token0 + t) * p.r + c;
        const float v[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (c + k < p.r) dst[k] = __float2bfloat16_rn(v[k]);
    }
}

// --------------------------------------------------------------------------------- backward
__global__ void __launch_bounds__(256) rib_generator_clear_kernel(const GenParams p)
{
    cudaTriggerProgrammaticLaunchCompletion();         // the main kernel waits for this one's end before its first atomic
    const int n_wh = p.in * p.dh, n_pp = p.dh * p.r, t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_wh) p.dw_h[t] = 0.f;
    if (t < p.dh) p.db_h[t] = 0.f;
    if (t < n_pp) { p.dw_pq[t] = 0.f; p.dw_pk[t] = 0.f; }
}

// adds columns c .. c + 3 of a row of `width` floats
__device__ __forceinline__ void add4(float* row, int c, int width, const float4& v)
{
    if ((width & 3) == 0) { atomicAdd(reinterpret_cast<float4*>(row + c), v); return; }
    const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (c + k < width) atomicAdd(row + c + k, f[k]);
}

// Per block: features and h as above, da = (dPq W_pq^T + dPk W_pk^T) o [h > 0], then dW_h = r_in^T da, db_h = sum da,
// dW_pq = h^T dPq, dW_pk = h^T dPk over the block's tokens.
__global__ void __launch_bounds__(kThreads) rib_generator_bwd_kernel(const GenParams p)
{
    extern __shared__ __align__(16) float sm[];
    GenSmem s = carve(p, sm);
    s.feat = s.dk + kTokens * s.rp;
    const int token0 = blockIdx.x * kTokens, tokens = min(kTokens, p.n - token0);
    stage(s.w_h, s.dhp, p.w_h, p.dh, p.in, p.in); stage(s.b_h, s.dhp, p.b_h, p.dh, 1, 1);
    stage(s.w_pq, s.rp, p.w_pq, p.r, p.dh, p.dh); stage(s.w_pk, s.rp, p.w_pk, p.r, p.dh, p.dh);
    stage(s.dq, s.rp, p.dpq + (size_t)token0 * p.r, p.r, kTokens, tokens);
    stage(s.dk, s.rp, p.dpk + (size_t)token0 * p.r, p.r, kTokens, tokens);
    features_and_hidden(p, s, token0);
    for (int e = threadIdx.x; e < kTokens * s.dhp; e += kThreads) {
        const int t = e / s.dhp, j = e - t * s.dhp;
        float g = 0.f;
        if (j < p.dh && s.h[e] > 0.f) {
            const float4 *dq = reinterpret_cast<const float4*>(s.dq + t * s.rp), *dk = reinterpret_cast<const float4*>(s.dk + t * s.rp);
            const float4 *wq = reinterpret_cast<const float4*>(s.w_pq + j * s.rp), *wk = reinterpret_cast<const float4*>(s.w_pk + j * s.rp);
            for (int c = 0; c < s.rp / 4; ++c) {
                const float4 a = dq[c], b = wq[c], u = dk[c], v = wk[c];
                g = fmaf(a.x, b.x, fmaf(u.x, v.x, g)); g = fmaf(a.y, b.y, fmaf(u.y, v.y, g));
                g = fmaf(a.z, b.z, fmaf(u.z, v.z, g)); g = fmaf(a.w, b.w, fmaf(u.w, v.w, g));
            }
        }
        s.da[e] = g;
    }
    __syncthreads();
    cudaGridDependencySynchronize();                   // the results are cleared
    const int ph = s.dhp / 4, pr = s.rp / 4, n_h = (p.in + 1) * ph, n_p = p.dh * pr;       // the row behind W_h's is b_h
    for (int e = threadIdx.x; e < n_h + 2 * n_p; e += kThreads) {
        const float *left, *right;                     // columns of the two factors: their strides
        int ls, rs, c, width;
        float* dst;
        if (e < n_h) {
            const int f = e / ph;
            c = 4 * (e - f * ph); width = p.dh;
            left = f < p.in ? s.feat + f : nullptr; ls = p.in;
            right = s.da + c; rs = s.dhp;
            dst = f < p.in ? p.dw_h + f * p.dh : p.db_h;
        } else {
            const bool is_k = e >= n_h + n_p;
            const int e2 = e - n_h - (is_k ? n_p : 0), j = e2 / pr;
            c = 4 * (e2 - j * pr); width = p.r;
            left = s.h + j; ls = s.dhp;
            right = (is_k ? s.dk : s.dq) + c; rs = s.rp;
            dst = (is_k ? p.dw_pk : p.dw_pq) + j * p.r;
        }
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kTokens; ++k) fma4(acc, left ? left[k * ls] : 1.f, *reinterpret_cast<const float4*>(right + k * rs));
        add4(dst, c, width, acc);
    }
}

}  // namespace

bool generator_supported(int window, int L, int dh, int r)
{
    return window >= 1 && window <= 256 && L >= 0 && L <= 16 && dh >= 1 && dh <= 64 && r >= 1 && r <= 64;
}

cudaError_t generator_fwd(const float* w_h, const float* b_h, const float* w_pq, const float* w_pk, int window, int L, int dh, int r,
                          __nv_bfloat16* pq, __nv_bfloat16* pk, cudaStream_t stream)
{
    GenParams p{};
    p.w_h = w_h; p.b_h = b_h; p.w_pq = w_pq; p.w_pk = w_pk; p.pq = pq; p.pk = pk;
    p.M = window; p.n = window * window; p.L = L; p.in = 2 + 4 * L; p.dh = dh; p.r = r;
    const size_t smem = sizeof(float) * smem_floats(p.in, dh, r, false);
    cudaError_t e = smem > 48 * 1024 ? cudaFuncSetAttribute(rib_generator_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                                     : cudaSuccess;
    if (e != cudaSuccess) return e;
    ProfileScope scope(RIB_KERNEL_GENERATOR_FWD, stream);
    rib_generator_fwd_kernel<<<(p.n + kTokens - 1) / kTokens, kThreads, smem, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t generator_bwd(const float* w_h, const float* b_h, const float* w_pq, const float* w_pk, const float* dpq, const float* dpk,
                          int window, int L, int dh, int r, float* dw_h, float* db_h, float* dw_pq, float* dw_pk, cudaStream_t stream)
{
    GenParams p{};
    p.w_h = w_h; p.b_h = b_h; p.w_pq = w_pq; p.w_pk = w_pk; p.dpq = dpq; p.dpk = dpk;
    p.dw_h = dw_h; p.db_h = db_h; p.dw_pq = dw_pq; p.dw_pk = dw_pk;
    p.M = window; p.n = window * window; p.L = L; p.in = 2 + 4 * L; p.dh = dh; p.r = r;
    const size_t smem = sizeof(float) * smem_floats(p.in, dh, r, true);
    cudaError_t e = smem > 48 * 1024 ? cudaFuncSetAttribute(rib_generator_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                                     : cudaSuccess;
    if (e != cudaSuccess) return e;
    const int most = p.in * dh > dh * r ? p.in * dh : dh * r;
    { ProfileScope scope(RIB_KERNEL_GENERATOR_CLEAR, stream); rib_generator_clear_kernel<<<(most + 255) / 256, 256, 0, stream>>>(p); }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ProfileScope scope(RIB_KERNEL_GENERATOR_BWD, stream);
    return launch_overtaking(rib_generator_bwd_kernel, (p.n + kTokens - 1) / kTokens, kThreads, smem, stream, p);
}

}  // namespace rib
