// CUDA-core kernels: max pooling, patch gather of a thin chain input (the band "split" step), zero-padding of weight
// rows.  Operators: Sec. IV-A of the paper (block-wise and element-wise local operators).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "lop.h"
#include "lop_kernels.cuh"
#include "lop_gather.cuh"

namespace lop {

namespace {

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void from_f32(float &d, float v) { d = v; }
__device__ __forceinline__ void from_f32(__nv_bfloat16 &d, float v) { d = __float2bfloat16_rn(v); }

// idx = ((n * rows + r) * Wo + ow) * inner + g, taken apart with 32-bit divisions where the count allows it (a 64-bit
// division is a routine of several dozen instructions: four of them per thread outweigh a light kernel's real work).
__device__ __forceinline__ void split_index(long long idx, long long total, int inner, int Wo, int rows, int &g, int &ow, int &r, int &n)
{
    if (total < (1LL << 31)) {
        unsigned q = (unsigned)idx;
        const unsigned q1 = q / (unsigned)inner; g = (int)(q - q1 * (unsigned)inner);
        const unsigned q2 = q1 / (unsigned)Wo; ow = (int)(q1 - q2 * (unsigned)Wo);
        const unsigned q3 = q2 / (unsigned)rows; r = (int)(q2 - q3 * (unsigned)rows);
        n = (int)q3;
    } else {
        long long q = idx;
        g = (int)(q % inner); q /= inner;
        ow = (int)(q % Wo); q /= Wo;
        r = (int)(q % rows);
        n = (int)(q / rows);
    }
}

// ---------------------------------------------------------------------------------------------
// Max pooling, NHWC.  One thread per (output pixel, group of VEC channels); a warp covers
// consecutive channel groups of consecutive pixels, so loads and stores are 16-byte and coalesced.
// HBM-bound: bytes = rows read once + rows written once.
// ---------------------------------------------------------------------------------------------
template <typename T, int VEC>
struct alignas(sizeof(T) * VEC) Pack {
    T v[VEC];
};

template <typename T, int VEC>
__global__ void __launch_bounds__(256) maxpool_kernel(PoolArgs p)
{
    grid_release();
    const int rows = p.oh_hi - p.oh_lo;
    const int cg = p.C / VEC;
    const long long total = (long long)p.N * rows * p.Wo * cg;
    grid_wait();
    const T *__restrict__ x = from_here(static_cast<const T *>(p.x));
    T *__restrict__ y = static_cast<T *>(p.y);
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        int g, ow, r, n;
        split_index(idx, total, cg, p.Wo, rows, g, ow, r, n);
        const int oh = p.oh_lo + r;
        float m[VEC];
#pragma unroll
        for (int i = 0; i < VEC; ++i) m[i] = -INFINITY;
        for (int a = 0; a < p.kh; ++a) {
            const int ih = oh * p.sh - p.ph + a * p.dh;
            if (ih < 0 || ih >= p.Hin) continue;
            for (int b = 0; b < p.kw; ++b) {
                const int iw = ow * p.sw - p.pw + b * p.dw;
                if (iw < 0 || iw >= p.Win) continue;
                const long long xo = (((long long)n * p.Hin + ih) * p.Win + iw) * p.C + (long long)g * VEC;
                if (!dbg_in_bounds(p.dbg, xo, VEC, (long long)p.N * p.Hin * p.Win * p.C)) continue;
                const Pack<T, VEC> v = *reinterpret_cast<const Pack<T, VEC> *>(x + xo);
#pragma unroll
                for (int i = 0; i < VEC; ++i) m[i] = fmaxf(m[i], to_f32(v.v[i]));
            }
        }
        Pack<T, VEC> o;
#pragma unroll
        for (int i = 0; i < VEC; ++i) from_f32(o.v[i], m[i]);
        const long long yo = (((long long)n * p.Ho + oh) * p.Wo + ow) * p.C + (long long)g * VEC;
        if (dbg_in_bounds(p.dbg, yo, VEC, (long long)p.N * p.Ho * p.Wo * p.C)) *reinterpret_cast<Pack<T, VEC> *>(y + yo) = o;
    }
}

// bf16, channels a multiple of 8, a KH x KW window known at compile time: every tap's 16-byte load is issued
// before the first maximum is taken (four to nine independent loads in flight per thread), one thread per
// (output pixel, 8-channel group), as many blocks as there is work.
template <int KH, int KW>
__global__ void __launch_bounds__(256) maxpool_bf16x8_kernel(PoolArgs p)
{
    grid_release();
    const int rows = p.oh_hi - p.oh_lo;
    const int cg = p.C >> 3;
    const long long total = (long long)p.N * rows * p.Wo * cg;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    grid_wait();
    if (idx >= total) return;
    const uint4 *__restrict__ x = from_here(static_cast<const uint4 *>(p.x));
    int g, ow, r, n;
    split_index(idx, total, cg, p.Wo, rows, g, ow, r, n);
    const int oh = p.oh_lo + r;
    uint4 v[KH * KW];
    bool ok[KH * KW];
#pragma unroll
    for (int a = 0; a < KH; ++a) {
        const int ih = oh * p.sh - p.ph + a * p.dh;
#pragma unroll
        for (int b = 0; b < KW; ++b) {
            const int iw = ow * p.sw - p.pw + b * p.dw;
            ok[a * KW + b] = ih >= 0 && ih < p.Hin && iw >= 0 && iw < p.Win;
            const long long xo = (((long long)n * p.Hin + ih) * p.Win + iw) * cg + g;           // in 16-byte vectors
            ok[a * KW + b] = ok[a * KW + b] && dbg_in_bounds(p.dbg, xo, 1, (long long)p.N * p.Hin * p.Win * cg);
            if (ok[a * KW + b]) v[a * KW + b] = __ldg(x + xo);
        }
    }
    float m[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) m[i] = -INFINITY;
#pragma unroll
    for (int tpos = 0; tpos < KH * KW; ++tpos)
        if (ok[tpos]) {
            const uint32_t w4[4] = {v[tpos].x, v[tpos].y, v[tpos].z, v[tpos].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                m[2 * i] = fmaxf(m[2 * i], __uint_as_float(w4[i] << 16));
                m[2 * i + 1] = fmaxf(m[2 * i + 1], __uint_as_float(w4[i] & 0xFFFF0000u));
            }
        }
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)                      // the values are bf16 already: dropping the low half is exact
        o[i] = (__float_as_uint(m[2 * i]) >> 16) | (__float_as_uint(m[2 * i + 1]) & 0xFFFF0000u);
    const long long yo = (((long long)n * p.Ho + oh) * p.Wo + ow) * cg + g;
    if (dbg_in_bounds(p.dbg, yo, 1, (long long)p.N * p.Ho * p.Wo * cg)) static_cast<uint4 *>(p.y)[yo] = make_uint4(o[0], o[1], o[2], o[3]);
}

// ---------------------------------------------------------------------------------------------
// Patch gather for a thin chain input, rows [lo, hi) of the patch tensor (see lop_gather.cuh).
// One thread per 16-byte group of eight patch elements: consecutive threads write consecutive
// 16 bytes, reads hit the few image rows of the band in L1/L2.  HBM-bound on the write.
// The same launch brings the convolution's weights into the order of the gathered values where wp is given (a launch of
// its own costs two microseconds for a few kilobytes).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void stem_weights(const StemWeights &g, int first, int stride)
{
    const int total = g.cout * g.K, taps_c = g.kh * g.kw * g.C;
    for (int i = first; i < total; i += stride) {
        const int k = i % g.K, co = i / g.K;
        int src = k < taps_c ? k : -1;
        if (g.col) {
            const int b = k / g.col, r = k - b * g.col, a = r / g.C;
            src = b < g.kw && a < g.kh ? (a * g.kw + b) * g.C + (r - a * g.C) : -1;
        }
        static_cast<uint16_t *>(g.wp)[i] = src >= 0 ? static_cast<const uint16_t *>(g.w)[co * taps_c + src] : (uint16_t)0;
    }
}

template <typename Index>
__global__ void __launch_bounds__(256) stem_gather_kernel(const uint16_t *x_given, uint16_t *__restrict__ y,
                                                          GatherGeom g, int lo, int hi, StemWeights wt, unsigned *dbg)
{
    grid_release();
    grid_wait();
    const uint16_t *__restrict__ x = from_here(x_given);
    if (wt.clear && blockIdx.x == 0 && threadIdx.x == 0) *wt.clear = 0u;
    const int k8n = g.Kcol >> 3;
    const Index total = (Index)g.N * (hi - lo) * g.Wo * k8n;
    for (Index idx = (Index)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (Index)gridDim.x * blockDim.x) {
        Index q = idx / k8n;
        const int k8 = (int)(idx - q * k8n);
        const Index row = q / g.Wo;
        const int ow = (int)(q - row * g.Wo);
        const int n = (int)(row / (hi - lo)), oh = lo + (int)(row - (Index)n * (hi - lo));
        const uint4 v = gather8<false>(x, g, n, oh, ow, k8);        // reads in-bounds taps only, by construction of the patch
        const long long yo = (((long long)n * g.Ho + oh) * g.Wo + ow) * g.Kcol + k8 * 8;
        if (dbg_in_bounds(dbg, yo, 8, (long long)g.N * g.Ho * g.Wo * g.Kcol)) *reinterpret_cast<uint4 *>(y + yo) = v;
    }
    if (wt.wp) stem_weights(wt, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void stem_weights_kernel(StemWeights wt) { stem_weights(wt, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x); }

// ---------------------------------------------------------------------------------------------
// The transfer step for plans that run on per-layer kernels: rows of the chain input, read straight from page-locked host
// memory by the SMs (around the caches: the host changes it between launches).  A copy-engine copy costs several
// microseconds of stream commands whatever its size, and a band of a small input is a microsecond of transfer; this is
// one launch.  Bound by the host link; four 16-byte loads per thread are in flight.  One 1-D grid of segments per image
// (blockIdx.y); elements before the first and behind the last 16-byte boundary are moved two bytes at a time.
// ---------------------------------------------------------------------------------------------
constexpr int FETCH_THREADS = 128, FETCH_VECS = 4;

__global__ void __launch_bounds__(FETCH_THREADS) fetch_rows_kernel(const uint8_t *__restrict__ src, uint8_t *__restrict__ dst, long long image_bytes,
                                                                   long long first, long long bytes)
{
    grid_release();
    grid_wait();                                                // the input tensor may still be read by the run before this one
    const uint8_t *s0 = src + blockIdx.y * image_bytes + first;
    uint8_t *d0 = dst + blockIdx.y * image_bytes + first;
    const long long mis = (16 - (reinterpret_cast<uintptr_t>(s0) & 15)) & 15, head = mis < bytes ? mis : bytes;
    const long long nvec = (bytes - head) >> 4;
    const uint4 *s4 = reinterpret_cast<const uint4 *>(s0 + head);
    uint4 *d4 = reinterpret_cast<uint4 *>(d0 + head);
    const long long v0 = (long long)blockIdx.x * (FETCH_THREADS * FETCH_VECS) + threadIdx.x;
    uint4 q[FETCH_VECS];
#pragma unroll
    for (int u = 0; u < FETCH_VECS; ++u)
        if (v0 + u * FETCH_THREADS < nvec) q[u] = __ldcv(s4 + v0 + u * FETCH_THREADS);
#pragma unroll
    for (int u = 0; u < FETCH_VECS; ++u)
        if (v0 + u * FETCH_THREADS < nvec) d4[v0 + u * FETCH_THREADS] = q[u];
    if (blockIdx.x == 0 && threadIdx.x < 16) {
        const int h = threadIdx.x;                              // lanes 0..7: the head, 8..15: the tail
        const long long o = h < 8 ? 2 * h : head + (nvec << 4) + 2 * (h - 8);
        if (o < (h < 8 ? head : bytes)) *reinterpret_cast<uint16_t *>(d0 + o) = __ldcv(reinterpret_cast<const uint16_t *>(s0 + o));
    }
}

inline int grid_for(long long work_items, int block, int max_blocks = 148 * 8)
{
    long long b = (work_items + block - 1) / block;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

}  // namespace

cudaError_t launch_maxpool(const PoolArgs &a, int dtype, cudaStream_t s)
{
    const int rows = a.oh_hi - a.oh_lo;
    if (rows <= 0) return cudaSuccess;
    const long long pix = (long long)a.N * rows * a.Wo;
    if (dtype == LOP_BF16) {
        const long long vecs = pix * (a.C / 8);
        const bool aligned = (reinterpret_cast<uintptr_t>(a.x) & 15) == 0 && (reinterpret_cast<uintptr_t>(a.y) & 15) == 0;
        const unsigned blocks = (unsigned)((vecs + 255) / 256);
        const bool wide = a.C % 8 == 0 && aligned && vecs < (1LL << 38);
        if (wide && a.kh == 2 && a.kw == 2) return launch_after(maxpool_bf16x8_kernel<2, 2>, dim3(blocks), 256, 0, s, a);
        if (wide && a.kh == 3 && a.kw == 3) return launch_after(maxpool_bf16x8_kernel<3, 3>, dim3(blocks), 256, 0, s, a);
        if (a.C % 8 == 0) return launch_after(maxpool_kernel<__nv_bfloat16, 8>, dim3(grid_for(pix * (a.C / 8), 256)), 256, 0, s, a);
        return launch_after(maxpool_kernel<__nv_bfloat16, 1>, dim3(grid_for(pix * a.C, 256)), 256, 0, s, a);
    }
    if (a.C % 4 == 0) return launch_after(maxpool_kernel<float, 4>, dim3(grid_for(pix * (a.C / 4), 256)), 256, 0, s, a);
    return launch_after(maxpool_kernel<float, 1>, dim3(grid_for(pix * a.C, 256)), 256, 0, s, a);
}

cudaError_t launch_stem_gather(const void *x, void *y, const GatherGeom &g, int lo, int hi, cudaStream_t s, unsigned *dbg, const StemWeights &wt)
{
    if (hi <= lo) return cudaSuccess;
    if (g.Kcol % 8 != 0) return cudaErrorInvalidValue;
    const long long work = (long long)g.N * (hi - lo) * g.Wo * (g.Kcol / 8);
    const int blocks = grid_for(work, 256);
    const uint16_t *xi = static_cast<const uint16_t *>(x);
    uint16_t *yi = static_cast<uint16_t *>(y);
    // (a 64-bit division is a routine of several dozen instructions, and a thread has four of them)
    if (work < (1LL << 30)) return launch_after(stem_gather_kernel<int>, dim3(blocks), 256, 0, s, xi, yi, g, lo, hi, wt, dbg);
    return launch_after(stem_gather_kernel<long long>, dim3(blocks), 256, 0, s, xi, yi, g, lo, hi, wt, dbg);
}

cudaError_t launch_fetch_rows(const void *src, void *dst, int N, int rows, long long row_bytes, int lo, int hi, cudaStream_t s)
{
    if (hi <= lo) return cudaSuccess;
    long long image = (long long)rows * row_bytes, bytes = (hi - lo) * row_bytes;
    int images = N;
    if (lo == 0 && hi == rows) { bytes *= N; images = 1; }                // whole images are one run
    const long long per_block = 16LL * FETCH_THREADS * FETCH_VECS;
    for (int n = 0; n < images; n += 65535) {
        const dim3 grid((unsigned)((bytes + per_block - 1) / per_block), (unsigned)(images - n < 65535 ? images - n : 65535));
        const cudaError_t e = launch_after(fetch_rows_kernel, grid, FETCH_THREADS, 0, s, static_cast<const uint8_t *>(src) + n * image,
                                           static_cast<uint8_t *>(dst) + n * image, image, lo * row_bytes, bytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_stem_weights(const StemWeights &wt, cudaStream_t s)
{
    stem_weights_kernel<<<grid_for((long long)wt.cout * wt.K, 256), 256, 0, s>>>(wt);
    return cudaGetLastError();
}

}  // namespace lop
