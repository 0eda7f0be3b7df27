// Launch interfaces of the device kernels (host-callable wrappers; each returns a cudaError_t).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace lop {

struct ConvArgs {
    const void *x;          // [N, Hin, Win, Cin]
    const void *w;          // [Cout, kh, kw, Cin]
    const float *scale, *shift;
    const void *res;        // [N, Ho, Wo, Cout] or nullptr
    void *y;                // [N, Ho, Wo, Cout]
    int N, Hin, Win, Cin, Ho, Wo, Cout;
    int kh, kw, sh, sw, ph, pw, dh, dw;
    int act, res_pos;
    int oh_lo, oh_hi;       // rows to compute
    int k_split;            // tensor-core kernels: parts of the channel chunks that are summed on their own, then in order
    // the input in elements: a pixel's channels (those up to Cin read as zeros), from a pixel to the next, from a row to
    // the next.  x_pixel < x_run only for a gathered stem, whose neighbouring pixels share values.
    int x_run, x_pixel;
    long long x_row;
    unsigned *dbg;          // checked execution: the status word that takes bit 0x100 on a violation, else nullptr
};

struct PoolArgs {
    const void *x;
    void *y;
    int N, Hin, Win, C, Ho, Wo;
    int kh, kw, sh, sw, ph, pw, dh, dw;
    int oh_lo, oh_hi;
    unsigned *dbg;          // as in ConvArgs
};

// Consecutive launches on a stream overlap where the second one's start allows it (programmatic dependent launch): a kernel's
// blocks are set up while the one before it drains, and everything that kernel reads or writes comes after grid_wait().
// Every thread of every kernel started by launch_after() calls it, so that a kernel's end still means that all before it
// have ended.  grid_release() lets the next launch begin; it stands behind a tensor-memory allocation, or a block of the next
// kernel could take the columns that a block of this one waits for.  A launch without the attribute, a copy or an event
// orders the stream as ever.  (About 2 us per launch: a DenseNet layer called in a row 18.2 -> 16.2 us,
// a VGG block by per-layer kernels 46.7 -> 39.7.)
#ifdef __CUDACC__
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// A pointer whose loads the compiler must not take to before this place: those of read-only data (__restrict__, __ldg) may move
// across grid_wait(), but not in front of the place that the pointer comes from.
template <typename T>
__device__ __forceinline__ T *from_here(T *p)
{
    asm volatile("" : "+l"(p));
    return p;
}
#endif
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, const A &...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = dim3(block); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Checked execution (LOP_FLAG_DEBUG_BOUNDS): elements [first, first + count) must lie inside a tensor of `limit`
// elements.  Without a status word the test costs one predictable branch.
#ifdef __CUDACC__
__device__ __forceinline__ bool dbg_in_bounds(unsigned *dbg, long long first, long long count, long long limit)
{
    if (!dbg || (first >= 0 && first + count <= limit)) return true;
    atomicOr(dbg, 0x100u);
    return false;
}
#endif

// CUDA-core convolution (fp32 accumulate); dtype: LOP_F32 / LOP_BF16 storage.
cudaError_t launch_conv_simt(const ConvArgs &a, int dtype, cudaStream_t s);
cudaError_t launch_maxpool(const PoolArgs &a, int dtype, cudaStream_t s);
// Depth-wise convolution (w: [C][kh][kw], Cout == Cin), layer normalisation over the channels (scale / shift = gain /
// offset; the window fields are unused) and channel concatenation (x: Cin channels, res: Cout - Cin channels).
// w_taps: the filters as [tap][C] (launch_dw_transpose), or nullptr -- the tiled bf16 kernel needs them.
cudaError_t launch_dwconv(const ConvArgs &a, int dtype, const void *w_taps, cudaStream_t s);
cudaError_t launch_layernorm(const ConvArgs &a, int dtype, cudaStream_t s);
cudaError_t launch_concat(const ConvArgs &a, int dtype, cudaStream_t s);
// depth-wise filters w[C][taps] -> wt[taps][C] (bf16 only), the layout the persistent kernel reads
cudaError_t launch_dw_transpose(const void *w, void *wt, int C, int taps, cudaStream_t s);
// w[cout][kh][kw][C] -> wp[cout][K], zero-padded, in the order of a gathered stem's values: (kw, kh, C) with each column's
// kh*C values padded to col elements, or (kh, kw, C) for col = 0 (bf16 only).  clear: a word to set to zero, if any.
struct StemWeights { const void *w = nullptr; void *wp = nullptr; int cout = 0, kh = 0, kw = 0, C = 0, col = 0, K = 0; unsigned *clear = nullptr; };
cudaError_t launch_stem_weights(const StemWeights &wt, cudaStream_t s);
// rows [lo,hi) of the gathered tensor y[N,Ho,Wo,Kcol] of a thin chain input x[N,H,W,C] (bf16 only).
struct GatherGeom;
// dbg: checked execution's status word (see ConvArgs), or nullptr.  wt: weights to bring along by the same launch, if any.
cudaError_t launch_stem_gather(const void *x, void *y, const GatherGeom &g, int lo, int hi, cudaStream_t s, unsigned *dbg = nullptr,
                               const StemWeights &wt = StemWeights());
// Rows [lo, hi) of each of N images of `rows` rows of row_bytes bytes: src (host memory as the device addresses it) -> dst.
// src and dst agree modulo 16.
cudaError_t launch_fetch_rows(const void *src, void *dst, int N, int rows, long long row_bytes, int lo, int hi, cudaStream_t s);

// cuTensorMapEncodeTiled, looked up through the runtime (no link-time dependency on the driver library); nullptr if absent.
typedef CUresult (*TensorMapEncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                      const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
TensorMapEncodeFn tensor_map_encoder();

// ---- tcgen05 tensor-core convolution ---------------------------------------------------------
struct ConvTcGeom {
    int TW, TR, TN;         // output tile = TN images x TR rows x TW columns, TW*TR*TN == 128 (powers of two)
    int BN;                 // output channels per CTA (multiple of 16, <= 256)
    int BK;                 // input channels per pipeline stage: 64, 32 or 16
    int stages;
};
struct ConvTcMaps {
    CUtensorMap a[4];       // activation maps, one per (row parity, column parity) of a strided window
    CUtensorMap w;          // weights as a [Cout][kh*kw*Cin] matrix
    int a_valid[4];
};
// Chooses the tile geometry for a layer and a number of rows.  fill_sms: a stand-alone launch prefers
// narrower channel tiles when there are too few pixel tiles to occupy every SM.
ConvTcGeom conv_tc_geometry(const ConvArgs &a, int rows, bool fill_sms = true);
// Encodes the tensor maps for a layer (x, w pointers and geometry are baked in).  Host only.
int conv_tc_encode(const ConvArgs &a, const ConvTcGeom &g, ConvTcMaps *maps);
cudaError_t launch_conv_tc(const ConvArgs &a, const ConvTcGeom &g, const ConvTcMaps &maps, unsigned *status,
                           cudaStream_t s);

}  // namespace lop
