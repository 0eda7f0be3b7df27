// Gather of a thin chain input (the tensor "split" an operator interceptor performs, Sec. III-B of the
// paper, combined with the block-wise operator's receptive field, Sec. IV-A), after which the first
// convolution is a pointwise product of `K` gathered values per output pixel with zero-padded weights.
// The gathered tensor has one row per output row, and its columns come in one of two layouts:
//
//   shared columns   one column per input column (padding included), holding that column's kh values of
//                    every channel as C' = kh*C rounded up to 8 elements, zero-padded.  An output pixel's
//                    kw columns are neighbours, so its K = kw*C' values are one contiguous run; the runs
//                    of neighbouring pixels overlap, and the convolution's tensor map steps sw columns per
//                    pixel.  Each input value is written kh times instead of kh*kw times: a 7x7 stride-2
//                    window over 3 channels takes 96 bytes per output pixel, where its patches take 320.
//   patches          one column per output pixel with its kh*kw*C values in (kh, kw, channel) order:
//                    dilated windows, whose columns are no neighbours, and windows so small that the
//                    rounding of C' would make the shared columns the larger tensor.
//
// Either way a gathered column is the patch of a window, kh x 1 in the first layout, so one description
// and one kernel serve both.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace lop {

struct GatherGeom {
    int N, H, W, C;           // chain input
    int Ho, Wo, Kcol;         // gathered tensor: rows, columns, elements of a column
    int kh, kw, sh, sw, ph, pw, dh, dw;       // window of a column
};

// The persistent kernel gathers from input rows staged in shared memory with the padding's zeros around them.  Bytes of
// zeros in front of a staged row (its data starts up to 15 bytes later, where its 16-byte vectors put it), and from a
// row to the next.
__host__ __device__ inline int gather_lead(const GatherGeom &g) { return (g.pw * g.C * 2 + 15) & ~15; }
__host__ __device__ inline int gather_pitch(const GatherGeom &g)
{
    const int end = ((g.Wo - 1) * g.sw - g.pw + (g.kw - 1) * g.dw + 1) * g.C * 2, row = g.W * g.C * 2;
    return (gather_lead(g) + 15 + (end > row ? end : row) + 15) & ~15;
}
// Input rows behind `rows` gathered ones.
__host__ __device__ inline int gather_rows_in(const GatherGeom &g, int rows) { return (rows - 1) * g.sh + (g.kh - 1) * g.dh + 1; }

// Eight consecutive patch elements k8*8 .. k8*8+7 of output pixel (n, oh, ow), as bf16 bit patterns.
// THROUGH_L2: read around L1 (for an input that another engine is still writing while the kernel runs,
// row band by row band; the caller has acquired the band's arrival flag).
template <bool THROUGH_L2>
__device__ __forceinline__ uint4 gather8(const uint16_t *__restrict__ x, const GatherGeom &g, int n, int oh, int ow, int k8)
{
    uint32_t h[8];
    const int klen = g.kh * g.kw * g.C;
    int k = k8 * 8;
    int tap = k / g.C, ci = k - tap * g.C;
    int a = tap / g.kw, b = tap - a * g.kw;
#pragma unroll
    for (int e = 0; e < 8; ++e, ++k) {
        uint32_t v = 0;
        if (k < klen) {
            const int ih = oh * g.sh - g.ph + a * g.dh, iw = ow * g.sw - g.pw + b * g.dw;
            if (ih >= 0 && ih < g.H && iw >= 0 && iw < g.W)
                v = THROUGH_L2 ? __ldcg(x + (((long long)n * g.H + ih) * g.W + iw) * g.C + ci)
                               : __ldg(x + (((long long)n * g.H + ih) * g.W + iw) * g.C + ci);
        }
        h[e] = v;
        if (++ci == g.C) { ci = 0; if (++b == g.kw) { b = 0; ++a; } }
    }
    return make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
}

}  // namespace lop
