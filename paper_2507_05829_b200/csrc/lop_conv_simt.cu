// Convolution on the CUDA cores: the fp32 path, the fall-back for shapes the tensor-core kernel does not take, and the
// library's second on-GPU opinion (LOP_FLAG_FORCE_SIMT).  Implicit GEMM with M = N*rows*Wo output pixels, N = Cout,
// K = kh*kw*Cin (Sec. IV-A of the paper: a block-wise local operator), any kernel / stride / padding / dilation /
// channel count.  Every variant accumulates a value with fused multiply-adds in ascending K, so a pixel's bits depend
// neither on the variant nor on the band it is computed in.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "lop.h"
#include "lop_kernels.cuh"
#include "lop_rowops.cuh"

namespace lop {

namespace {

using rowop::f32x2;
using rowop::fma2;
using rowop::pack2;
using rowop::unpack2;

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void from_f32(float &d, float v) { d = v; }
__device__ __forceinline__ void from_f32(__nv_bfloat16 &d, float v) { d = __float2bfloat16_rn(v); }

// SiLU and GELU stay out of line: a thread finishes up to 64 values in straight-line code, and 64 copies of the library's
// exp and erf made the kernels wait for their own instructions (a 3-channel layer spent 12 of 16 cycles per issue so).
__device__ __noinline__ float activate_smooth(float t, int act)
{
    return act == LOP_ACT_SILU ? t / (1.0f + expf(-t)) : 0.5f * t * (1.0f + erff(t * 0.70710678f));
}
__device__ __forceinline__ float activate(float t, int act)
{
    if (act == LOP_ACT_RELU) return fmaxf(t, 0.0f);
    return act > LOP_ACT_RELU ? activate_smooth(t, act) : t;
}

// Four consecutive elements as fp32 (p is aligned to four elements).
__device__ __forceinline__ void load4(const float *p, float (&v)[4])
{
    const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load4(const __nv_bfloat16 *p, float (&v)[4])
{
    const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p));
    v[0] = __uint_as_float(q.x << 16); v[1] = __uint_as_float(q.x & 0xFFFF0000u);
    v[2] = __uint_as_float(q.y << 16); v[3] = __uint_as_float(q.y & 0xFFFF0000u);
}
__device__ __forceinline__ void store4(float *p, const float (&v)[4]) { *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void store4(__nv_bfloat16 *p, const float (&v)[4])
{
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
}

// Output pixel m of a launch over `rows` rows: image, row, column (32-bit divisions wherever M fits, which is practically
// always: a 64-bit division is a routine of several dozen instructions).
struct Pixel { int n, oh, ow; };
__device__ __forceinline__ Pixel pixel_of(const ConvArgs &p, long long m, long long M, int rows)
{
    Pixel q;
    if (M < (1LL << 31)) {
        const unsigned u = (unsigned)m, r = u / (unsigned)p.Wo, n = r / (unsigned)rows;
        q.ow = (int)(u - r * (unsigned)p.Wo);
        q.oh = p.oh_lo + (int)(r - n * (unsigned)rows);
        q.n = (int)n;
    } else {
        const long long r = m / p.Wo;
        q.ow = (int)(m - r * p.Wo);
        q.n = (int)(r / rows);
        q.oh = p.oh_lo + (int)(r - (long long)q.n * rows);
    }
    return q;
}

template <typename T>
__device__ __forceinline__ float finish(const ConvArgs &p, const T *res, long long o, int co, float acc)
{
    float v = fmaf(p.scale ? p.scale[co] : 1.0f, acc, p.shift ? p.shift[co] : 0.0f);
    if (res && p.res_pos == LOP_RES_PRE_ACT) v += to_f32(res[o]);
    v = activate(v, p.act);
    if (res && p.res_pos == LOP_RES_POST_ACT) v += to_f32(res[o]);
    return v;
}

// Epilogue and store of output channels co .. co + 3 of the pixel whose output starts at element o.
template <typename T>
__device__ __forceinline__ void store_quad(const ConvArgs &p, long long o, int co, int oh, int rows, long long y_elems, const float (&acc)[4])
{
    if (co >= p.Cout) return;
    const int live = min(4, p.Cout - co);
    // the elements inside the tensor, the row inside the rows of this launch (tested as a one-row "tensor")
    if (!dbg_in_bounds(p.dbg, o + co, live, y_elems) || !dbg_in_bounds(p.dbg, oh - p.oh_lo, 1, rows)) return;
    T *__restrict__ y = static_cast<T *>(p.y);
    const T *__restrict__ res = static_cast<const T *>(p.res);
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (e < live) v[e] = finish(p, res, o + co + e, co + e, acc[e]);
    if ((p.Cout & 3) == 0) store4(y + o + co, v);
    else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (e < live) from_f32(y[o + co + e], v[e]);
    }
}

// ---------------------------------------------------------------------------------------------
// Register-tiled kernel: BM pixels x BN output channels per block, TM x TN of them per thread, K in slabs of 16 through
// two shared-memory buffers (one barrier per slab; the next slab's operands are on their way to registers meanwhile).
// Cin is a multiple of 16, so a slab lies inside one filter tap.  Bound by the fp32 multiply-add rate: with 8 x 8 outputs
// a thread reads 16 shared values for 64 multiply-adds (4 x 4 read 8 for 16, which left the shared-memory pipe the
// bound).  Four lanes read a pixel's (an output channel's) 64 bytes of a slab: lanes on 32 pixels instead would cost the
// L1 32 tag look-ups per load, which held the kernel at 40 % of the rate.  The transposed stores are spread over the
// banks by exchanging column groups of eight with the K quad (slab_col).
// ---------------------------------------------------------------------------------------------
constexpr int SM_BK = 16;

__device__ __forceinline__ int slab_col(int k, int col) { return col ^ (((k >> 2) & 3) << 3); }

template <typename T, int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN)) conv_simt_kernel(const __grid_constant__ ConvArgs p)
{
    constexpr int NT = (BM / TM) * (BN / TN);
    constexpr int MG = TM / 4, NG = TN / 4;                   // groups of four consecutive pixels / channels per thread
    constexpr int A4 = BM * 4 / NT, B4 = BN * 4 / NT;         // groups of four K values staged per thread
    static_assert(BM * 4 % NT == 0 && BN * 4 % NT == 0 && TM % 4 == 0 && TN % 4 == 0 && BM % 32 == 0 && BN % 32 == 0, "tile shape");
    __shared__ __align__(16) float As[2][SM_BK][BM];
    __shared__ __align__(16) float Bs[2][SM_BK][BN];

    const T *__restrict__ x = static_cast<const T *>(p.x);
    const T *__restrict__ w = static_cast<const T *>(p.w);
    const int rows = p.oh_hi - p.oh_lo;
    const long long M = (long long)p.N * rows * p.Wo;
    const int K = p.kh * p.kw * p.Cin;
    const long long m0 = (long long)blockIdx.x * BM;
    const int n0 = blockIdx.y * BN;
    const int t = threadIdx.x, kq = t & 3, r0 = t >> 2;        // this thread stages K values 4 kq .. 4 kq + 3 of rows r0 + e * NT / 4
    const long long x_elems = (long long)p.N * p.Hin * p.Win * p.Cin, y_elems = (long long)p.N * p.Ho * p.Wo * p.Cout;

    long long xoff[A4];                                        // element offset of the pixel's first tap (possibly outside the tensor)
    int ih0[A4], iw0[A4];
#pragma unroll
    for (int e = 0; e < A4; ++e) {
        const long long m = m0 + r0 + e * (NT / 4);
        const bool ok = m < M;
        const Pixel q = pixel_of(p, ok ? m : 0, M, rows);
        ih0[e] = q.oh * p.sh - p.ph;
        iw0[e] = q.ow * p.sw - p.pw;
        xoff[e] = (((long long)q.n * p.Hin + ih0[e]) * p.Win + iw0[e]) * p.Cin + 4 * kq;
        if (!ok) ih0[e] = -(1 << 30);                          // no tap of a surplus pixel is inside
    }

    float av[A4][4], bv[B4][4];
    int ta = 0, tb = 0, tc = 0;                                // filter row, column and first channel of the next slab
    auto load_slab = [&](int k0) {
        const long long step = ((long long)ta * p.dh * p.Win + tb * p.dw) * p.Cin + tc;
#pragma unroll
        for (int e = 0; e < A4; ++e) {
            const int ih = ih0[e] + ta * p.dh, iw = iw0[e] + tb * p.dw;
#pragma unroll
            for (int i = 0; i < 4; ++i) av[e][i] = 0.0f;
            if ((unsigned)ih < (unsigned)p.Hin && (unsigned)iw < (unsigned)p.Win && dbg_in_bounds(p.dbg, xoff[e] + step, 4, x_elems))
                load4(x + xoff[e] + step, av[e]);
        }
#pragma unroll
        for (int e = 0; e < B4; ++e) {
            const int co = n0 + r0 + e * (NT / 4);
#pragma unroll
            for (int i = 0; i < 4; ++i) bv[e][i] = 0.0f;
            const long long wo = (long long)co * K + k0 + 4 * kq;
            if (co < p.Cout && dbg_in_bounds(p.dbg, wo, 4, (long long)p.Cout * K)) load4(w + wo, bv[e]);
        }
        tc += SM_BK;
        if (tc == p.Cin) { tc = 0; if (++tb == p.kw) { tb = 0; ++ta; } }
    };
    auto store_slab = [&](int buf) {
#pragma unroll
        for (int e = 0; e < A4; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i) As[buf][4 * kq + i][slab_col(4 * kq, r0 + e * (NT / 4))] = av[e][i];
#pragma unroll
        for (int e = 0; e < B4; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i) Bs[buf][4 * kq + i][slab_col(4 * kq, r0 + e * (NT / 4))] = bv[e][i];
    };

    const int tn = t % (BN / TN), tm = t / (BN / TN);
    f32x2 acc[TM][TN / 2];                                     // pairs of adjacent output channels
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;

    auto load_frag = [&](int buf, int q, float (&ar)[TM], f32x2 (&br)[TN / 2]) {
#pragma unroll
        for (int i = 0; i < MG; ++i) {
            const float4 v = *reinterpret_cast<const float4 *>(&As[buf][q][slab_col(q, tm * 4 + i * (BM / MG))]);
            ar[4 * i] = v.x; ar[4 * i + 1] = v.y; ar[4 * i + 2] = v.z; ar[4 * i + 3] = v.w;
        }
#pragma unroll
        for (int j = 0; j < NG; ++j) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&Bs[buf][q][slab_col(q, tn * 4 + j * (BN / NG))]);
            br[2 * j] = v.x; br[2 * j + 1] = v.y;
        }
    };
    load_slab(0);
    store_slab(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += SM_BK, buf ^= 1) {
        const bool more = k0 + SM_BK < K;
        if (more) load_slab(k0 + SM_BK);
        float ar[2][TM];
        f32x2 br[2][TN / 2];
        load_frag(buf, 0, ar[0], br[0]);
#pragma unroll
        for (int q = 0; q < SM_BK; ++q) {
            if (q + 1 < SM_BK) load_frag(buf, q + 1, ar[(q + 1) & 1], br[(q + 1) & 1]);       // under this step's multiply-adds
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const f32x2 aa = pack2(ar[q & 1][i], ar[q & 1][i]);
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], aa, br[q & 1][j]);
            }
        }
        if (more) store_slab(buf ^ 1);                      // the other buffer: its readers passed the previous barrier
        __syncthreads();
    }

#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const long long m = m0 + tm * 4 + (i / 4) * (BM / MG) + (i & 3);
        if (m >= M) continue;
        const Pixel q = pixel_of(p, m, M, rows);
        const long long o = (((long long)q.n * p.Ho + q.oh) * p.Wo + q.ow) * p.Cout;
#pragma unroll
        for (int j = 0; j < NG; ++j) {
            float v[4];
            unpack2(acc[i][2 * j], v[0], v[1]);
            unpack2(acc[i][2 * j + 1], v[2], v[3]);
            store_quad<T>(p, o, n0 + tn * 4 + j * (BN / NG), q.oh, rows, y_elems, v);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Small layers: 16 pixels x 16 output channels per block of 64 threads.  With a few blocks per SM at most, latency is
// all there is, so both operands' whole K extent goes to shared memory in one go -- every load of the block in flight at
// once, one barrier -- and a thread then walks its pixel's K for four output channels.  fp32 with Cin a multiple of
// four.  Row pitch: an odd multiple of four floats, so that the eight pixels and the four channel rows a warp reads fall
// into different banks.  Divisions and other index arithmetic stand before the wait for the launch in front, every read
// behind it (with the divisions behind it, too, a 16-channel 3x3 layer of 32x32 called in a row takes 6.1 us, 4.6 so).
// ---------------------------------------------------------------------------------------------
constexpr int SMALL_PX = 16, SMALL_CO = 16, SMALL_THREADS = 64;

__host__ __device__ inline int small_pitch(int K) { return (K & 4) ? K : K + 4; }

__global__ void __launch_bounds__(SMALL_THREADS) conv_simt_small_kernel(const __grid_constant__ ConvArgs p)
{
    extern __shared__ __align__(16) float small_sm[];
    const int rows = p.oh_hi - p.oh_lo;
    const long long M = (long long)p.N * rows * p.Wo;
    const int K = p.kh * p.kw * p.Cin, pitch = small_pitch(K), c4n = p.Cin >> 2, taps = p.kh * p.kw;
    const long long m0 = (long long)blockIdx.x * SMALL_PX;
    const int n0 = blockIdx.y * SMALL_CO;
    const long long x_elems = (long long)p.N * p.Hin * p.Win * p.Cin, y_elems = (long long)p.N * p.Ho * p.Wo * p.Cout;
    grid_release();
    float *As = small_sm, *Bs = small_sm + SMALL_PX * pitch;
    const float *__restrict__ x = static_cast<const float *>(p.x);
    const float *__restrict__ w = static_cast<const float *>(p.w);
    auto copy16 = [](float *dst, const float *src, bool live) {
        const unsigned n = live ? 16u : 0u;                    // 0: the sixteen bytes are zero-filled, nothing is read
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(n) : "memory");
    };
    // four threads per pixel (each every fourth filter tap) and per output channel (each every fourth group of four K values)
    const int part = threadIdx.x & 3, r = threadIdx.x >> 2;
    const bool ok = m0 + r < M, has_row = n0 + r < p.Cout;
    const Pixel at = pixel_of(p, ok ? m0 + r : 0, M, rows);
    const int ih0 = at.oh * p.sh - p.ph, iw0 = at.ow * p.sw - p.pw;
    const long long x0 = (((long long)at.n * p.Hin + ih0) * p.Win + iw0) * p.Cin, w0 = (long long)(n0 + r) * K;
    int a = part / p.kw, b = part - a * p.kw;
    const int a4 = 4 / p.kw, b4 = 4 - a4 * p.kw;               // four taps further on
    grid_wait();                                               // before the weights too: the launch before this one may have written them
    for (int k = 4 * part; k < K; k += 16) {                   // K contiguous floats per output channel
        const bool live = has_row && dbg_in_bounds(p.dbg, w0 + k, 4, (long long)p.Cout * K);
        copy16(Bs + r * pitch + k, live ? w + w0 + k : w, live);
    }
    for (int tap = part; tap < taps; tap += 4) {
        const int ih = ih0 + a * p.dh, iw = iw0 + b * p.dw;
        const long long xo = x0 + ((long long)a * p.dh * p.Win + b * p.dw) * p.Cin;
        const bool live = ok && ih >= 0 && ih < p.Hin && iw >= 0 && iw < p.Win && dbg_in_bounds(p.dbg, xo, p.Cin, x_elems);
        for (int c = 0; c < c4n; ++c) copy16(As + r * pitch + tap * p.Cin + 4 * c, live ? x + xo + 4 * c : x, live);
        a += a4; b += b4;
        if (b >= p.kw) { b -= p.kw; ++a; }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    const float *xa = As + r * pitch;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        const float4 xv = *reinterpret_cast<const float4 *>(xa + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 wv = *reinterpret_cast<const float4 *>(Bs + (part + 4 * j) * pitch + k);
            acc[j] = fmaf(xv.w, wv.w, fmaf(xv.z, wv.z, fmaf(xv.y, wv.y, fmaf(xv.x, wv.x, acc[j]))));
        }
    }
    if (!ok) return;
    const long long o = (((long long)at.n * p.Ho + at.oh) * p.Wo + at.ow) * p.Cout;
    const float *__restrict__ res = from_here(static_cast<const float *>(p.res));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int co = n0 + part + 4 * j;
        if (co >= p.Cout || !dbg_in_bounds(p.dbg, o + co, 1, y_elems) || !dbg_in_bounds(p.dbg, at.oh - p.oh_lo, 1, rows)) continue;
        static_cast<float *>(p.y)[o + co] = finish(p, res, o + co, co, acc[j]);
    }
}

// ---------------------------------------------------------------------------------------------
// Any channel count, for short K (a thin image: three channels, a few dozen products): 128 pixels x 64 output channels per
// block of 256 threads, sixteen channels of two pixels per thread.  The block's filters go to shared memory as
// [k][channel], THIN_KC values of K at a time; the pixels' inputs are read where they are (four lanes share an address).
// Bound by the output's stores: K = 27 on 181 x 203 pixels writes 9.4 MB.  Also the general fall-back (channels not a
// multiple of 16, weights not aligned to a vector), where it is bound by its scalar loads.
// ---------------------------------------------------------------------------------------------
constexpr int THIN_PX = 128, THIN_CO = 64, THIN_THREADS = 256, THIN_KC = 64;

template <typename T>
__global__ void __launch_bounds__(THIN_THREADS) conv_simt_thin_kernel(const __grid_constant__ ConvArgs p)
{
    __shared__ __align__(16) float Ws[THIN_KC][THIN_CO + 4];
    const T *__restrict__ x = static_cast<const T *>(p.x);
    const T *__restrict__ w = static_cast<const T *>(p.w);
    const int rows = p.oh_hi - p.oh_lo;
    const long long M = (long long)p.N * rows * p.Wo;
    const int K = p.kh * p.kw * p.Cin, n0 = blockIdx.y * THIN_CO;
    const long long x_elems = (long long)p.N * p.Hin * p.Win * p.Cin, y_elems = (long long)p.N * p.Ho * p.Wo * p.Cout;
    const int cq = threadIdx.x & 3;                            // channels 16 j + 4 cq .. + 3, j = 0..3
    long long xo0[2], o[2], xo[2];
    int ih0[2], iw0[2], oh[2];
    bool in[2], live_px[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const long long m = (long long)blockIdx.x * THIN_PX + e * (THIN_PX / 2) + (threadIdx.x >> 2);
        live_px[e] = m < M;
        const Pixel q = pixel_of(p, live_px[e] ? m : 0, M, rows);
        ih0[e] = q.oh * p.sh - p.ph;
        iw0[e] = q.ow * p.sw - p.pw;
        oh[e] = q.oh;
        xo0[e] = xo[e] = (((long long)q.n * p.Hin + ih0[e]) * p.Win + iw0[e]) * p.Cin;
        o[e] = (((long long)q.n * p.Ho + q.oh) * p.Wo + q.ow) * p.Cout;
        if (!live_px[e]) ih0[e] = -(1 << 30);                  // no tap of a surplus pixel is inside
        in[e] = (unsigned)ih0[e] < (unsigned)p.Hin && (unsigned)iw0[e] < (unsigned)p.Win;
    }
    f32x2 acc[2][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[0][j] = acc[1][j] = 0ull;
    int a = 0, b = 0, ci = 0;                                  // filter position and channel of k
    for (int k0 = 0; k0 < K; k0 += THIN_KC) {
        const int kn = min(THIN_KC, K - k0);
        if (k0 > 0) __syncthreads();
        {
            const int r = threadIdx.x >> 2, co = n0 + r;
            for (int k = threadIdx.x & 3; k < kn; k += 4) {
                const long long wo = (long long)co * K + k0 + k;
                Ws[k][r] = (co < p.Cout && dbg_in_bounds(p.dbg, wo, 1, (long long)p.Cout * K)) ? to_f32(w[wo]) : 0.0f;
            }
        }
        __syncthreads();
#pragma unroll 3
        for (int k = 0; k < kn; ++k) {
            float xv[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                xv[e] = 0.0f;
                if (in[e] && dbg_in_bounds(p.dbg, xo[e], 1, x_elems)) xv[e] = to_f32(x[xo[e]]);
                ++xo[e];
            }
            if (++ci == p.Cin) {
                ci = 0;
                if (++b == p.kw) { b = 0; ++a; }
                const long long step = ((long long)a * p.dh * p.Win + b * p.dw) * p.Cin;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int ih = ih0[e] + a * p.dh, iw = iw0[e] + b * p.dw;
                    xo[e] = xo0[e] + step;
                    in[e] = (unsigned)ih < (unsigned)p.Hin && (unsigned)iw < (unsigned)p.Win;
                }
            }
            const f32x2 x0 = pack2(xv[0], xv[0]), x1 = pack2(xv[1], xv[1]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const ulonglong2 wv = *reinterpret_cast<const ulonglong2 *>(&Ws[k][16 * j + 4 * cq]);
                fma2(acc[0][2 * j], x0, wv.x);
                fma2(acc[0][2 * j + 1], x0, wv.y);
                fma2(acc[1][2 * j], x1, wv.x);
                fma2(acc[1][2 * j + 1], x1, wv.y);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
        if (live_px[e]) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float v[4];
                unpack2(acc[e][2 * j], v[0], v[1]);
                unpack2(acc[e][2 * j + 1], v[2], v[3]);
                store_quad<T>(p, o[e], n0 + 16 * j + 4 * cq, oh[e], rows, y_elems, v);
            }
        }
}

template <typename T, int BM, int BN, int TM, int TN>
cudaError_t launch_tiles(const ConvArgs &a, long long M, cudaStream_t s)
{
    const dim3 grid((unsigned)((M + BM - 1) / BM), (unsigned)((a.Cout + BN - 1) / BN));
    constexpr int NT = (BM / TM) * (BN / TN);
    // (not begun before the launch in front has ended: its blocks, a few per SM, would go to the SMs that are free first, three
    // on some and one on others -- a VGG block of 181x203 pixels 94 us so, 125 begun early)
    conv_simt_kernel<T, BM, BN, TM, TN><<<grid, NT, 0, s>>>(a);
    return cudaGetLastError();
}

// The tile with the least work on the busiest SM: tiles per SM (rounded up) times the tile's multiply-adds, weighted by
// how far the tile's inner loop stays below the multiply-add rate.
template <typename T>
cudaError_t launch_typed(const ConvArgs &a, long long M, cudaStream_t s)
{
    // (the caller's weights need not be aligned beyond their element)
    const bool aligned = ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.w)) & (4 * sizeof(T) - 1)) == 0;
    if (a.Cin % SM_BK != 0 || !aligned) {
        const dim3 grid((unsigned)((M + THIN_PX - 1) / THIN_PX), (unsigned)((a.Cout + THIN_CO - 1) / THIN_CO));
        conv_simt_thin_kernel<T><<<grid, THIN_THREADS, 0, s>>>(a);
        return cudaGetLastError();
    }
    auto cost = [&](int bm, int bn, double weight) {
        const double tiles = (double)((M + bm - 1) / bm) * ((a.Cout + bn - 1) / bn);
        return (double)(long long)((tiles + 147.0) / 148.0) * bm * bn * weight;
    };
    const double big = cost(128, 64, 1.0), mid = cost(64, 64, 1.15), little = cost(64, 32, 1.4);
    if (big <= mid && big <= little) return launch_tiles<T, 128, 64, 8, 8>(a, M, s);
    if (mid <= little) return launch_tiles<T, 64, 64, 4, 8>(a, M, s);
    return launch_tiles<T, 64, 32, 4, 4>(a, M, s);
}

}  // namespace

cudaError_t launch_conv_simt(const ConvArgs &a, int dtype, cudaStream_t s)
{
    const int rows = a.oh_hi - a.oh_lo;
    if (rows <= 0) return cudaSuccess;
    const long long M = (long long)a.N * rows * a.Wo;
    const int K = a.kh * a.kw * a.Cin;
    if (dtype == LOP_BF16) return launch_typed<__nv_bfloat16>(a, M, s);
    // Layers the small blocks serve, if their operands fit (K up to about 380): those with at most four such blocks per
    // SM, those too narrow for the tiles (at most 16 output channels) and those the tiles cannot read (Cin a multiple of
    // four but not of 16; the alternative there reads element by element).
    const long long small_blocks = ((M + SMALL_PX - 1) / SMALL_PX) * ((a.Cout + SMALL_CO - 1) / SMALL_CO);
    const size_t small_bytes = (size_t)(SMALL_PX + SMALL_CO) * small_pitch(K) * sizeof(float);
    const bool aligned = ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.w)) & 15) == 0;
    if (a.Cin % 4 == 0 && aligned && small_bytes <= 48u * 1024u && (small_blocks <= 4 * 148 || a.Cout <= SMALL_CO || a.Cin % SM_BK != 0)) {
        const dim3 grid((unsigned)((M + SMALL_PX - 1) / SMALL_PX), (unsigned)((a.Cout + SMALL_CO - 1) / SMALL_CO));
        return launch_after(conv_simt_small_kernel, grid, SMALL_THREADS, small_bytes, s, a);
    }
    return launch_typed<float>(a, M, s);
}

}  // namespace lop
