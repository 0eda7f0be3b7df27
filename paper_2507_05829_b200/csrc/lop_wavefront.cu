// Persistent wavefront kernel (see lop_wavefront.cuh for the execution model).
//
// CTA layout (three special warps + WF_WORKER_WARPS worker warps, one CTA per SM):
//   warp 0      all lanes poll the item's producer row groups in parallel (the dependency list of the
//               next item is prefetched while this one runs); lane 0 then streams the item's activation
//               and weight boxes by TMA into a shared-memory ring of entries that lives across items
//   warp 1      one lane issues tcgen05.mma into one of two fp32 accumulators in tensor memory, so the
//               next item's main loop overlaps this item's epilogue
//   warp 2      one lane issues the bulk stores of finished output units and publishes finished items: it fences and does
//               the release increment of the item's row-group counter, so that this latency is off the workers' path
//   workers     epilogue of convolution items: TMEM -> scale/shift/residual/activation -> bf16 rows in an output
//               unit in shared memory (results in host memory and folded poolings they copy out themselves); and
//               the whole of pooling, patch-gather, depth-wise convolution, layer-normalisation and concatenation items.
//               Many of them because straight-line per-element code needs several warps per scheduler to
//               hide its own latency; the four warps that share a TMEM lane group split a tile's columns.
//
// Convolution as implicit GEMM: accumulator row m is an *anchor*, a position in a flat list of pixels
// with a row pitch of P pixels.  In slab mode the activation box holds the tile's rows plus the halo of
// the filter, P pixels wide; filter tap (a, b) reads the same box starting (a*dh*P + b*dw) pixels later,
// so one TMA box per 64-channel chunk serves all taps (the shared-memory matrix descriptor simply starts
// later: the swizzle is a function of the address).  Anchors in the last (kw-1)*dw columns of a
// pitch would wrap into the next row; they are computed and dropped.  K is walked as (channel chunk, kh,
// kw, 16-channel step) whatever the tile, so a pixel's bits do not depend on who computes it.  (A gathered stem is a
// pointwise layer here: its K is the order of the gathered values, lop_gather.cuh.)  Where the plan sums K in parts, a
// tile's parts are items of neighbouring CTAs of a cluster, which exchange slices of their partial sums (split_item).
//
// Deadlock freedom: items are numbered in a topological order, every CTA is resident and takes its
// items in increasing order, so the lowest unfinished item never waits on an unstarted one (the parts of a split tile
// wait for one another, and for nothing that has a higher number than the first of them).  All waits are bounded all the
// same; one that runs out raises the status word and the abort flag.
#include <atomic>

#include <cuda_bf16.h>

#include "lop_gather.cuh"
#include "lop_kernels.cuh"
#include "lop_ptx.cuh"
#include "lop_rowops.cuh"
#include "lop_wavefront.cuh"

namespace lop {

namespace {

using namespace ptx;

constexpr int EPI_THREADS = 32 * WF_WORKER_WARPS;
#ifndef LOP_PREFETCH
#define LOP_PREFETCH 32
#endif
constexpr int PREFETCH_BOXES = LOP_PREFETCH;                // weight boxes of a tile asked for ahead of its dependencies
static_assert(8 * (2 * WF_ENTRIES + 4 + 2 * WF_PUBQ + 4 + 3 * WF_UNITS + 2 + WF_GROUPS + 4) + 128 + 2048 + 8 * (128 + 32) <= WF_FIXED_SMEM, "barriers and tables");
constexpr int COL_GROUPS = WF_WORKER_WARPS / 4;            // worker warps sharing a TMEM lane group split the columns

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// An increment behind everything this thread has done or seen done.
__device__ __forceinline__ void add_release(unsigned *p)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

#ifdef LOP_WF_TRACE
// Developer build only: per-item time stamps (global timer, ns) of the three roles.
constexpr int TRACE_ITEMS = 1 << 15;
constexpr int TRACE_FETCH0 = 1 << 14;                       // fetch entry j is stamped at row TRACE_FETCH0 + j
__device__ unsigned long long g_wf_trace[TRACE_ITEMS * 16];
__device__ __forceinline__ void tr(int item, int slot)
{
    if (item < TRACE_ITEMS) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        g_wf_trace[item * 16 + slot] = t;
    }
}
__device__ __forceinline__ void trv(int item, int slot, unsigned long long v)
{
    if (item < TRACE_ITEMS) g_wf_trace[item * 16 + slot] = v;
}
#else
#define tr(item, slot) ((void)0)
#define trv(item, slot, v) ((void)0)
#endif

// ---- item records -------------------------------------------------------------------------------
__device__ __forceinline__ int rec_stage(const int4 &r) { return r.x & 0xFFFF; }
__device__ __forceinline__ int rec_cout(const int4 &r) { return (int)((unsigned)r.x >> 16); }
__device__ __forceinline__ int rec_tw(const int4 &r) { return r.y & 0xFFFF; }
__device__ __forceinline__ int rec_tn(const int4 &r) { return (int)((unsigned)r.y >> 16); }
__device__ __forceinline__ int rec_tr(const int4 &r) { return r.z & 0xFFFFF; }
__device__ __forceinline__ int rec_ndep(const int4 &r) { return (int)((unsigned)r.z >> 20); }
__device__ __forceinline__ int rec_dep0(const int4 &r) { return r.w; }

// Bounded wait of a whole warp for an item's dependencies: lane j polls entry j of the list (its first
// 32 entries were prefetched into `mine`).  Counters only grow (compare modulo 2^32).  The result is
// uniform across the warp.  idle() runs once if the first look finds a producer unfinished: there is time then.  (No
// sleep between two looks: a ResNet-50 of batch 8 442 us with 32 ns, 439 without.  A wait of more than 1024 looks, a
// third of a millisecond, sleeps 2 us every 64, which takes a look to 256 ns on average, as 32 ns after each do -- 210 without any:
// the limit is a number of looks and stands for a time.  Slept from the first 64 on, a ResNet-18 streamed one image takes 131.4 us, 126.5 so.)
template <typename Idle>
__device__ __forceinline__ bool wait_deps_warp(const WfParams &P, int first, int count, int2 mine, unsigned run, int lane, Idle idle)
{
    bool idled = false;
    for (int j0 = 0; j0 < count; j0 += 32) {
        const bool have = j0 + lane < count;
        int2 d = mine;
        if (j0 > 0 && have) d = __ldg(&P.deps[first + j0 + lane]);
        // d.y > 0: a row-group counter that grows by d.y per run; d.y < 0: an arrival flag set to >= -d.y
        const unsigned target = !have ? 0u : (d.y > 0 ? run * (unsigned)d.y : (unsigned)(-d.y));
        const unsigned *ctr = P.counters + (have ? d.x : 0);
        bool done = !have;
        for (uint32_t i = 0;; ++i) {
            if (!done) done = (int)(ld_acquire(ctr) - target) >= 0;
            if (__all_sync(0xffffffffu, done)) break;
            if (!idled) { idled = true; idle(); }
            if (i >= P.spin_limit) return false;
            if ((i & 63u) == 63u) {
                if (__any_sync(0xffffffffu, ld_relaxed(P.counters + 2) != 0u)) return false;
                if (i > 1024u) __nanosleep(2048);
            }
        }
    }
    __syncwarp();            // every lane's acquire now orders the whole warp's later reads
    return true;
}

// What waits at a barrier may wait for the loader, which waits for rows: the limits below, five to eight seconds, are above
// that wait's default of 1.5, and a role that gives up ends the others' waits by the abort flag.
constexpr uint32_t BARRIER_TRIES = 8u * WAIT_LIMIT, BARRIER_TESTS = 64u * WAIT_LIMIT;

// Bounded mbarrier wait that also gives up when the CTA's abort flag is raised.
__device__ __forceinline__ bool mbar_wait_abortable(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag)
{
    for (uint32_t i = 0; i < BARRIER_TRIES; ++i) {
        uint32_t done;
        asm volatile(
            "{\n"
            ".reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((i & 255u) == 255u && *abort_flag) return false;
    }
    return false;
}

// The same by looking again and again: for the one thread that issues the MMAs, which a wait that suspends it costs the time to
// wake up (a ResNet-50 of batch 32 795 us suspended, 790 so).
__device__ __forceinline__ bool mbar_spin_abortable(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag)
{
    for (uint32_t i = 0; i < BARRIER_TESTS; ++i) {
        uint32_t done;
        asm volatile(
            "{\n"
            ".reg .pred p;\n"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((i & 255u) == 255u && *abort_flag) return false;
    }
    return false;
}

// The 16-channel MMA steps of one (tap, channel chunk): descriptors differ only in their start-address field.
// desc_hi: upper word of the operand descriptors (stride between 8-row groups, version, swizzle mode).
// la, lb: low words of the two descriptors (address >> 4 in the start field, leading-offset field 1).
template <int KSTEPS>
__device__ __forceinline__ void mma_ksteps_f(uint32_t acc, uint32_t la, uint32_t lb, uint32_t desc_hi, uint32_t idesc, uint32_t &accumulate)
{
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk) {
        const uint64_t ad = ((uint64_t)desc_hi << 32) | (uint64_t)(la + 2u * kk);
        const uint64_t bd = ((uint64_t)desc_hi << 32) | (uint64_t)(lb + 2u * kk);
        umma_bf16(acc, ad, bd, idesc, accumulate);
        accumulate = 1u;
    }
}
__device__ __forceinline__ uint32_t desc_lo(uint32_t smem_addr) { return ((smem_addr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ void mma_tap_f(uint32_t acc, uint32_t la, uint32_t lb, uint32_t desc_hi, uint32_t idesc, int ksteps, uint32_t &accumulate)
{
    if (ksteps == 4) mma_ksteps_f<4>(acc, la, lb, desc_hi, idesc, accumulate);
    else if (ksteps == 2) mma_ksteps_f<2>(acc, la, lb, desc_hi, idesc, accumulate);
    else mma_ksteps_f<1>(acc, la, lb, desc_hi, idesc, accumulate);
}
// One weight box of three taps of a 3x3 filter row over a 64-channel chunk: twelve MMAs whose descriptors differ
// from the first one by compile-time constants.  One thread issues every MMA of the CTA and each instruction it
// executes in between costs as much as a quarter of an N = 64 MMA, so the common case gets straight-line code.
// la, lb: start-address fields (address >> 4) of the slab row this filter row starts at and of the weight box;
// tap16: bytes of one tap's weights >> 4.
__device__ __forceinline__ void mma_row3x64(uint32_t acc, uint32_t la, uint32_t lb, uint32_t tap16, uint32_t desc_hi, uint32_t idesc,
                                            uint32_t &accumulate)
{
    const uint64_t hi = (uint64_t)desc_hi << 32;
#pragma unroll
    for (int tb = 0; tb < 3; ++tb)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            umma_bf16(acc, hi | (uint64_t)(la + 8u * tb + 2u * kk), hi | (uint64_t)(lb + tap16 * tb + 2u * kk), idesc, accumulate);
            accumulate = 1u;
        }
}

__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory"); }

template <typename T>
__device__ __forceinline__ T ldg_ptr(const void *const *p)
{
    return reinterpret_cast<T>(__ldg(reinterpret_cast<const unsigned long long *>(p)));
}

// ---- the memory-bound operators, run by all worker threads (tid = 0 .. EPI_THREADS-1) on one item.  Kept out of line:
// they are rare and long, and inlined they cost the convolution roles registers.
// Depth-wise convolution item: 2^tr_log output rows x tw_valid columns x BN channels of image n (see
// rowop::dwconv_tile); the window is read through L2 -- other SMs produced it during this launch.
__device__ __noinline__ void dwconv_item(const WfStage *sp, int n, int tile_r, int tile_w, int tile_c, int tid, uint8_t *stg)
{
    rowop::DwGeom g;
    g.Hin = __ldg(&sp->Hin); g.Win = __ldg(&sp->Win); g.C = __ldg(&sp->Cin); g.Ho = __ldg(&sp->Ho); g.Wo = __ldg(&sp->Wo);
    g.kh = __ldg(&sp->kh); g.kw = __ldg(&sp->kw); g.sh = __ldg(&sp->sh); g.sw = __ldg(&sp->sw);
    g.ph = __ldg(&sp->ph); g.pw = __ldg(&sp->pw); g.dh = __ldg(&sp->dh); g.dw = __ldg(&sp->dw);
    g.act = __ldg(&sp->act);
    g.t.R = 1 << __ldg(&sp->tr_log); g.t.tw = __ldg(&sp->tw_valid); g.t.cc = __ldg(&sp->BN);
    g.x = ldg_ptr<const uint16_t *>(&sp->x);
    g.res = ldg_ptr<const uint16_t *>(&sp->res);
    g.res_pos = g.res ? __ldg(&sp->res_pos) : LOP_RES_NONE;
    g.w_taps = ldg_ptr<const uint16_t *>(&sp->w_taps);
    g.scale = ldg_ptr<const float *>(reinterpret_cast<const void *const *>(&sp->scale));
    g.shift = ldg_ptr<const float *>(reinterpret_cast<const void *const *>(&sp->shift));
    g.y = ldg_ptr<uint16_t *>(reinterpret_cast<const void *const *>(&sp->y));
    g.dbg = nullptr; g.N = __ldg(&sp->N);                     // checked execution runs the stand-alone kernels
    const int oh0 = __ldg(&sp->oh_lo) + tile_r * g.t.R, ow0 = tile_w * g.t.tw;
    rowop::dwconv_tile<true, 1, EPI_THREADS>(g, n, oh0, min(g.t.R, __ldg(&sp->oh_hi) - oh0), ow0, min(g.t.tw, g.Wo - ow0), tile_c * g.t.cc,
                                             reinterpret_cast<float *>(stg), tid);
}

// Layer normalisation over the channels of the pixels of output row oh of image n (rowop::ln_pixels: a group of
// lanes per pixel, four vectors in flight per lane).
template <int VPL>
__device__ __forceinline__ void layernorm_row(const uint16_t *x, uint16_t *y, const float *gain, const float *offset, int C, int Wo, long long row0,
                                              int tid)
{
    constexpr int PPG = 4 / VPL;
    const int lanes_log = rowop::ln_lanes_log(C >> 3);
    const int sub = tid & ((1 << lanes_log) - 1), slot = tid >> lanes_log, per_pass = (EPI_THREADS >> lanes_log) * PPG;
    for (int w0 = 0; w0 < Wo; w0 += per_pass) {               // the same trip count for every lane
        long long o[PPG];
        bool live[PPG];
#pragma unroll
        for (int q = 0; q < PPG; ++q) {
            const int ow = w0 + slot * PPG + q;
            live[q] = ow < Wo;
            o[q] = (row0 + ow) * C;
        }
        rowop::ln_pixels<true, VPL, PPG>(x, y, C, lanes_log, sub, o, live, gain, offset);
    }
}
__device__ __noinline__ void layernorm_item(const WfStage *sp, int n, int oh, int tid)
{
    const int C = __ldg(&sp->Cin), Ho = __ldg(&sp->Ho), Wo = __ldg(&sp->Wo);
    const uint16_t *x = ldg_ptr<const uint16_t *>(&sp->x);
    uint16_t *y = ldg_ptr<uint16_t *>(reinterpret_cast<const void *const *>(&sp->y));
    const float *gain = ldg_ptr<const float *>(reinterpret_cast<const void *const *>(&sp->scale));
    const float *offset = ldg_ptr<const float *>(reinterpret_cast<const void *const *>(&sp->shift));
    const long long row0 = ((long long)n * Ho + oh) * Wo;
    const int vpl = rowop::ln_vpl(C >> 3);
    if (vpl == 1) layernorm_row<1>(x, y, gain, offset, C, Wo, row0, tid);
    else if (vpl == 2) layernorm_row<2>(x, y, gain, offset, C, Wo, row0, tid);
    else layernorm_row<4>(x, y, gain, offset, C, Wo, row0, tid);
}

// Channel concatenation of output row oh of image n: the main input's Cin channels, then the second input's Cout - Cin.
__device__ __noinline__ void concat_item(const WfStage *sp, int n, int oh, int tid)
{
    const int Cin = __ldg(&sp->Cin), Cout = __ldg(&sp->Cout), Ho = __ldg(&sp->Ho), Wo = __ldg(&sp->Wo);
    const int va = Cin >> 3, vo = Cout >> 3;
    const long long row = ((long long)n * Ho + oh) * Wo;
    const uint4 *xa = reinterpret_cast<const uint4 *>(ldg_ptr<const __nv_bfloat16 *>(&sp->x) + row * Cin);
    const uint4 *xb = reinterpret_cast<const uint4 *>(ldg_ptr<const __nv_bfloat16 *>(&sp->res) + row * (Cout - Cin));
    uint4 *y = reinterpret_cast<uint4 *>(ldg_ptr<__nv_bfloat16 *>(reinterpret_cast<const void *const *>(&sp->y)) + row * Cout);
    for (int idx = tid; idx < Wo * vo; idx += EPI_THREADS) {
        const int ow = idx / vo, v = idx - ow * vo;
        y[idx] = v < va ? __ldcg(xa + (long long)ow * va + v) : __ldcg(xb + (long long)ow * (vo - va) + (v - va));
    }
}

// len bytes (a multiple of 2) from host memory the device can address to device memory, by the 32 lanes of a warp.
// Host lines are read around the caches (they change between launches without the device knowing); eight 16-byte
// loads per lane are in flight to cover the host link's latency.  src and dst agree modulo 16.
#ifndef LOP_FETCH_DEPTH
#define LOP_FETCH_DEPTH 8
#endif
constexpr int FETCH_DEPTH = LOP_FETCH_DEPTH;
__device__ __forceinline__ void fetch_bytes(const uint8_t *src, uint8_t *dst, int len, int lane)
{
    int head = (16 - (int)(reinterpret_cast<uintptr_t>(src) & 15)) & 15;
    if (head > len) head = len;
    const int nvec = (len - head) >> 4, tail = head + (nvec << 4);
    // elements before the first and behind the last 16-byte boundary: lanes 0..7 and 8..15, on their way with the vectors
    const int edge = lane < 8 ? 2 * lane : tail + 2 * (lane - 8);
    const bool has_edge = lane < 16 && edge < (lane < 8 ? head : len);
    uint16_t edge_value = 0;
    if (has_edge) edge_value = __ldcv(reinterpret_cast<const uint16_t *>(src + edge));
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src + head);
    uint4 *d4 = reinterpret_cast<uint4 *>(dst + head);
    // A warp's loads start at 128-byte lines of the source.  (Rows of 4656 bytes, read from where they start, came at 11 GB/s
    // for the lines that two loads shared, from line starts at twice that and more: a 674x777 stack streamed 457 -> 278 us.)
    const int skew = (int)(reinterpret_cast<uintptr_t>(s4) & 127) >> 4;
    for (int v0 = -skew; v0 < nvec; v0 += FETCH_DEPTH * 32) {
        uint4 q[FETCH_DEPTH];
#pragma unroll
        for (int u = 0; u < FETCH_DEPTH; ++u) {
            const int v = v0 + u * 32 + lane;
            if (v >= 0 && v < nvec) q[u] = __ldcv(s4 + v);
        }
#pragma unroll
        for (int u = 0; u < FETCH_DEPTH; ++u) {
            const int v = v0 + u * 32 + lane;
            if (v >= 0 && v < nvec) d4[v] = q[u];
        }
    }
    if (has_edge) *reinterpret_cast<uint16_t *>(dst + edge) = edge_value;
}

// The functions below are kept out of line: inlined, they cost the epilogue's path registers and instruction cache (a
// ResNet-50 of batch 32: 998 us with pooling and gather inside the kernel's body, 974 outside; a ConvNeXt block 47 -> 45).

// 16-byte chunk j of staged row `row` of an output unit (the swizzle of the unit's tensor maps).
__device__ __forceinline__ uint4 unit_chunk(const uint8_t *unit, int row, int j, int sub_log)
{
    const int sw = sub_log == 6 ? row & 7 : (sub_log == 5 ? (row >> 1) & 3 : (row >> 2) & 1);
    return *reinterpret_cast<const uint4 *>(unit + (row << (sub_log + 1)) + ((j ^ sw) << 4));
}

// Staged rows of a unit -> global: consecutive threads write consecutive 16 bytes of a pixel's channels.
__device__ __noinline__ void copy_unit(const uint8_t *unit, const long long *row_pix, uint4 *y, int rows_n, int sub_log, int tid)
{
    const int cpr_log = sub_log - 3;                           // 16-byte chunks per staged row
#pragma unroll 4
    for (int idx = tid; idx < rows_n << cpr_log; idx += EPI_THREADS) {
        const int row = idx >> cpr_log, j = idx - (row << cpr_log);
        const long long rp = row_pix[row];
        if (rp >= 0) y[(rp >> 3) + j] = unit_chunk(unit, row, j, sub_log);
    }
}

// 2x2 windows of staged rows -> their maxima (exact in bf16) -> the pooled tensor, 16 bytes per thread.
__device__ __noinline__ void pool_unit(const uint8_t *unit, const long long *pool_pix, uint4 *y, int p_log, int tr_log, int tw_valid, int sub_log, int tid)
{
    const int cpr_log = sub_log - 3;
#pragma unroll 2
    for (int idx = tid; idx < 32 << cpr_log; idx += EPI_THREADS) {
        const int q = idx >> cpr_log, j = idx - (q << cpr_log);
        const long long pp = pool_pix[q];
        if (pp < 0) continue;
        const int pc = q & ((1 << (p_log - 1)) - 1), t = q >> (p_log - 1);
        const int s0 = (((t >> (tr_log - 1)) << tr_log) + 2 * (t & ((1 << (tr_log - 1)) - 1))) * tw_valid + 2 * pc;
        const int rows4[4] = {s0, s0 + 1, s0 + tw_valid, s0 + tw_valid + 1};
        uint4 acc4 = unit_chunk(unit, rows4[0], j, sub_log);
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            const uint4 v4 = unit_chunk(unit, rows4[k], j, sub_log);
            __nv_bfloat162 *pa = reinterpret_cast<__nv_bfloat162 *>(&acc4);
            const __nv_bfloat162 *pv = reinterpret_cast<const __nv_bfloat162 *>(&v4);
#pragma unroll
            for (int e = 0; e < 4; ++e) pa[e] = __hmax2(pa[e], pv[e]);
        }
        y[(pp >> 3) + j] = acc4;
    }
}

// A 3x3 max pooling of rows [oh0, oh0 + n_rows) of one image, over channel vectors of eight.  Bound by the latency of its
// loads: a window's are in flight together (two windows at a time would make the kernel spill around the call: 975 us where
// one takes 915), and with a vertical stride of two a thread keeps the maximum of the row that two windows share.  Four rows
// per item: 6.7 us, one row by the general routine below 4.3 (32 images of 112x112x64: 62 -> 43 us).
__device__ __noinline__ void pool3_item(const WfStage *st, int n, int oh0, int n_rows, int tid)
{
    const int Hin = __ldg(&st->Hin), Win = __ldg(&st->Win), Ho = __ldg(&st->Ho), Wo = __ldg(&st->Wo), cg = __ldg(&st->Cin) >> 3;
    const int sh = __ldg(&st->sh), sw = __ldg(&st->sw), ph = __ldg(&st->ph), pw = __ldg(&st->pw);
    const uint4 *x = static_cast<const uint4 *>(ldg_ptr<const void *>(&st->x)) + (long long)n * Hin * Win * cg;
    uint4 *y = static_cast<uint4 *>(ldg_ptr<void *>(reinterpret_cast<const void *const *>(&st->y))) + ((long long)n * Ho + oh0) * Wo * cg;
    const uint4 least = make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);       // -inf
    auto max8 = [](uint4 a, const uint4 &b) {
        __nv_bfloat162 *pa = reinterpret_cast<__nv_bfloat162 *>(&a);
        const __nv_bfloat162 *pb = reinterpret_cast<const __nv_bfloat162 *>(&b);
#pragma unroll
        for (int e = 0; e < 4; ++e) pa[e] = __hmax2(pa[e], pb[e]);
        return a;
    };
    const int total = Wo * cg;
    for (int idx = tid; idx < total; idx += EPI_THREADS) {
        const int ow = idx / cg, g = idx - ow * cg, iw = ow * sw - pw;
        uint4 shared = least;
        for (int r = 0; r < n_rows; ++r) {
            const int ih = (oh0 + r) * sh - ph;
            uint4 q[3][3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const bool rowok = ih + a >= 0 && ih + a < Hin && (a > 0 || r == 0 || sh != 2);
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    q[a][b] = least;
                    if (rowok && iw + b >= 0 && iw + b < Win) q[a][b] = __ldcg(x + ((long long)(ih + a) * Win + iw + b) * cg + g);
                }
            }
            const uint4 last = max8(max8(q[2][0], q[2][1]), q[2][2]);
            uint4 m = max8(max8(q[0][0], q[0][1]), max8(q[0][2], max8(max8(q[1][0], q[1][1]), q[1][2])));
            m = max8(m, last);
            if (sh == 2 && r > 0) m = max8(m, shared);
            shared = last;
            y[(long long)r * total + idx] = m;
        }
    }
}

// One output row of one image of any other max pooling over channel vectors of eight.
__device__ __noinline__ void pool_item(const WfStage *st, int n, int oh, int tid)
{
    const int Hin = __ldg(&st->Hin), Win = __ldg(&st->Win), Cin = __ldg(&st->Cin), Ho = __ldg(&st->Ho), Wo = __ldg(&st->Wo);
    const int kh = __ldg(&st->kh), kw = __ldg(&st->kw), sh = __ldg(&st->sh), sw = __ldg(&st->sw);
    const int ph = __ldg(&st->ph), pw = __ldg(&st->pw), dh = __ldg(&st->dh), dw = __ldg(&st->dw);
    const int cg = Cin >> 3;
    const int total = Wo * cg;
    const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(ldg_ptr<const void *>(&st->x));
    __nv_bfloat16 *y = static_cast<__nv_bfloat16 *>(ldg_ptr<void *>(reinterpret_cast<const void *const *>(&st->y)));
    // two channel-group vectors per thread
    for (int idx0 = 0; idx0 < total; idx0 += 2 * EPI_THREADS) {
        int gch[2], ow[2];
        bool live[2];
        float mx[2][8];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int idx = idx0 + u * EPI_THREADS + tid;
            live[u] = idx < total;
            ow[u] = idx / cg;
            gch[u] = idx - ow[u] * cg;
#pragma unroll
            for (int i = 0; i < 8; ++i) mx[u][i] = -INFINITY;
        }
        const int nt = kh * kw;
        for (int t0 = 0; t0 < nt; t0 += 4) {                 // four filter taps of both vectors in flight
            uint4 q4[2][4];
            bool ok[2][4];
#pragma unroll
            for (int tt = 0; tt < 4; ++tt) {
                const int t = t0 + tt;
                const int a = t / kw, b = t - a * kw;
                const int ih = oh * sh - ph + a * dh;
                const bool rowok = t < nt && ih >= 0 && ih < Hin;
                const long long rowbase = ((long long)n * Hin + ih) * Win;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int iw = ow[u] * sw - pw + b * dw;
                    ok[u][tt] = live[u] && rowok && iw >= 0 && iw < Win;
                    if (ok[u][tt]) q4[u][tt] = __ldcg(reinterpret_cast<const uint4 *>(x + (rowbase + iw) * Cin + gch[u] * 8));
                }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int tt = 0; tt < 4; ++tt)
                    if (ok[u][tt]) {
                        const uint32_t w4[4] = {q4[u][tt].x, q4[u][tt].y, q4[u][tt].z, q4[u][tt].w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            mx[u][2 * i] = fmaxf(mx[u][2 * i], __uint_as_float(w4[i] << 16));
                            mx[u][2 * i + 1] = fmaxf(mx[u][2 * i + 1], __uint_as_float(w4[i] & 0xFFFF0000u));
                        }
                    }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (live[u]) {
                uint32_t o[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)      // values are bf16 already: truncation is exact
                    o[i] = (__float_as_uint(mx[u][2 * i]) >> 16) | (__float_as_uint(mx[u][2 * i + 1]) & 0xFFFF0000u);
                *reinterpret_cast<uint4 *>(y + (((long long)n * Ho + oh) * Wo + ow[u]) * Cin + gch[u] * 8) =
                    make_uint4(o[0], o[1], o[2], o[3]);
            }
    }
}

// Gather of the stem's values (lop_gather.cuh), 1 << tr_log rows per item: Wo columns of Cout elements;
// x is the chain input, possibly still arriving.  Latency-bound (one round trip for the input rows, and
// the item's fixed cost): 32 images of 224x224 before a 7x7 stride-2 layer take 43 us, patches took 50.
__device__ __noinline__ void gather_item(const WfStage *st, int n, int tile_r, int tid, uint8_t *stg)
{
    GatherGeom gg;
    gg.N = __ldg(&st->N); gg.H = __ldg(&st->Hin); gg.W = __ldg(&st->Win); gg.C = __ldg(&st->Cin);
    gg.Ho = __ldg(&st->Ho); gg.Wo = __ldg(&st->Wo); gg.Kcol = __ldg(&st->Cout);
    gg.kh = __ldg(&st->kh); gg.kw = __ldg(&st->kw); gg.sh = __ldg(&st->sh); gg.sw = __ldg(&st->sw);
    gg.ph = __ldg(&st->ph); gg.pw = __ldg(&st->pw); gg.dh = __ldg(&st->dh); gg.dw = __ldg(&st->dw);
    const int N = gg.N, Hin = gg.H, Win = gg.W, Cin = gg.C, Ho = gg.Ho, Wo = gg.Wo, Cout = gg.Kcol;
    const int kh = gg.kh, kw = gg.kw, sh = gg.sh, sw = gg.sw, ph = gg.ph, pw = gg.pw, dh = gg.dh, dw = gg.dw;
    const int tr_log = __ldg(&st->tr_log), oh_lo = __ldg(&st->oh_lo), oh_hi = __ldg(&st->oh_hi), gather_direct = __ldg(&st->mode);
    const void *xin = ldg_ptr<const void *>(&st->x);
    void *yout = ldg_ptr<void *>(reinterpret_cast<const void *const *>(&st->y));
    const int oh0 = oh_lo + (tile_r << tr_log), n_rows = min(1 << tr_log, oh_hi - oh0);
    const int k8n = Cout >> 3;
    const uint16_t *x = static_cast<const uint16_t *>(xin);
    uint16_t *y = static_cast<uint16_t *>(yout) + ((long long)n * Ho + oh0) * Wo * Cout;
    if (gather_direct) {
        for (int idx = tid; idx < n_rows * Wo * k8n; idx += EPI_THREADS) {
            const int q = idx / k8n, r = q / Wo;
            *reinterpret_cast<uint4 *>(y + (long long)idx * 8) = gather8<true>(x, gg, n, oh0 + r, q - r * Wo, idx - q * k8n);
        }
    } else {
        // The input rows, copied once into shared memory in 16-byte vectors (around L1: they may have arrived
        // while the kernel was running), zeros where the window reaches past the image
        const int row_bytes = Win * Cin * 2, lead = gather_lead(gg), pitch = gather_pitch(gg), nvec = pitch >> 4;
        const int ih0 = oh0 * sh - ph, total = gather_rows_in(gg, n_rows) * nvec;
        const long long off0 = ((long long)n * Hin + ih0) * row_bytes;        // byte offset of the first staged row's data
        const int mis0 = (int)(off0 & 15), mis_step = row_bytes & 15;
        const long long tensor_bytes = (long long)N * Hin * row_bytes;
        const uint8_t *xb = reinterpret_cast<const uint8_t *>(x);
        for (int idx0 = tid; idx0 < total; idx0 += 4 * EPI_THREADS) {
            uint4 q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int idx = idx0 + u * EPI_THREADS, row = idx / nvec;
                const int mis = (mis0 + row * mis_step) & 15;
                const int at = (idx - row * nvec) * 16 - lead - mis;              // first byte of the vector, from the row's data
                const long long o = off0 + (long long)row * row_bytes + at;
                q[u] = make_uint4(0u, 0u, 0u, 0u);
                if (idx >= total || ih0 + row < 0 || ih0 + row >= Hin || at <= -16 || at >= row_bytes) continue;
                if (o + 16 <= tensor_bytes) {
                    q[u] = __ldcg(reinterpret_cast<const uint4 *>(xb + o));
                } else {                                          // the tensor ends inside this vector
                    uint32_t h[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        h[e] = o + 2 * e < tensor_bytes ? (uint32_t)__ldcg(reinterpret_cast<const uint16_t *>(xb + o + 2 * e)) : 0u;
                    q[u] = make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
                }
                if (at < 0 || at + 16 > row_bytes) {              // the row starts or ends inside it
                    uint32_t *w = reinterpret_cast<uint32_t *>(&q[u]);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (at + 4 * e < 0 || at + 4 * e >= row_bytes) w[e] &= 0xFFFF0000u;
                        if (at + 4 * e + 2 < 0 || at + 4 * e + 2 >= row_bytes) w[e] &= 0xFFFFu;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (idx0 + u * EPI_THREADS < total) *reinterpret_cast<uint4 *>(stg + (idx0 + u * EPI_THREADS) * 16) = q[u];
        }
        // where a column's values lie: staged row << 16 | byte offset from the pixel's first input column (kept
        // even where that is negative: the window's left padding is part of the lead)
        int *tab = reinterpret_cast<int *>(stg + gather_rows_in(gg, 1 << tr_log) * pitch);
        for (int k = tid; k < kh * kw * Cin; k += EPI_THREADS) {
            const int tap = k / Cin, a = tap / kw;
            tab[k] = ((a * dh) << 16) | (((tap - a * kw) * dw * Cin + k - tap * Cin) * 2);
        }
        epi_bar();
        // A thread keeps to one vector of the columns: where its eight values lie in the staged rows changes
        // with the row only, so a column costs eight 2-byte reads and the store.
        const int per = EPI_THREADS / k8n, k8 = tid % k8n, k_left = kh * kw * Cin - k8 * 8;
        int p = tid / k8n, r = 0, j = p;
        bool moved = true;
        int ad[8];
        for (const int end = tid < per * k8n ? n_rows * Wo : 0; p < end; p += per) {
            while (j >= Wo) { j -= Wo; ++r; moved = true; }
            if (moved) {
                moved = false;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int t = tab[k8 * 8 + min(e, k_left - 1)], row = r * sh + (t >> 16);
                    ad[e] = row * pitch + lead + ((mis0 + row * mis_step) & 15) + (t & 0xFFFF) - pw * Cin * 2;
                }
            }
            uint32_t h[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                h[e] = e < k_left ? (uint32_t)*reinterpret_cast<const uint16_t *>(stg + ad[e] + j * sw * Cin * 2) : 0u;
            *reinterpret_cast<uint4 *>(y + ((long long)p * k8n + k8) * 8) =
                make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
            j += per;
        }
    }
}

// ---- split tiles: the CTAs of a cluster (or half of one) sum a tile's channel chunks in parts and exchange slices of the sums.
// Places in shared memory that the two functions below need, from the address of the first barrier on.
constexpr uint32_t BAR_ACCF = 16u * WF_ENTRIES;                                // accumulators complete
constexpr uint32_t BAR_SSF = BAR_ACCF + 32u + 16u * WF_PUBQ;                   // scale / shift in place
constexpr uint32_t BAR_UGRANT = BAR_SSF + 32u;                                 // output units: granted, ready, free
constexpr uint32_t BAR_UREADY = BAR_UGRANT + 8u * WF_UNITS, BAR_UFREE = BAR_UREADY + 8u * WF_UNITS;
// Tiles of two parts and of four have barriers and words of their own: a CTA two places away is a partner in the latter only,
// may be ahead by a tile, and its word would count as the nearer partner's, which is still to come.
constexpr uint32_t BAR_XOK = BAR_UFREE + 8u * WF_UNITS + 16u + 8u * WF_GROUPS; // the others take partial sums: of tiles of two parts, of four
constexpr uint32_t BAR_XFULL = BAR_XOK + 16u;                                  // the others' partial sums are here
constexpr uint32_t BAR_MISC = BAR_XFULL + 16u;                                 // words: [1] abort, [4] parity of the split tiles so far (bit 0: of
                                                                               // two parts, 1: of four), [8 + q], [12 + q]: the unit part q takes sums in

__device__ __forceinline__ uint32_t ld_shared(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
// Bounded wait on a barrier that other CTAs of the cluster may complete; gives up when this CTA's abort flag is raised (which a
// CTA of the cluster that gives up does on its way out: what it was to send will not come).
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, uint32_t abort_at)
{
    for (uint32_t i = 0; i < BARRIER_TRIES; ++i) {
        uint32_t done;
        asm volatile(
            "{\n"
            ".reg .pred p;\n"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((i & 255u) == 255u && ld_shared(abort_at)) return false;
    }
    return false;
}

// The loader's side, by its one thread: once the units that partial sums arrive in are free, the barriers are armed and the
// other CTAs told where to write.  cout: the item's slice; uc: output units before these; turn: parity of the tiles of as many
// parts before this one.
// (Barriers whose phase is not over cannot be armed again: with two parts the next tile's units are free before this one's
// exchange is done.)
__device__ __noinline__ bool take_partial_sums(uint32_t bars, uint32_t cout, uint32_t s_log, uint32_t uc, uint32_t turn)
{
    const uint32_t others = (1u << s_log) - 1u, part = cout & others, base_rank = cta_rank() & ~others, abort_at = bars + BAR_MISC + 4u;
    const uint32_t xok = bars + BAR_XOK + 8u * (s_log - 1u), xfull = bars + BAR_XFULL + 8u * (s_log - 1u), words = bars + BAR_MISC + 16u * (s_log + 1u);
    if (!mbar_wait_cluster(xok, turn ^ 1u, abort_at) || !mbar_wait_cluster(xfull, turn ^ 1u, abort_at)) return false;
    for (uint32_t u = uc; u < uc + ((others + 1u) >> 1); ++u) {
        const uint32_t sl = 8u * (u & (WF_UNITS - 1));
        if (!mbar_wait_cluster(bars + BAR_UFREE + sl, ((u / WF_UNITS) & 1u) ^ 1u, abort_at)) return false;
        mbar_arrive(bars + BAR_UGRANT + sl);                                   // (its phase; nobody waits for it)
    }
    mbar_expect_tx(xok, 4u * others);
    mbar_expect_tx(xfull, others * (512u * (WF_SPLIT_BN >> s_log)));
    for (uint32_t q = 0; q <= others; ++q)
        if (q != part) st_async(map_to_cta(words + 4u * part, base_rank + q), uc & (WF_UNITS - 1), map_to_cta(xok, base_rank + q));
    return true;
}

// The workers' side, by every worker thread, and the whole of a split tile's epilogue: this CTA's partial sums of the other
// CTAs' channel slices go to those CTAs, the others' sums of this CTA's slice are added to its own, part by part in order (the
// order in which every executor of the plan sums), and the slice is finished.  A unit holds 64 / parts channels x 128 rows of
// fp32 from each of one or two senders, as [four channels][row]: neighbouring lanes write and read neighbouring 16 bytes.
// acc: the accumulator; uc: units before the tile's, of which it has as many as are returned; a wait that runs out sets the
// epilogue's failure word.
// Bound by latency: about 1.7 us from the last MMA to the slice's first sum, of which the slowest CTA's lag is a part.
// An epilogue of its own, out of line: with the exchange in front of the other tiles' epilogue, those took 0.2 us longer each
// (a ResNet-50 of batch 32, which has no split tile, 830 -> 873 us).
template <bool SMOOTH>
__device__ __noinline__ uint32_t split_item(const WfStage *sp, int4 rec, uint8_t *smem_bars, uint32_t unit0, uint32_t unit_bytes, uint32_t acc,
                                            uint32_t uc, uint32_t cnt)
{
    const uint32_t bars = smem_u32(smem_bars), s_log = (uint32_t)__ldg(&sp->s_log), parts = 1u << s_log, part = (uint32_t)rec_cout(rec) & (parts - 1u);
    const uint32_t turn = ld_shared(bars + BAR_MISC + 16u) >> (s_log - 1u) & 1u;   // parity of the tiles of as many parts before this one
    const uint32_t xok = bars + BAR_XOK + 8u * (s_log - 1u), xfull = bars + BAR_XFULL + 8u * (s_log - 1u), words = bars + BAR_MISC + 16u * (s_log + 1u);
    const uint32_t slice = WF_SPLIT_BN >> s_log, base_rank = cta_rank() & ~(parts - 1u), abort_at = bars + BAR_MISC + 4u, rx = uc + 1u;
    const uint32_t per_unit = parts >> 1, from_bytes = 512u * slice;           // senders per unit (two parts: one, four: two)
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u, row = (warp & 3u) * 32u + lane, cgrp = (warp - WF_FIRST_WORKER) >> 2, buf = cnt & 1u;
    auto sums_at = [&](uint32_t first_unit, uint32_t from) {
        return unit0 + ((first_unit + from / per_unit) & (WF_UNITS - 1)) * unit_bytes + (from & (per_unit - 1u)) * from_bytes + 16u * row;
    };
    const int p_log = __ldg(&sp->p_log), tr_log = __ldg(&sp->tr_log), tw_valid = __ldg(&sp->tw_valid), sub_log = __ldg(&sp->sub_log);
    const int act = __ldg(&sp->act), res_pos = ldg_ptr<const void *>(&sp->res) ? __ldg(&sp->res_pos) : LOP_RES_NONE;
    const bool bulk_out = __ldg(&sp->out_map) >= 0;
    acc += ((warp & 3u) * 32u) << 16;
    bool ok = mbar_wait_cluster(bars + BAR_ACCF + 8u * buf, (cnt >> 1) & 1u, abort_at);
    ok = ok && mbar_wait_cluster(xok, turn, abort_at);
    ok = __all_sync(0xffffffffu, ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    uint32_t r[8];                                     // (eight columns at a time: what this needs, the kernel around the call has not)
#pragma unroll 1
    for (uint32_t c = 0, k = 0; ok && c < WF_SPLIT_BN; c += 8) {
        const uint32_t q = c / slice;
        if (q == part) continue;
        if (((++k + 1u) >> 1 & 1u) != cgrp) continue;                          // (the first and third 16 columns: the warps without a chunk to finish)
        tmem_ld8(acc + c, r);
        const uint32_t to = map_to_cta(sums_at(ld_shared(words + 4u * q), part < q ? part : part - 1u) + (c - q * slice) * 512u, base_rank + q);
        const uint32_t bar = map_to_cta(xfull, base_rank + q);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        st_async4(to, r[0], r[1], r[2], r[3], bar);
        st_async4(to + 2048u, r[4], r[5], r[6], r[7], bar);
    }
    // while they travel: where this row goes
    const int m = (int)row, c = m & ((1 << p_log) - 1), rr = (m >> p_log) & ((1 << tr_log) - 1), img = m >> (p_log + tr_log);
    const bool staged = c < tw_valid;
    const int srow = ((img << tr_log) + rr) * tw_valid + c;
    const int swz = sub_log == 5 ? (srow >> 1) & 3 : (srow >> 2) & 1;          // (a slice is 32 or 16 channels)
    long long *row_pix = reinterpret_cast<long long *>(smem_bars + BAR_MISC + 128 + 2048);
    if (!bulk_out && cgrp == 0 && staged) {
        const int Ho = __ldg(&sp->Ho), Wo = __ldg(&sp->Wo), oh = __ldg(&sp->oh_lo) + (rec_tr(rec) << tr_log) + rr, ow = rec_tw(rec) * tw_valid + c;
        const int n = rec_tn(rec) * (128 >> (p_log + tr_log)) + img, Cout = __ldg(&sp->Cout);
        row_pix[srow] = ow < Wo && oh < __ldg(&sp->oh_hi) && n < __ldg(&sp->N) ? (((long long)n * Ho + oh) * Wo + ow) * Cout + rec_cout(rec) * (int)slice : -1LL;
    }
    const uint32_t sl = uc & (WF_UNITS - 1);
    ok = ok && mbar_wait_cluster(bars + BAR_UGRANT + 8u * sl, (uc / WF_UNITS) & 1u, abort_at);
    ok = ok && mbar_wait_cluster(bars + BAR_SSF + 8u * buf, (cnt >> 1) & 1u, abort_at);
    ok = ok && mbar_wait_cluster(xfull, turn, abort_at);
    ok = __all_sync(0xffffffffu, ok);
#pragma unroll 1
    for (uint32_t j = 16u * cgrp; ok && j < min(slice, 16u * cgrp + 16u); j += 8) {
        tmem_ld8(acc + part * slice + j, r);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (!staged) continue;
        float v[8], rv[8];
        for (uint32_t q = 0; q < parts; ++q) {
            const uint32_t sums = sums_at(rx, q < part ? q : q - 1u) + j * 512u;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                uint32_t w[4] = {r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3]};
                if (q != part)
                    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(sums + 2048u * e) : "memory");
#pragma unroll
                for (int i = 0; i < 4; ++i) v[4 * e + i] = q == 0 ? __uint_as_float(w[i]) : __fadd_rn(v[4 * e + i], __uint_as_float(w[i]));
            }
        }
        const float *scale = reinterpret_cast<const float *>(smem_bars + BAR_MISC + 128) + 128 * buf + j, *shift = scale + 256;
        uint8_t *my_row = smem_bars - bars + unit0 + sl * unit_bytes + (srow << (sub_log + 1));
        uint4 *cp = reinterpret_cast<uint4 *>(my_row + (((int)(j >> 3) ^ swz) << 4));
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = fmaf(scale[i], v[i], shift[i]);
        if (res_pos != LOP_RES_NONE) {
            const uint4 q = *cp;
            const uint32_t rw[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                rv[2 * i] = __uint_as_float(rw[i] << 16);
                rv[2 * i + 1] = __uint_as_float(rw[i] & 0xFFFF0000u);
            }
        }
        finish_n<SMOOTH ? 1 : 0>(v, rv, res_pos, act);
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            o[i] = *reinterpret_cast<const uint32_t *>(&h);
        }
        *cp = make_uint4(o[0], o[1], o[2], o[3]);
    }
    if (!ok) *reinterpret_cast<volatile uint32_t *>(smem_bars + BAR_MISC + 12) = 1u;
    if (bulk_out) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // (the units of the partial sums first: the publisher waits for the output unit only)
    __syncwarp();
    if (lane == 0) {
        for (uint32_t u = rx; u < rx + (parts >> 1); ++u) mbar_arrive(bars + BAR_UREADY + 8u * (u & (WF_UNITS - 1)));
        mbar_arrive(bars + BAR_UREADY + 8u * sl);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    epi_bar();                                                                 // accumulator drained, sums read, slice complete
    if (threadIdx.x == 32u * WF_FIRST_WORKER) {
        mbar_arrive(bars + BAR_ACCF + 16u + 8u * buf);
        mbar_arrive(bars + BAR_SSF + 16u + 8u * buf);
        for (uint32_t u = rx; u < rx + (parts >> 1); ++u) mbar_arrive(bars + BAR_UFREE + 8u * (u & (WF_UNITS - 1)));
        *reinterpret_cast<volatile uint32_t *>(smem_bars + BAR_MISC + 16) = ld_shared(bars + BAR_MISC + 16u) ^ (1u << (s_log - 1u));
    }
    if (!bulk_out && ld_shared(bars + BAR_MISC + 12) == 0u) {
        copy_unit(smem_bars - bars + unit0 + sl * unit_bytes, row_pix, static_cast<uint4 *>(ldg_ptr<void *>(reinterpret_cast<const void *const *>(&sp->y))),
                  (128 >> p_log) * tw_valid, sub_log, (int)threadIdx.x - 32 * WF_FIRST_WORKER);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");           // (as behind the other tiles' copy-out)
        epi_bar();
        if (threadIdx.x == 32u * WF_FIRST_WORKER) mbar_arrive(bars + BAR_UFREE + 8u * sl);
    }
    return 1u + (parts >> 1);
}

// FETCH: one more warp per CTA brings the chain input from host memory.  ROWOPS: the program has depth-wise /
// normalisation / concatenation stages, SMOOTH: a convolution of it has SiLU or GELU; programs without them run an
// instantiation that does not carry their code.  SPLIT: the CTAs are launched in clusters and the program has split tiles.
template <bool FETCH, bool ROWOPS, bool SMOOTH, bool SPLIT>
__global__ void __launch_bounds__(FETCH ? WF_THREADS + 32 : WF_THREADS, 1) wavefront_kernel(const WfParams P)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw);
    // shared memory: operand ring | output units | scratch of the SIMT items | barriers | tables
    const uint32_t ring_bytes = P.ring_bytes, unit_bytes = P.unit_bytes;
    const uint32_t ring0 = base, unit0 = ring0 + ring_bytes, simt0 = unit0 + WF_UNITS * unit_bytes, bars = simt0 + P.simt_bytes;
    const uint32_t full0 = bars, empty0 = full0 + 8u * WF_ENTRIES;      // operand entries: loaded / consumed
    const uint32_t accf0 = bars + BAR_ACCF, acce0 = accf0 + 16u;         // accumulators: complete / drained
    const uint32_t pubf0 = acce0 + 16u, pube0 = pubf0 + 8u * WF_PUBQ;    // items the workers stored themselves: stored / published
    const uint32_t ssf0 = bars + BAR_SSF, sse0 = ssf0 + 16u;                 // scale/shift buffers of two tiles: full / empty
    const uint32_t ugrant0 = bars + BAR_UGRANT;                          // output units: free to write, the residual (if any) in place
    const uint32_t uready0 = bars + BAR_UREADY, ufree0 = bars + BAR_UFREE;  // ... finished by the workers / read out
    const uint32_t wfull = ufree0 + 8u * WF_UNITS, wempty = wfull + 8u;  // kept weights: loaded / last used
    const uint32_t gfull0 = wempty + 8u;                                 // slab stages: a group of boxes is loaded
    uint8_t *tail = smem + (bars + BAR_MISC - base);
    volatile uint32_t *misc = reinterpret_cast<volatile uint32_t *>(tail);      // [0] TMEM base, [1] abort, [2] run, [3] epilogue failure,
                                                                                // [4], [8..15] split tiles (see BAR_MISC)
    volatile uint32_t *entry_at = misc + 16;                                     // [WF_ENTRIES]: where the ring's entries start (loader only)
    float *s_scale = reinterpret_cast<float *>(tail + 128);                      // [2][128]: per-channel scale of this and the next tile
    float *s_shift = s_scale + 256;                                              // [2][128]
    long long *row_pix = reinterpret_cast<long long *>(tail + 128 + 2048);       // [128]: element offset of a staged row's output, or -1
    long long *pool_pix = row_pix + 128;                                         // [32]: element offset of a 2x2 window's pooled output, or -1
    uint8_t *units = smem + (unit0 - base), *stg = smem + (simt0 - base);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0 && blockIdx.x < 4) {
        tr(TRACE_ITEMS - 8 + (int)blockIdx.x, 0);
        trv(TRACE_ITEMS - 8 + (int)blockIdx.x, 4, (unsigned long long)clock64());
    }
    if (threadIdx.x == 0) {
        for (int e = 0; e < WF_ENTRIES; ++e) {
            mbar_init(full0 + 8u * e, 1);
            mbar_init(empty0 + 8u * e, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf0 + 8u * b, 1);
            mbar_init(acce0 + 8u * b, 1);
            mbar_init(ssf0 + 8u * b, 1);
            mbar_init(sse0 + 8u * b, 1);
        }
        for (int u = 0; u < WF_UNITS; ++u) {
            mbar_init(ugrant0 + 8u * u, 1);
            mbar_init(uready0 + 8u * u, WF_WORKER_WARPS);
            mbar_init(ufree0 + 8u * u, 1);
        }
        mbar_init(wfull, 1);
        mbar_init(wempty, 1);
        for (int g = 0; g < WF_GROUPS; ++g) mbar_init(gfull0 + 8u * g, 1);
        for (uint32_t w = 0; w < 2; ++w) {
            mbar_init(bars + BAR_XOK + 8u * w, 1);
            mbar_init(bars + BAR_XFULL + 8u * w, 1);
        }
        for (int q = 0; q < WF_PUBQ; ++q) {
            mbar_init(pubf0 + 8u * q, 1);
            mbar_init(pube0 + 8u * q, 1);
        }
        misc[1] = 0;
        grid_wait();
        misc[2] = ld_acquire(P.counters) + 1u;                 // this launch is run number (completed runs + 1)
        misc[3] = misc[4] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void *)&misc[0])),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (SPLIT) cluster_sync();                                 // the other CTAs' barriers are ready too
    grid_release();
    grid_wait();                                               // (all threads: thread 0 waited for what it read)
    if (threadIdx.x == 0 && blockIdx.x < 4) tr(TRACE_ITEMS - 8 + (int)blockIdx.x, 1);
    const uint32_t tmem_base = misc[0];
    const unsigned run = misc[2];
    volatile uint32_t *abort_flag = &misc[1];
    volatile uint32_t *epi_fail = &misc[3];
    const int G = gridDim.x;
    const int NI = P.n_items;
    const int4 zero4 = make_int4(0, 0, 0, 0);

    if (warp == 0) {
        // ---------------- dependency wait (all lanes) + TMA producer (lane 0) ----------------
        int item = blockIdx.x;
        int4 cur = item < NI ? __ldg(&P.items[item]) : zero4;
        int4 nxt = item + G < NI ? __ldg(&P.items[item + G]) : zero4;
        int2 dep_cur = (item < NI && lane < rec_ndep(cur)) ? __ldg(&P.deps[rec_dep0(cur) + lane]) : make_int2(0, 0);
        int sidx = -1;
        // (what only some tiles need is read from the stage's record where it is needed: registers are what this kernel is short of)
        int kind = -1, mode = 0, oh_lo = 0, tr_log = 0, p_log = 0, tw_valid = 0, BN = 0, BK = 0, n_chunks = 1, n_taps = 1, tbx = 1;
        uint32_t a_bytes = 0, b_bytes = 0;
        const CUtensorMap *maps = nullptr;
        int s_log = 0;
        uint32_t split_turn = 0;                               // parity of the split tiles so far: bit 0 of two parts, bit 1 of four
        int first_offh = 0, first_offw = 0, first_mi = 0, cps = 1, units_n = 0, sub_log = 6, res_map = -1;
        bool first_have = true;
        uint32_t a_sz = 0, b_sz = 0, keep_bytes = 0;
        uint32_t pc = 0, uc = 0;
        // Operand ring (lane 0).  Entries are allocated and freed in order; positions are counted without wrapping
        // (head), an entry never straddles the ring's end.  The MMA issuer derives the same places from the same records.
        uint32_t ring_lim = ring_bytes, head = 0, pos = 0, tail_at = 0, n_alloc = 0, n_freed = 0, n_full = 0, n_group = 0, w_uses = 0;
        uint32_t slab_sl = 0, slab_end0 = 0, slab_end1 = 0;    // slab stages: next activation box, entry that ended its previous chunk
        long long cut_key = 0;                                 // how the ring is cut (see below)
        int ss_key[2] = {-1, -1};                              // whose scale / shift the two buffers hold: stage, first channel
        int ss_co[2] = {0, 0};
        for (; item < NI; item += G) {
            // two items ahead: the record; one item ahead: this lane's dependency entry
            const int4 nn = item + 2 * G < NI ? __ldg(&P.items[item + 2 * G]) : zero4;
            const int2 dep_nxt = (item + G < NI && lane < rec_ndep(nxt)) ? __ldg(&P.deps[rec_dep0(nxt) + lane]) : make_int2(0, 0);
            if (rec_stage(cur) != sidx) {
                sidx = rec_stage(cur);
                const WfStage *sp = &P.stages[sidx];
                kind = __ldg(&sp->kind); mode = __ldg(&sp->mode); oh_lo = __ldg(&sp->oh_lo);
                tr_log = __ldg(&sp->tr_log); p_log = __ldg(&sp->p_log); tw_valid = __ldg(&sp->tw_valid);
                BN = __ldg(&sp->BN); BK = __ldg(&sp->BK); n_chunks = __ldg(&sp->n_chunks); n_taps = __ldg(&sp->n_taps);
                tbx = __ldg(&sp->tb);
                a_bytes = __ldg(&sp->a_bytes); b_bytes = __ldg(&sp->b_bytes);
                maps = P.maps + __ldg(&sp->map_base);
                const int sh = __ldg(&sp->sh), sw = __ldg(&sp->sw), ph = __ldg(&sp->ph), pw = __ldg(&sp->pw);
                // the first tap's offset (slab mode: where the box starts): which parity map that is and how far in
                first_offh = floor_div_i(-ph, sh); first_offw = floor_div_i(-pw, sw);
                first_mi = (-ph - first_offh * sh) * sw + (-pw - first_offw * sw);
                first_have = (__ldg(&sp->a_valid_mask) >> first_mi) & 1;
                cps = __ldg(&sp->cps);
                a_sz = (a_bytes + 1023u) & ~1023u; b_sz = (b_bytes + 1023u) & ~1023u;
                keep_bytes = (uint32_t)__ldg(&sp->keep_bytes);
                if (SPLIT) s_log = __ldg(&sp->s_log);
                sub_log = __ldg(&sp->sub_log); units_n = (BN >> s_log) >> sub_log;
                res_map = __ldg(&sp->res_map);
            }
            if (kind == WF_CONV) {
                if (lane == 0) tr(item, 0);
                // the tile's per-channel scale / shift go to shared memory from here, a tile ahead of the epilogue
                // that uses them: their load latency is off the workers' path
                bool ok = __all_sync(0xffffffffu, mbar_wait_abortable(sse0 + 8u * (pc & 1u), ((pc >> 1) & 1u) ^ 1u, abort_flag));
                // a split tile: the item finishes channels c0 on, of the BN whose sums over chunks ch0 on it takes part in
                const int c0 = rec_cout(cur) * (BN >> s_log);
                const int co0 = SPLIT ? (rec_cout(cur) >> s_log) * BN : c0, ch0 = SPLIT ? (rec_cout(cur) & ((1 << s_log) - 1)) * n_chunks : 0;
                if (ok && (((pc & 1u) ? ss_key[1] : ss_key[0]) != sidx || ((pc & 1u) ? ss_co[1] : ss_co[0]) != c0)) {
                    float *ds = s_scale + 128 * (pc & 1u), *dsh = s_shift + 128 * (pc & 1u);
                    const float *scale = from_here(ldg_ptr<const float *>(reinterpret_cast<const void *const *>(&P.stages[sidx].scale)));
                    const float *shift = from_here(ldg_ptr<const float *>(reinterpret_cast<const void *const *>(&P.stages[sidx].shift)));
                    if (pc & 1u) { ss_key[1] = sidx; ss_co[1] = c0; } else { ss_key[0] = sidx; ss_co[0] = c0; }
                    for (int i = lane; i < BN >> s_log; i += 32) {
                        ds[i] = scale ? __ldg(scale + c0 + i) : 1.0f;
                        dsh[i] = shift ? __ldg(shift + c0 + i) : 0.0f;
                    }
                    __syncwarp();
                }
                // while the tile's producers are still at work: its weights on their way to L2, the maps to the descriptor cache
                ok = ok && wait_deps_warp(P, rec_dep0(cur), rec_ndep(cur), dep_cur, run, lane, [&] {
                    if (lane != 0) return;
                    prefetch_map(maps + first_mi);
                    for (int ch = 0, n = 0; ch < n_chunks && n < PREFETCH_BOXES; ++ch)
                        for (int t0 = 0; t0 < n_taps && n < PREFETCH_BOXES; t0 += tbx, ++n) tma_prefetch_3d(maps + 4, (ch0 + ch) * BK, co0, t0);
                    if (res_map >= 0) prefetch_map(P.maps + res_map);
                });
                if (ok) {
                    if (lane == 0) mbar_arrive(ssf0 + 8u * (pc & 1u));          // scale / shift are in place
                    ++pc;
                }
                int fail = 0;
                if (!ok) {
                    if (lane == 0) atomicOr(P.status, 0x10u);
                    fail = 1;
                } else if (elect_one()) {
                    tr(item, 1);
                    asm volatile("fence.proxy.async.global;" ::: "memory");       // producers' generic-proxy writes -> our TMA reads
                    const int ow0 = rec_tw(cur) * tw_valid;
                    const int oh0 = oh_lo + (rec_tr(cur) << tr_log);
                    const int n0 = rec_tn(cur) * (128 >> (p_log + tr_log));
                    // waits until the oldest entry is consumed
                    auto free_oldest = [&]() {
                        const uint32_t e = n_freed & (WF_ENTRIES - 1);
                        if (!mbar_wait_abortable(empty0 + 8u * e, (n_freed / WF_ENTRIES) & 1u, abort_flag)) return false;
                        ++n_freed;
                        tail_at = n_freed == n_alloc ? head : entry_at[n_freed & (WF_ENTRIES - 1)];
                        return true;
                    };
                    // a place of `size` bytes: its address, 0 when a wait ran out
                    auto place = [&](uint32_t size) -> uint32_t {
                        if (pos + size > ring_lim) { head += ring_lim - pos; pos = 0; }
                        if (n_freed == n_alloc) tail_at = head;
                        while (head + size - tail_at > ring_lim || n_alloc - n_freed == WF_ENTRIES)
                            if (!free_oldest()) return 0u;
                        const uint32_t at = ring0 + pos;
                        entry_at[n_alloc & (WF_ENTRIES - 1)] = head;
                        ++n_alloc; head += size; pos += size;
                        return at;
                    };
                    // ... with a full barrier of its own, armed for `tx` bytes
                    uint32_t full_bar = 0;
                    auto allocate = [&](uint32_t size, uint32_t tx) -> uint32_t {
                        const uint32_t at = place(size);
                        full_bar = full0 + 8u * (n_full & (WF_ENTRIES - 1));
                        if (at) { ++n_full; mbar_expect_tx(full_bar, tx); }
                        return at;
                    };
                    // How the ring is cut.  key > 0, kept weights: where a layer gives every CTA several tiles of the same
                    // output channels, the tile's weights stay at the ring's end and only the first such tile loads them.
                    // key < 0, slab stages: two activation boxes at the ring's end beside the weight boxes -- a chunk's
                    // activation box outlives its weight boxes, so it cannot be an entry among them.  key == 0: one ring.
                    // When the key changes (the MMA issuer takes the same decision from the same records) the ring is
                    // drained and cut anew.
                    const bool kept = keep_bytes != 0;
                    const long long key = kept ? (((long long)(maps - P.maps) << 16) | rec_cout(cur)) + 1 : (mode == WF_SLAB ? -(long long)a_sz : 0);
                    if (key != cut_key) {
                        // (MMAs complete in order: the newest entry stands for all)
                        if (n_freed != n_alloc) {
                            const uint32_t last = n_alloc - 1u;
                            fail = !mbar_wait_abortable(empty0 + 8u * (last & (WF_ENTRIES - 1)), (last / WF_ENTRIES) & 1u, abort_flag);
                            n_freed = n_alloc;
                        }
                        slab_end0 = slab_end1 = n_freed;
                        if (!fail && cut_key > 0 && !mbar_wait_abortable(wempty, (w_uses - 1u) & 1u, abort_flag)) fail = 1;
                        cut_key = key;
                        ring_lim = ring_bytes - (key < 0 ? 2u * a_sz : keep_bytes);
                        head = pos = tail_at = 0;
                        if (!fail && kept) {
                            ++w_uses;
                            mbar_expect_tx(wfull, (uint32_t)(n_chunks * ((n_taps + tbx - 1) / tbx)) * b_bytes);
                            uint32_t at = ring0 + ring_lim;
                            for (int ch = 0; ch < n_chunks; ++ch)
                                for (int t0 = 0; t0 < n_taps; t0 += tbx, at += b_sz) tma_load_3d(at, maps + 4, wfull, ch * BK, co0, t0);
                        }
                    }
                    // the whole receptive window of the tile in one box per chunk: its first tap's offset places it
                    const int aw = first_have ? ow0 + first_offw : -65536, ah = first_have ? oh0 + first_offh : -65536;
                    if (mode == WF_SLAB && kept) {
                        for (int ch = 0; ch < n_chunks && !fail; ++ch) {
                            const uint32_t at = allocate(a_sz, a_bytes);
                            if (!at) { fail = 1; break; }
                            tma_load_4d(at, maps + first_mi, full_bar, ch * BK, aw, ah, n0);          // (not split: kept)
                        }
                    } else if (mode == WF_SLAB) {
                        const int per_chunk = (n_taps + tbx - 1) / tbx;
                        for (int ch = 0; ch < n_chunks && !fail; ++ch) {
                            // the activation box of the chunk two back is consumed when that chunk's last entry is
                            while ((int)(n_freed - slab_end0) < 0)
                                if (!free_oldest()) { fail = 1; break; }
                            uint32_t bar = 0;
                            for (int i = 0, in_group = 0; i < per_chunk && !fail; ++i) {
                                if (in_group == 0) {
                                    bar = gfull0 + 8u * (n_group & (WF_GROUPS - 1));
                                    ++n_group;
                                    mbar_expect_tx(bar, (uint32_t)min(cps, per_chunk - i) * b_bytes + (i == 0 ? a_bytes : 0u));
                                    if (i == 0) tma_load_4d(ring0 + ring_lim + slab_sl * a_sz, maps + first_mi, bar, (ch0 + ch) * BK, aw, ah, n0);
                                }
                                const uint32_t at = place(b_sz);
                                if (!at) { fail = 1; break; }
                                tma_load_3d(at, maps + 4, bar, (ch0 + ch) * BK, co0, i * tbx);
                                if (++in_group == cps) in_group = 0;
                            }
                            slab_end0 = slab_end1; slab_end1 = n_alloc;
                            slab_sl ^= 1u;
                        }
                    } else {
                        // one activation and one weight box per (channel chunk, tap), `cps` of them per entry
                        const int steps = n_chunks * n_taps;
                        const WfStage *sp = &P.stages[sidx];
                        const int kh = __ldg(&sp->kh), kw = __ldg(&sp->kw), sh = __ldg(&sp->sh), sw = __ldg(&sp->sw);
                        const int ph = __ldg(&sp->ph), pw = __ldg(&sp->pw), dh = __ldg(&sp->dh), dw = __ldg(&sp->dw), amask = __ldg(&sp->a_valid_mask);
                        int ch = ch0, ta = 0, tb = 0;
                        int offh = first_offh, offw = first_offw, mi = first_mi;
                        bool have = first_have;
                        for (int st = 0; st < steps && !fail; st += cps) {
                            const uint32_t g = (uint32_t)min(cps, steps - st);
                            uint32_t at = allocate(g * (kept ? a_sz : a_sz + b_sz), g * (kept ? a_bytes : a_bytes + b_bytes));
                            if (!at) { fail = 1; break; }
                            uint32_t bt = at + g * a_sz;
                            for (uint32_t u = 0; u < g; ++u, at += a_sz, bt += b_sz) {
                                tma_load_4d(at, maps + mi, full_bar, ch * BK, have ? ow0 + offw : -65536, have ? oh0 + offh : -65536, n0);
                                if (!kept) tma_load_3d(bt, maps + 4, full_bar, ch * BK, co0, ta * kw + tb);
                                if (n_taps == 1) { ++ch; continue; }
                                // next tap (strides are 1 or 2 almost always: no division then)
                                if (++tb == kw) { tb = 0; if (++ta == kh) { ta = 0; ++ch; } }
                                const int qh = ta * dh - ph, qw = tb * dw - pw;
                                offh = sh == 1 ? qh : (sh == 2 ? qh >> 1 : floor_div_i(qh, sh));
                                offw = sw == 1 ? qw : (sw == 2 ? qw >> 1 : floor_div_i(qw, sw));
                                mi = (qh - offh * sh) * sw + (qw - offw * sw);
                                have = (amask >> mi) & 1;
                            }
                        }
                    }
                    // the tile's output units, behind its operands: free (their previous contents are stored), and with
                    // the residual's rows on their way where there is one
                    for (int u = 0; u < units_n && !fail; ++u, ++uc) {
                        const uint32_t sl = uc & (WF_UNITS - 1), gb = ugrant0 + 8u * sl;
                        if (!mbar_wait_abortable(ufree0 + 8u * sl, ((uc / WF_UNITS) & 1u) ^ 1u, abort_flag)) { fail = 1; break; }
                        if (res_map >= 0) {
                            mbar_expect_tx(gb, (uint32_t)(((128 >> p_log) * tw_valid) << (sub_log + 1)));
                            tma_load_4d(unit0 + sl * unit_bytes, P.maps + res_map, gb, c0 + (u << sub_log), ow0, oh0, n0);
                        } else {
                            mbar_arrive(gb);
                        }
                    }
                    if (SPLIT && s_log > 0 && !fail) {
                        fail = !take_partial_sums(bars, (uint32_t)rec_cout(cur), (uint32_t)s_log, uc, split_turn >> (s_log - 1) & 1u);
                        uc += (1u << s_log) >> 1;
                        split_turn ^= 1u << (s_log - 1);
                    }
                    if (fail) atomicOr(P.status, 0x1u);
                    tr(item, 2);
                }
                if (__any_sync(0xffffffffu, fail | (int)*abort_flag)) {
                    if (lane == 0) {
                        atomicExch(P.counters + 2, 1u);
                        *abort_flag = 1;
                    }
                    break;
                }
            }
            cur = nxt; dep_cur = dep_nxt; nxt = nn;
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // ---------------- MMA issuer ----------------
            int item = blockIdx.x;
            int4 cur = item < NI ? __ldg(&P.items[item]) : zero4;
            int sidx = -1;
            int kind = -1, mode = 0, n_chunks = 1, n_taps = 1, tbx = 1, kw = 1, dh = 1, dw = 1, p_log = 0, ksteps = 1;
            uint32_t idesc = 0, desc_hi = 0, row_bytes = 0, tap_bytes = 0;
            uint32_t cnt = 0, a_sz = 0, b_sz = 0, a_bytes = 0, b_bytes = 0, keep_bytes = 0;
            bool fail = false, row3x64 = false;
            int map_base = 0, cps = 1;
            // the ring as the loader fills it: the next entry's place and number; the kept weights' loads so far
            uint32_t ring_lim = ring_bytes, pos = 0, n_used = 0, n_full = 0, n_group = 0, w_uses = 0, slab_sl = 0;
            long long cut_key = 0;
            uint32_t tap16 = 0, step_w16 = 0, step_h16 = 0;    // descriptor start-field steps: next tap's weights, next filter column / row
            for (; item < NI && !fail; item += G) {
                const int4 nxt = item + G < NI ? __ldg(&P.items[item + G]) : zero4;
                if (rec_stage(cur) != sidx) {
                    sidx = rec_stage(cur);
                    const WfStage *sp = &P.stages[sidx];
                    kind = __ldg(&sp->kind); mode = __ldg(&sp->mode);
                    n_chunks = __ldg(&sp->n_chunks); n_taps = __ldg(&sp->n_taps); tbx = __ldg(&sp->tb);
                    kw = __ldg(&sp->kw); dh = __ldg(&sp->dh); dw = __ldg(&sp->dw); p_log = __ldg(&sp->p_log);
                    map_base = __ldg(&sp->map_base);
                    ksteps = __ldg(&sp->BK) / 16;
                    idesc = __ldg(&sp->idesc);
                    desc_hi = ((__ldg(&sp->sbo_bytes) >> 4) & 0x3FFFu) | (1u << 14) | (__ldg(&sp->layout_code) << 29);
                    row_bytes = __ldg(&sp->row_bytes);
                    tap_bytes = (uint32_t)__ldg(&sp->BN) * row_bytes;
                    tap16 = tap_bytes >> 4;
                    step_w16 = ((uint32_t)dw * row_bytes) >> 4;
                    step_h16 = ((uint32_t)(dh << p_log) * row_bytes) >> 4;
                    row3x64 = mode == WF_SLAB && n_taps == 9 && kw == 3 && tbx == 3 && ksteps == 4 && dw == 1;
                    a_bytes = __ldg(&sp->a_bytes); b_bytes = __ldg(&sp->b_bytes);
                    a_sz = (a_bytes + 1023u) & ~1023u; b_sz = (b_bytes + 1023u) & ~1023u;
                    keep_bytes = (uint32_t)__ldg(&sp->keep_bytes);
                    cps = __ldg(&sp->cps);
                }
                if (kind == WF_CONV) {
                    const uint32_t buf = cnt & 1u;
                    if (!mbar_wait_abortable(acce0 + 8u * buf, ((cnt >> 1) & 1u) ^ 1u, abort_flag)) { fail = true; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    tr(item, 3);
                    const uint32_t acc = tmem_base + buf * 256u;
                    uint32_t accumulate = 0;
                    // (this thread issues every MMA of the CTA, some 60 cycles each whatever N up to 128, and every other
                    // instruction it executes is a bubble of the tensor pipe: addresses are ready before the waits, no
                    // division or modulo)
                    const bool kept = keep_bytes != 0;
                    const long long key = kept ? (((long long)map_base << 16) | rec_cout(cur)) + 1 : (mode == WF_SLAB ? -(long long)a_sz : 0);
                    if (key != cut_key) {                      // see the loader: the ring is cut anew
                        if (cut_key > 0) umma_commit(wempty);  // the MMAs so far were the kept weights' last users
                        cut_key = key;
                        ring_lim = ring_bytes - (key < 0 ? 2u * a_sz : keep_bytes);
                        pos = 0;
                        if (kept) {
                            if (!mbar_wait_abortable(wfull, w_uses & 1u, abort_flag)) { fail = true; break; }
                            ++w_uses;
                        }
                    }
                    uint32_t kept_at = ring0 + ring_lim;       // next kept weight box
                    // the next entry; its empty barrier goes to `eb`
                    uint32_t eb = 0;
                    auto next_place = [&](uint32_t size) -> uint32_t {
                        if (pos + size > ring_lim) pos = 0;
                        const uint32_t at = ring0 + pos;
                        eb = empty0 + 8u * (n_used & (WF_ENTRIES - 1));
                        ++n_used; pos += size;
                        return at;
                    };
                    // waits until the next entry / box group is loaded
                    auto next_full = [&]() {
                        if (!mbar_spin_abortable(full0 + 8u * (n_full & (WF_ENTRIES - 1)), (n_full / WF_ENTRIES) & 1u, abort_flag)) return false;
                        ++n_full;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        return true;
                    };
                    auto next_group = [&]() {
                        if (!mbar_spin_abortable(gfull0 + 8u * (n_group & (WF_GROUPS - 1)), (n_group / WF_GROUPS) & 1u, abort_flag)) return false;
                        ++n_group;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        return true;
                    };
                    if (row3x64 && !kept) {
                        // the common 3x3 chunk, its three weight boxes behind one barrier, two or three: nothing but the
                        // commits stands between the MMAs (the general loop below spends some 330 cycles of this thread's
                        // arithmetic per box, half of a box's MMAs: 3700 -> 2614 cycles per 64-channel chunk)
                        for (int ch = 0; ch < n_chunks; ++ch) {
                            const uint32_t la = desc_lo(ring0 + ring_lim + slab_sl * a_sz);
                            const uint32_t lb0 = desc_lo(next_place(b_sz)), e0 = eb, lb1 = desc_lo(next_place(b_sz)), e1 = eb, lb2 = desc_lo(next_place(b_sz)), e2 = eb;
                            slab_sl ^= 1u;
                            if (!next_group()) { fail = true; break; }
                            if (ch == 0) { tr(item, 13); tr(item, 14); }
                            mma_row3x64(acc, la, lb0, tap16, desc_hi, idesc, accumulate);
                            umma_commit(e0);
                            if (cps == 1 && !next_group()) { fail = true; break; }
                            mma_row3x64(acc, la + step_h16, lb1, tap16, desc_hi, idesc, accumulate);
                            umma_commit(e1);
                            if (cps < 3 && !next_group()) { fail = true; break; }
                            mma_row3x64(acc, la + 2u * step_h16, lb2, tap16, desc_hi, idesc, accumulate);
                            umma_commit(e2);
                        }
                    } else if (row3x64 && kept) {
                        // the same with the weights in place
                        const uint32_t b16 = b_sz >> 4;
                        for (int ch = 0; ch < n_chunks; ++ch, kept_at += 3u * b_sz) {
                            const uint32_t la = desc_lo(next_place(a_sz)), lb0 = desc_lo(kept_at);
                            if (!next_full()) { fail = true; break; }
                            if (ch == 0) { tr(item, 13); tr(item, 14); }
                            mma_row3x64(acc, la, lb0, tap16, desc_hi, idesc, accumulate);
                            mma_row3x64(acc, la + step_h16, lb0 + b16, tap16, desc_hi, idesc, accumulate);
                            mma_row3x64(acc, la + 2u * step_h16, lb0 + 2u * b16, tap16, desc_hi, idesc, accumulate);
                            umma_commit(eb);
                        }
                    } else if (mode == WF_SLAB) {
                        for (int ch = 0; ch < n_chunks && !fail; ++ch) {
                            uint32_t sa, a_empty = 0;
                            if (kept) {
                                sa = next_place(a_sz);
                                a_empty = eb;
                                if (!next_full()) { fail = true; break; }
                            } else {
                                if (!next_group()) { fail = true; break; }
                                sa = ring0 + ring_lim + slab_sl * a_sz;
                                slab_sl ^= 1u;
                            }
                            if (ch == 0) tr(item, 13);
                            // start field of the tap's activation operand: one pixel further per filter column, one slab row
                            // further per filter row (kept incrementally)
                            uint32_t la_row = desc_lo(sa), la = la_row;
                            int tb = 0, in_group = 0;                        // filter column of tap t0, boxes used of the group
                            for (int t0 = 0; t0 < n_taps; t0 += tbx) {
                                uint32_t sb = kept_at;
                                if (kept) {
                                    kept_at += b_sz;
                                } else {
                                    if (in_group == cps) {
                                        if (!next_group()) { fail = true; break; }
                                        in_group = 0;
                                    }
                                    ++in_group;
                                    sb = next_place(b_sz);
                                }
                                if (ch == 0 && t0 == 0) tr(item, 14);
                                uint32_t lb = desc_lo(sb);
                                const int t1 = min(t0 + tbx, n_taps);
                                for (int t = t0; t < t1; ++t, lb += tap16) {
                                    // tap (a, b): the same box, read (a*dh*P + b*dw) pixels further on
                                    mma_tap_f(acc, la, lb, desc_hi, idesc, ksteps, accumulate);
                                    la += step_w16;
                                    if (++tb == kw) { tb = 0; la_row += step_h16; la = la_row; }
                                }
                                if (!kept) umma_commit(eb);
                            }
                            if (kept) umma_commit(a_empty);
                        }
                    } else {
                        const uint32_t a16 = a_sz >> 4, b16 = b_sz >> 4;
                        uint32_t lbk = desc_lo(kept_at);
                        for (int left = n_chunks * n_taps; left > 0; left -= cps) {
                            const uint32_t g = (uint32_t)min(cps, left);
                            const uint32_t at = next_place(g * (kept ? a_sz : a_sz + b_sz));
                            uint32_t la = desc_lo(at), lb = kept ? lbk : desc_lo(at + g * a_sz);
                            if (!next_full()) { fail = true; break; }
                            if (left == n_chunks * n_taps) tr(item, 13);
                            if (ksteps == 4) {
                                mma_ksteps_f<4>(acc, la, lb, desc_hi, idesc, accumulate);
                                if (g > 1) mma_ksteps_f<4>(acc, la + a16, lb + b16, desc_hi, idesc, accumulate);
                                if (g > 2) mma_ksteps_f<4>(acc, la + 2u * a16, lb + 2u * b16, desc_hi, idesc, accumulate);
                                if (g > 3) mma_ksteps_f<4>(acc, la + 3u * a16, lb + 3u * b16, desc_hi, idesc, accumulate);
                            } else {
                                for (uint32_t u = 0; u < g; ++u, la += a16, lb += b16) mma_tap_f(acc, la, lb, desc_hi, idesc, ksteps, accumulate);
                            }
                            umma_commit(eb);
                            lbk += g * b16;
                        }
                    }
                    if (fail) break;
                    tr(item, 15);
                    umma_commit(accf0 + 8u * buf);
                    tr(item, 4);
                    ++cnt;
                }
                cur = nxt;
            }
            if (fail) {
                atomicOr(P.status, 0x2u);
                atomicExch(P.counters + 2, 1u);
                *abort_flag = 1;
            }
        }
    } else if (warp == 2) {
        if (elect_one()) {
            // ---------------- publisher ----------------
            // Makes finished items visible: the workers' stores happen before their barrier and the arrive that
            // this thread waits for, so its fence orders them before the release increment of the counter.
            int item = blockIdx.x;
            int4 cur = item < NI ? __ldg(&P.items[item]) : zero4;
            // A convolution's output units leave from here too, as bulk stores: this thread issues a unit's store as soon as
            // the workers have finished it, hands the unit back when it has been read out, and waits for the stores'
            // completion before the increment -- the workers are at the next tile by then.
            int sidx = -1, ctr_base = 0, kind = -1, out_map = -1, sub_log = 6, units_n = 0, oh_lo = 0, p_log = 0, tr_log = 0, tw_valid = 0, BN = 0;
            uint32_t rx_units = 0;                             // units of a tile that partial sums arrive in
            uint32_t uc = 0, k = 0;
            bool fail = false;
            for (; item < NI; item += G) {
                const int4 nxt = item + G < NI ? __ldg(&P.items[item + G]) : zero4;
                if (rec_stage(cur) != sidx) {
                    sidx = rec_stage(cur);
                    const WfStage *sp = &P.stages[sidx];
                    ctr_base = __ldg(&sp->ctr_base); kind = __ldg(&sp->kind); out_map = __ldg(&sp->out_map);
                    sub_log = __ldg(&sp->sub_log); oh_lo = __ldg(&sp->oh_lo); p_log = __ldg(&sp->p_log); tr_log = __ldg(&sp->tr_log);
                    tw_valid = __ldg(&sp->tw_valid); BN = __ldg(&sp->BN);
                    if (SPLIT) {
                        const int s_log = __ldg(&sp->s_log);
                        BN >>= s_log;                          // (the channels the item finishes)
                        rx_units = (1u << s_log) >> 1;
                    }
                    units_n = BN >> sub_log;
                }
                if (SPLIT && kind == WF_NONE) {
                    cur = nxt;
                    continue;
                }
                if (kind == WF_CONV && out_map >= 0) {
                    const int ow0 = rec_tw(cur) * tw_valid, oh0 = oh_lo + (rec_tr(cur) << tr_log), n0 = rec_tn(cur) * (128 >> (p_log + tr_log));
                    for (int u = 0; u < units_n; ++u) {
                        const uint32_t sl = (uc + u) & (WF_UNITS - 1);
                        if (!mbar_wait_abortable(uready0 + 8u * sl, ((uc + u) / WF_UNITS) & 1u, abort_flag)) { fail = true; break; }
                        tma_store_4d(P.maps + out_map, unit0 + sl * unit_bytes, rec_cout(cur) * BN + (u << sub_log), ow0, oh0, n0);
                        bulk_commit();
                        if (units_n > WF_UNITS) {              // more units than places: each goes back before the next is needed
                            bulk_wait_read();
                            mbar_arrive(ufree0 + 8u * sl);
                        }
                    }
                    bulk_wait_read();
                    if (fail) { fail = !*abort_flag; break; }
                    for (int u = 0; u < units_n && units_n <= WF_UNITS; ++u) mbar_arrive(ufree0 + 8u * ((uc + u) & (WF_UNITS - 1)));
                    uc += units_n + rx_units;
                    bulk_wait_all();
                    add_release(P.counters + ctr_base + rec_tr(cur));
                } else {
                    if (kind == WF_CONV) uc += units_n + rx_units; // stored, and handed back, by the workers
                    const uint32_t q = k % WF_PUBQ, round = k / WF_PUBQ;
                    if (!mbar_wait_abortable(pubf0 + 8u * q, round & 1u, abort_flag)) { fail = !*abort_flag; break; }
                    add_release(P.counters + ctr_base + rec_tr(cur));
                    mbar_arrive(pube0 + 8u * q);
                    ++k;
                }
                cur = nxt;
            }
            bulk_wait_all();
            if (fail) {
                atomicOr(P.status, 0x8u);
                atomicExch(P.counters + 2, 1u);
                *abort_flag = 1;
            }
        }
    } else if (FETCH && warp == WF_FIRST_WORKER + WF_WORKER_WARPS) {
        // ---------------- fetch warp: the chain input, host memory -> device, in list order ----------------
        const unsigned done_before = (run - 1u) * (unsigned)P.n_fetch;          // counters[3] never resets
        const uint8_t *src0 = static_cast<const uint8_t *>(P.fetch_src);
        uint8_t *dst0 = static_cast<uint8_t *>(P.fetch_dst);
        for (int j = blockIdx.x; j < P.n_fetch; j += G) {
            const int4 rec = __ldg(&P.fetch_items[j]);
            if (j >= P.fetch_window) {
                // the window keeps the link's queue short, so that early rows are not stuck behind late ones
                const unsigned target = done_before + (unsigned)(j - P.fetch_window + 1);
                int ok = 1;
                if (lane == 0) {
                    for (uint32_t i = 0; (int)(ld_acquire(P.counters + 3) - target) < 0; ++i) {
                        if (i >= P.spin_limit) { ok = 0; atomicOr(P.status, 0x20u); break; }
                        if ((i & 63u) == 63u && (ld_relaxed(P.counters + 2) != 0u || *abort_flag)) { ok = -1; break; }
                        __nanosleep(64);
                    }
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (ok <= 0) {
                    if (ok == 0 && lane == 0) {
                        atomicExch(P.counters + 2, 1u);
                        *abort_flag = 1;
                    }
                    break;
                }
            }
            const long long off = (long long)(((unsigned long long)(unsigned)rec.y << 32) | (unsigned)rec.x);
            if (lane == 0) tr(TRACE_FETCH0 + j, 0);
            fetch_bytes(src0 + off, dst0 + off, rec.z, lane);
            __syncwarp();
            if (lane == 0) {
                tr(TRACE_FETCH0 + j, 1);
                add_release(P.counters + rec.w);                   // the warp's stores, then the increments
                atomicAdd(P.counters + 3, 1u);                     // (the window orders nothing)
                tr(TRACE_FETCH0 + j, 2);
            }
        }
    } else {
        // ---------------- epilogue / SIMT warps ----------------
        const int tid = threadIdx.x - 32 * WF_FIRST_WORKER;
        const int g = warp & 3;                               // TMEM lane group this warp may read
        const int m = g * 32 + lane;                          // accumulator row = anchor of this thread
        const int cgrp = (warp - WF_FIRST_WORKER) >> 2;                     // which share of the tile's 16-column chunks is this warp's
        int item = blockIdx.x;
        int4 cur = item < NI ? __ldg(&P.items[item]) : zero4;
        // the dependency entry of this lane for the next item that has one to wait for here
        auto dep_of = [&](const int4 &rec) { return warp == WF_FIRST_WORKER && lane < rec_ndep(rec) ? __ldg(&P.deps[rec_dep0(rec) + lane]) : make_int2(0, 0); };
        int2 dep = dep_of(cur);
        int sidx = -1;
        uint32_t cnt = 0, done_items = 0, uc = 0;
        int sub_log = 6, units_n = 0;
        bool bulk_out = false;
        int kind = -1, p_log = 0, tr_log = 0, tw_valid = 0, act = 0, res_pos = 0;
        for (; item < NI; item += G) {
            // (the record one item ahead, not two as for the loader: registers)
            const int4 nxt = item + G < NI ? __ldg(&P.items[item + G]) : zero4;
            if (rec_stage(cur) != sidx) {
                sidx = rec_stage(cur);
                const WfStage *sp = &P.stages[sidx];
                kind = SPLIT && __ldg(&sp->s_log) > 0 ? (int)WF_SPLIT : __ldg(&sp->kind);
                p_log = __ldg(&sp->p_log); tr_log = __ldg(&sp->tr_log); tw_valid = __ldg(&sp->tw_valid);
                act = __ldg(&sp->act);
                res_pos = ldg_ptr<const void *>(&sp->res) ? __ldg(&sp->res_pos) : LOP_RES_NONE;
                sub_log = __ldg(&sp->sub_log); units_n = __ldg(&sp->BN) >> sub_log;
                bulk_out = __ldg(&sp->out_map) >= 0;
            }
            const int tile_r = rec_tr(cur);
            if (tid == 0) tr(item, 7);
            if (kind == WF_CONV) {
                const uint32_t buf = cnt & 1u;
                const int c = m & ((1 << p_log) - 1);
                const int r = (m >> p_log) & ((1 << tr_log) - 1);
                const bool staged = c < tw_valid;                      // the other anchors are the slab's halo gap
                // staged rows are packed: image, row, column below tw_valid (the box of a bulk load or store)
                const int srow = (((m >> (p_log + tr_log)) << tr_log) + r) * tw_valid + c;
                int fuse_pool = 0;
                void *yout = nullptr;
                if (!bulk_out) {
                    const WfStage *sp = &P.stages[sidx];
                    fuse_pool = __ldg(&sp->fuse_pool);
                    yout = ldg_ptr<void *>(reinterpret_cast<const void *const *>(&sp->y));
                    const int oh_hi = __ldg(&sp->oh_hi), Ho = __ldg(&sp->Ho), Wo = __ldg(&sp->Wo), Cout = __ldg(&sp->Cout);
                    const int pool_Ho = __ldg(&sp->pool_Ho), pool_Wo = __ldg(&sp->pool_Wo), co0 = rec_cout(cur) * (units_n << sub_log);
                    const int ow = rec_tw(cur) * tw_valid + c;
                    const int oh = __ldg(&sp->oh_lo) + (tile_r << tr_log) + r;
                    const int n = rec_tn(cur) * (128 >> (p_log + tr_log)) + (m >> (p_log + tr_log));
                    const bool valid = staged && ow < Wo && oh < oh_hi && n < __ldg(&sp->N);
                    if (cgrp == 0 && staged) row_pix[srow] = valid ? (((long long)n * Ho + oh) * Wo + ow) * Cout + co0 : -1LL;
                    if (fuse_pool && cgrp == 0 && !((r | c) & 1)) {
                        // top-left anchor of a 2x2 window: where its maximum goes, if the whole window is inside the stage
                        const int q = (((m >> (p_log + tr_log)) << (tr_log - 1)) + (r >> 1)) * ((1 << p_log) >> 1) + (c >> 1);
                        const bool ok = valid && c + 1 < tw_valid && ow + 1 < Wo && oh + 1 < oh_hi;
                        pool_pix[q] = ok ? (((long long)n * pool_Ho + (oh >> 1)) * pool_Wo + (ow >> 1)) * Cout + co0 : -1LL;
                    }
                }
                const float *t_scale = s_scale + 128 * buf, *t_shift = s_shift + 128 * buf;   // filled by warp 0 a tile ahead
                const uint32_t row_stride = 2u << sub_log;             // bytes of a staged row in a unit
                // position of a 16-byte chunk in a staged row: the swizzle of the unit's tensor maps (128, 64 or 32 bytes)
                const int swz = sub_log == 6 ? srow & 7 : (sub_log == 5 ? (srow >> 1) & 3 : (srow >> 2) & 1);
                if (!mbar_wait_abortable(ssf0 + 8u * buf, (cnt >> 1) & 1u, abort_flag)) *epi_fail = 1;
                if (!mbar_wait_abortable(accf0 + 8u * buf, (cnt >> 1) & 1u, abort_flag)) *epi_fail = 1;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (tid == 0) tr(item, 5);
                for (int u = 0; u < units_n; ++u) {
                    const uint32_t sl = (uc + u) & (WF_UNITS - 1);
                    // the unit is free, and the residual's rows are in it where the layer has one
                    if (!mbar_wait_abortable(ugrant0 + 8u * sl, ((uc + u) / WF_UNITS) & 1u, abort_flag)) *epi_fail = 1;
                    uint8_t *my_row = units + sl * unit_bytes + srow * row_stride;
                    const uint32_t acc = tmem_base + buf * 256u + ((uint32_t)(g * 32) << 16) + ((uint32_t)u << sub_log);
                    // the two warps of a TMEM lane group take alternate 16-column chunks
                    for (int j = 16 * cgrp; j < (1 << sub_log); j += 16 * COL_GROUPS) {
                        uint32_t rr[16];
                        tmem_ld16(acc + (uint32_t)j, rr);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        if (!staged) continue;
                        const int ct = (u << sub_log) + j;             // channel inside the tile
                        float v[16];
#pragma unroll
                        for (int i = 0; i < 16; i += 4) {                  // 16-byte broadcast reads of the tile's scale / shift
                            const float4 sc = *reinterpret_cast<const float4 *>(t_scale + ct + i);
                            const float4 sf = *reinterpret_cast<const float4 *>(t_shift + ct + i);
                            v[i] = fmaf(sc.x, __uint_as_float(rr[i]), sf.x);
                            v[i + 1] = fmaf(sc.y, __uint_as_float(rr[i + 1]), sf.y);
                            v[i + 2] = fmaf(sc.z, __uint_as_float(rr[i + 2]), sf.z);
                            v[i + 3] = fmaf(sc.w, __uint_as_float(rr[i + 3]), sf.w);
                        }
                        uint4 *c0p = reinterpret_cast<uint4 *>(my_row + (((j >> 3) ^ swz) << 4));
                        uint4 *c1p = reinterpret_cast<uint4 *>(my_row + ((((j >> 3) + 1) ^ swz) << 4));
                        float rv[16];
                        if (res_pos != LOP_RES_NONE) {
                            const uint4 q0 = *c0p, q1 = *c1p;
                            const uint32_t rw[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                rv[2 * i] = __uint_as_float(rw[i] << 16);
                                rv[2 * i + 1] = __uint_as_float(rw[i] & 0xFFFF0000u);
                            }
                        }
                        finish_n<SMOOTH ? 1 : 0>(v, rv, res_pos, act);
                        uint32_t o[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                            o[i] = *reinterpret_cast<const uint32_t *>(&h);
                        }
                        *c0p = make_uint4(o[0], o[1], o[2], o[3]);
                        *c1p = make_uint4(o[4], o[5], o[6], o[7]);
                    }
                    // this warp's part of the unit is done (the publisher stores a bulk unit; the phase advances for all)
                    if (bulk_out) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(uready0 + 8u * sl);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                if (tid == 0) tr(item, 11);
                epi_bar();                                             // accumulator drained, units complete
                if (tid == 0) {
                    mbar_arrive(acce0 + 8u * buf);
                    mbar_arrive(sse0 + 8u * buf);
                }
                ++cnt;
                if (!bulk_out && !*epi_fail) {
                    for (int u = 0; u < units_n; ++u) {
                        const uint8_t *unit = units + ((uc + u) & (WF_UNITS - 1)) * unit_bytes;
                        uint4 *y = static_cast<uint4 *>(yout) + (u << (sub_log - 3));
                        if (fuse_pool) pool_unit(unit, pool_pix, y, p_log, tr_log, tw_valid, sub_log, tid);
                        else copy_unit(unit, row_pix, y, (128 >> p_log) * tw_valid, sub_log, tid);
                    }
                    // This thread's writes to the units come before a bulk load of the next tile's residual into the same
                    // places.  (Not where the writes are: without the condition there a ConvNeXt block takes 44.3 us, 43.9 so.)
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                }
                if (tid == 0) tr(item, 12);
                dep = dep_of(nxt);
            } else {
                // an item of the worker warps alone: output rows of one image (or a depth-wise tile)
                if (!SPLIT || kind < WF_NONE) {
                    if (warp == WF_FIRST_WORKER && !wait_deps_warp(P, rec_dep0(cur), rec_ndep(cur), dep, run, lane, [] {}) && lane == 0) *epi_fail = 1;
                    epi_bar();
                }
                dep = dep_of(nxt);                                     // on its way while the item is worked on
                if (tid == 0) tr(item, 1);
                const int n = rec_tn(cur), oh_lo = __ldg(&P.stages[sidx].oh_lo), oh = oh_lo + tile_r;
                if (SPLIT && kind == WF_SPLIT) {
                    // (also when a wait has run out: no barrier stands between the word's last write, behind the item before, and
                    // this place, and warps that saw different values would meet at different barriers for good)
                    uc += split_item<SMOOTH>(&P.stages[sidx], cur, smem + (bars - base), unit0, unit_bytes, tmem_base + (cnt & 1u) * 256u, uc, cnt);
                    ++cnt;
                } else if ((SPLIT && kind == WF_NONE) || *epi_fail) {
                    // on to the barrier and the common exit below
                } else if (kind == WF_POOL) {
                    const int oh0 = oh_lo + (tile_r << tr_log);
                    if (__ldg(&P.stages[sidx].mode)) pool3_item(&P.stages[sidx], n, oh0, min(1 << tr_log, __ldg(&P.stages[sidx].oh_hi) - oh0), tid);
                    else pool_item(&P.stages[sidx], n, oh, tid);
                } else if (ROWOPS && kind == WF_DWCONV) {
                    dwconv_item(&P.stages[sidx], n, tile_r, rec_tw(cur), rec_cout(cur), tid, stg);
                } else if (ROWOPS && kind == WF_LAYERNORM) {
                    layernorm_item(&P.stages[sidx], n, oh, tid);
                } else if (ROWOPS && kind == WF_CONCAT) {
                    concat_item(&P.stages[sidx], n, oh, tid);
                } else {
                    gather_item(&P.stages[sidx], n, tile_r, tid, stg);
                }
            }
            if (kind != WF_CONV && tid == 0) tr(item, 12);
            epi_bar();                                                 // every worker's stores of this item are issued
            if (*epi_fail) {                                           // uniform: written only before a barrier
                if (tid == 0) {
                    atomicOr(P.status, 0x4u);
                    atomicExch(P.counters + 2, 1u);
                    *abort_flag = 1;
                }
                break;
            }
            const bool stored_here = kind == WF_CONV || (SPLIT && kind == WF_SPLIT) ? !bulk_out : !SPLIT || kind != WF_NONE;
            if (kind == WF_CONV) {
                if (stored_here && tid == 0)
                    for (int u = 0; u < units_n; ++u) mbar_arrive(ufree0 + 8u * ((uc + u) & (WF_UNITS - 1)));
                uc += units_n;
            }
            if (stored_here) {
                if (tid == 0) {
                    // hand the item to the publisher warp, which fences and increments the row group's counter while
                    // the workers go on; it may lag WF_PUBQ items behind
                    const uint32_t q = done_items % WF_PUBQ, round = done_items / WF_PUBQ;
                    if (!mbar_wait_abortable(pube0 + 8u * q, (round & 1u) ^ 1u, abort_flag)) *epi_fail = 1;
                    mbar_arrive(pubf0 + 8u * q);
                }
                ++done_items;
            }
            if (tid == 0) tr(item, 6);
            cur = nxt;
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // A CTA that gave up may have copies on their way into its shared memory (operands, residual rows, the other parts' partial
    // sums) or messages to other CTAs, and MMAs that read it.  Each takes microseconds: the memory is held for a hundred of them
    // before another block may have it.  (Not a wait for the barriers that would tell: keeping the loader's counts for it to the
    // end cost every run of a ResNet-50 0.3 to 0.6 %.)  Every role has ended: misc[1] changes now only by another CTA that gives
    // up, and a warp sees one value of it.
    if (misc[1]) {
        // (the cluster's other CTAs hear of it first: a role of theirs may wait for this CTA's part of a tile, and for nothing
        // else that would tell it.  Looks at the device-wide flag in those waits cost a ResNet-18 streamed one image 1.5 us.)
        if (SPLIT && threadIdx.x < (unsigned)P.cluster) st_cluster(map_to_cta(bars + BAR_MISC + 4u, threadIdx.x), 1u);
#pragma unroll 1
        for (int i = 0; i < 100; ++i) __nanosleep(1000);
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    if (threadIdx.x == 0 && blockIdx.x < 4) {
        tr(TRACE_ITEMS - 8 + (int)blockIdx.x, 2);
        trv(TRACE_ITEMS - 8 + (int)blockIdx.x, 5, (unsigned long long)clock64());
    }
    if (SPLIT) cluster_sync();                                 // no CTA's shared memory goes while another may write to it
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned done = atomicAdd(P.counters + 1, 1u);
        if (done == gridDim.x - 1) {                                  // last CTA out: this run is complete
            for (int f = 0; f < P.n_flags; ++f) P.counters[P.flag_base + f] = 0u;   // arrival flags of the next run
            atomicExch(P.counters + 1, 0u);
            __threadfence();
            atomicAdd(P.counters, 1u);
        }
    }
}

#ifdef LOP_WF_TRACE
static WfParams g_last_params;
#endif

}  // namespace

#ifdef LOP_WF_TRACE
extern "C" int lop_debug_last_stages(void *host, int max_stages)
{
    const int n = g_last_params.n_stages < max_stages ? g_last_params.n_stages : max_stages;
    if (cudaMemcpy(host, g_last_params.stages, (size_t)n * sizeof(WfStage), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    return n;
}
extern "C" int lop_debug_last_items(void *host, int max_items)
{
    const int n = g_last_params.n_items < max_items ? g_last_params.n_items : max_items;
    if (cudaMemcpy(host, g_last_params.items, (size_t)n * sizeof(int4), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    return n;
}
extern "C" int lop_debug_trace_copy(void *host, size_t bytes, int clear)
{
    if (bytes > sizeof(unsigned long long) * TRACE_ITEMS * 16) bytes = sizeof(unsigned long long) * TRACE_ITEMS * 16;
    if (clear) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_wf_trace) != cudaSuccess) return -1;
        return cudaMemset(p, 0, sizeof(unsigned long long) * TRACE_ITEMS * 16) == cudaSuccess ? 0 : -1;
    }
    return cudaMemcpyFromSymbol(host, g_wf_trace, bytes) == cudaSuccess ? 0 : -1;
}
#endif

size_t wavefront_smem_bytes(const WfParams &p)
{
    return 1024 + (size_t)p.ring_bytes + (size_t)WF_UNITS * p.unit_bytes + p.simt_bytes + WF_FIXED_SMEM;
}

namespace {

typedef void (*WfKernel)(const WfParams);
template <bool FETCH, bool SMOOTH>
WfKernel kernel_with(bool row_ops, bool split)
{
    if (row_ops) return split ? wavefront_kernel<FETCH, true, SMOOTH, true> : wavefront_kernel<FETCH, true, SMOOTH, false>;
    return split ? wavefront_kernel<FETCH, false, SMOOTH, true> : wavefront_kernel<FETCH, false, SMOOTH, false>;
}
WfKernel kernel_for(bool fetch, bool row_ops, bool smooth, bool split)
{
    if (fetch) return smooth ? kernel_with<true, true>(row_ops, split) : kernel_with<true, false>(row_ops, split);
    return smooth ? kernel_with<false, true>(row_ops, split) : kernel_with<false, false>(row_ops, split);
}
WfKernel kernel_for(const WfParams &p) { return kernel_for(p.n_fetch > 0, p.row_ops != 0, p.smooth != 0, p.cluster > 1); }
int threads_of(const WfParams &p) { return p.n_fetch > 0 ? WF_THREADS + 32 : WF_THREADS; }

}  // namespace

// How many CTAs of the kernel this device can hold at once (the kernel's dependency waits assume that every CTA of
// a launch is resident: a CTA that has not started cannot produce what a running one waits for).
cudaError_t wavefront_resident_ctas(const WfParams &p, int *ctas)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const size_t smem = wavefront_smem_bytes(p);
    WfKernel k = kernel_for(p);
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)) != cudaSuccess) return e;
    if (p.cluster > 1) {
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)p.cluster; attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(sms / p.cluster * p.cluster)); cfg.blockDim = dim3((unsigned)threads_of(p)); cfg.dynamicSmemBytes = smem;
        cfg.attrs = &attr; cfg.numAttrs = 1;
        int clusters = 0;
        if ((e = cudaOccupancyMaxActiveClusters(&clusters, k, &cfg)) != cudaSuccess) return e;
        *ctas = clusters * p.cluster;
        return cudaSuccess;
    }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads_of(p), smem);
    if (e != cudaSuccess) return e;
    *ctas = per_sm * sms;
    return cudaSuccess;
}

cudaError_t launch_wavefront(const WfParams &p, int grid, cudaStream_t s)
{
    const size_t smem = wavefront_smem_bytes(p);
    // the attribute is per device: set it once on each device a launch is made from
    static std::atomic<bool> configured[64];            // set after the (idempotent) attribute call: plans on several host threads may race here
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !configured[dev].load(std::memory_order_acquire)) {
        for (int k = 0; k < 16; ++k) {
            e = cudaFuncSetAttribute(kernel_for(k & 4, k & 2, k & 1, k & 8), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
            if (e != cudaSuccess) return e;
        }
        if (dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
    }
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
#ifdef LOP_WF_TRACE
    g_last_params = p;
#endif
    // A program that fetches much of its input does not begin early: its CTAs would take the SMs in the order in which the
    // previous launch leaves them, and a long transfer suffers from that more than the launch's two microseconds (up to 300 KB:
    // a VGG block streamed 33.5 us without, 31.9 begun early, a DenseNet layer 24.9 and 22.7; 0.8 MB: four images' VGG block
    // 66.2 and 69.9; 1.6 MB: a ConvNeXt block 105 and 131).  Nor do clusters of four, which need not find their places while
    // CTAs of another launch still hold some.
    const bool early = p.fetch_bytes <= 512 * 1024 && p.cluster <= 2;
    cudaLaunchAttribute attrs[2]{};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3((unsigned)threads_of(p)); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cfg.attrs = attrs;
    if (early) {
        attrs[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attrs[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (p.cluster > 1) {
        attrs[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attrs[cfg.numAttrs].val.clusterDim.x = (unsigned)p.cluster;
        attrs[cfg.numAttrs].val.clusterDim.y = attrs[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    return cudaLaunchKernelEx(&cfg, kernel_for(p), p);
}

}  // namespace lop
