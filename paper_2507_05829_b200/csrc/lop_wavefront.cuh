// The wavefront kernel: one persistent launch executes a whole list of (band, layer) stages.
//
// Sec. III-A / IV-B of the paper: the operations of later layers start as soon as the rows they
// depend on exist, without waiting for the whole earlier layer.  A *program* is the topologically
// ordered list of stages of one launch; every stage is cut into items (output tiles of a
// convolution, output rows of a pooling or patch-gather stage); resident CTAs take items
// round-robin in program order and an item waits -- with a bounded spin -- only for the producer
// row groups its receptive field touches.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace lop {

// WF_FETCH: rows of the chain input brought from host memory by the CTAs' fetch warps.  Such a stage has row-group
// counters like any producer but no items in the main list: its work is the program's fetch list.
// WF_DWCONV / WF_LAYERNORM / WF_CONCAT: the memory-bound operators, run by the worker warps like pooling.  A depth-wise
// item is 1 << tr_log output rows of one image, tw_valid columns wide and BN channels deep (its receptive window is staged
// in shared memory); a normalisation or concatenation item is one whole output row of one image; a gather or 3x3 pooling
// item is 1 << tr_log of them.
// WF_SPLIT is what the worker warps call a split tile of a WF_CONV stage.  WF_NONE: an item without work, in front of a split
// tile whose items have to start at a cluster's first CTA.
enum WfKind { WF_GATHER = 0, WF_CONV = 1, WF_POOL = 2, WF_FETCH = 3, WF_DWCONV = 4, WF_LAYERNORM = 5, WF_CONCAT = 6, WF_NONE = 7, WF_SPLIT = 8 };
// How a convolution stage feeds the tensor cores.
//   WF_SLAB  one activation box per channel chunk: the output tile's receptive window (tile plus halo),
//            laid out in shared memory as rows of P pixels; every filter tap is the same box read at a
//            shifted start address.  Weights arrive as boxes of several taps.
//   WF_TAP   one activation box and one weight box per (channel chunk, tap): pointwise layers, strided
//            windows and channel chunks narrower than 64.
enum WfMode { WF_SLAB = 0, WF_TAP = 1 };

// One (band, layer) stage: rows [oh_lo, oh_hi) of a bound operator.
struct WfStage {
    int kind, mode;
    int oh_lo, oh_hi;
    int ctr_base;             // counters[ctr_base + tile_r]: finished items of that row group
    // convolution tile: accumulator row m is the anchor at column m & (P-1), row (m >> p_log) & (TR-1),
    // image m >> (p_log + tr_log) of the tile; columns >= tw_valid are the slab's halo gap and are dropped
    int p_log, tr_log, tw_valid;
    int BN, BK, n_chunks, n_taps, tb;     // tb: taps per weight box
    int map_base;             // first of 5 tensor maps (4 activation parity classes + weights)
    int a_valid_mask;
    uint32_t a_bytes, b_bytes;            // bytes of one activation / weight box
    uint32_t idesc, layout_code, sbo_bytes, row_bytes;
    // the operator, with its tensors bound (a gathered stem appears as the pointwise convolution it runs as)
    int N, Hin, Win, Cin, Ho, Wo, Cout;
    int kh, kw, sh, sw, ph, pw, dh, dw;
    int act, res_pos;
    const void *x;            // main input, full-size NHWC tensor
    const void *res;          // residual tensor or nullptr
    const float *scale, *shift;
    void *y;                  // full-size output (of the pooling layer when fuse_pool is set)
    // fuse_pool: the convolution's only consumer is a 2x2 stride-2 max pooling; the tile's epilogue takes the
    // maximum of each 2x2 window of staged rows and writes the pooled tensor [N, pool_Ho, pool_Wo, Cout] instead
    int fuse_pool, pool_Ho, pool_Wo;
    // per-tap mode: `cps` consecutive (chunk, tap) steps share one ring entry and its barrier pair; slab mode: `cps` weight
    // boxes of a chunk (the first group with the chunk's activation box) share one full barrier
    int cps;
    const void *w_taps;       // depth-wise stage: the filters as [tap][channel] bf16
    // the tile's output leaves shared memory as `BN / sub` units of `sub` channels (64, 32 or 16)
    int sub_log;
    int out_map;              // tensor map of the output's rows below oh_hi (a unit is one bulk store), or -1: the workers store it
    int res_map;              // tensor map of the residual (a unit is one bulk load), or -1
    int keep_bytes;           // > 0: a tile's weights stay in shared memory (this many bytes at the ring's end) from tile to tile
    // A split tile (s_log > 0): 1 << s_log consecutive items on as many CTAs of a cluster, each of which sums its share of the
    // channel chunks (n_chunks of them) over all BN channels, hands the other CTAs their slices of the partial sums, and
    // finishes the slice of BN >> s_log channels that is its own.  An item's cout_tile counts slices.
    int s_log;
    int pad_[5];
};
static_assert(sizeof(WfStage) == 256, "WfStage layout");

// One item, 16 bytes: x = stage | cout_tile << 16, y = tile_w | tile_n << 16, z = tile_r | dep_count << 20,
// w = first entry of its dependency list.
struct WfParams {
    const WfStage *stages;
    const int4 *items;
    const CUtensorMap *maps;
    const int2 *deps;         // (counter index, completions expected per run); y < 0: an arrival flag, target -y
    unsigned *counters;       // [0] runs completed, [1] CTAs finished, [2] abort, [3] fetch entries finished, [4..] row-group counters,
                              // then n_flags band-arrival flags (set by the copy stream, cleared at run end)
    int flag_base, n_flags;
    unsigned *status;
    int n_stages, n_items;
    uint32_t ring_bytes;      // operand ring
    uint32_t unit_bytes;      // one of the WF_UNITS output units in flight between the workers and the bulk stores
    uint32_t simt_bytes;      // scratch of the gather and depth-wise items
    // In-kernel input transfer (Sec. IV-B transmission, done by the kernel itself): every CTA has one more warp that
    // walks this list round-robin; entry j copies z bytes at byte offset (x | y << 32) from fetch_src (host memory
    // the device can address) to fetch_dst and then increments counters[w].  At most fetch_window entries are in
    // flight at a time (counters[3] counts finished ones), so the rows arrive in list order at the link's rate.
    uint32_t spin_limit;      // polls of a row-group counter, an arrival flag or the fetch window before the kernel gives up
    const int4 *fetch_items;
    const void *fetch_src;
    void *fetch_dst;
    int n_fetch, fetch_window;
    long long fetch_bytes;    // of all entries
    int row_ops;              // the program has WF_DWCONV / WF_LAYERNORM / WF_CONCAT stages
    int cluster;              // CTAs per cluster (1, 2 or 4): the most parts a tile of the program is split in
    int smooth;               // a convolution of the program is activated by SiLU or GELU
};

#ifndef LOP_WF_WORKER_WARPS
#define LOP_WF_WORKER_WARPS 8
#endif
constexpr int WF_WORKER_WARPS = LOP_WF_WORKER_WARPS;      // epilogue / SIMT warps (a multiple of 4)
constexpr int WF_FIRST_WORKER = 3;                         // warps 0..2: loader, MMA issuer, publisher
constexpr int WF_THREADS = 32 * (WF_FIRST_WORKER + WF_WORKER_WARPS);
constexpr int WF_ENTRIES = 16;                             // operand ring entries in flight at most (a power of two)
constexpr int WF_GROUPS = 8;                               // slab mode: box groups in flight at most (a power of two)
constexpr int WF_UNITS = 4;                                // output units in flight (a power of two)
constexpr uint32_t WF_FIXED_SMEM = 4096;                  // barriers, scale / shift and pixel tables
constexpr uint32_t WF_SPLIT_BN = 64, WF_SPLIT_UNIT = 16 * 1024;     // channels of a split tile; bytes of an output unit that partial sums arrive in
constexpr int WF_PUBQ = 4;                                 // finished items the publisher may lag behind the workers
constexpr int WF_CTR_FIRST = 4;
constexpr int WF_MAX_DEPS = 4095;

size_t wavefront_smem_bytes(const WfParams &p);
cudaError_t launch_wavefront(const WfParams &p, int grid, cudaStream_t s);
cudaError_t wavefront_resident_ctas(const WfParams &p, int *ctas);
constexpr uint32_t WF_SPIN_LIMIT_DEFAULT = 1u << 22;

}  // namespace lop
