// Host side of the wavefront kernel: turns a list of (band, layer, row range) requests into a
// device-resident program (stages, item records, tensor maps, dependency lists, counters).
//
// Dependencies follow Sec. IV-B of the paper: a tile depends on a producer row group as soon as
// any row of that group lies inside the tile's receptive rows (for the residual: its own rows).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <map>
#include <numeric>
#include <vector>

#include "lop_internal.h"
#include "lop_kernels.cuh"
#include "lop_layerargs.h"
#include "lop_program.h"
#include "lop_rowops.cuh"
#include "lop_wavefront.cuh"

namespace lop {

struct Program {
    void *dev = nullptr;            // one allocation holding every table
    unsigned *counters = nullptr;
    WfParams params{};
    int grid = 0;
    int flag_base = 0, n_flags = 0;
    const lop_plan_t *owner = nullptr;  // the first plan: its wait limit applies to the launches
};

void program_destroy(Program *p)
{
    if (!p) return;
    if (p->dev) cudaFree(p->dev);
    delete p;
}

namespace {

#ifndef LOP_FETCH_ENTRY_BYTES
#define LOP_FETCH_ENTRY_BYTES 3072
#endif
#ifndef LOP_FETCH_WINDOW_BYTES
#define LOP_FETCH_WINDOW_BYTES (96 * 1024)
#endif
#ifndef LOP_FETCH_WINDOW_MAX_BYTES
#define LOP_FETCH_WINDOW_MAX_BYTES (256 * 1024)
#endif
// Bytes one ring entry of a per-tap stage aims at: the issuing thread pays for every entry with a wait and a commit, while
// two entries must fit the ring to keep the loads on their way, with a rest that is not wasted.  A ResNet-50 of batch 8 streamed:
// 420 us with 48 KB, 418 with 64, 420 with 72, 443 with 96; of batch 32, whose steps of 128 channels take 32 KB: 824, 795, 815, 859.
#ifndef LOP_ENTRY_BYTES
#define LOP_ENTRY_BYTES (64 * 1024)
#endif
#ifndef LOP_KEEP_BYTES
#define LOP_KEEP_BYTES (80 * 1024)
#endif
constexpr uint32_t A_BOX_MAX = 48u * 1024u;     // largest activation box of a slab stage: two of them and a weight box share the ring
constexpr uint32_t LOP_ROWOP_STAGING_BYTES = 64u * 1024u;    // largest receptive window a depth-wise item stages
constexpr uint32_t B_BOX_MAX = 48u * 1024u;     // largest weight box of several taps: a 3x3 filter row of 128 x 64 weights

int ilog2i(int v) { int l = 0; while ((1 << l) < v) ++l; return l; }
uint32_t round_up_u32(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

// Channels of one output unit of a tile bn channels wide: what a swizzled bulk store takes.
int unit_channels(int bn) { return bn % 64 == 0 ? 64 : (bn % 32 == 0 ? 32 : 16); }

// Tile geometry of one convolution stage.
struct Geom {
    int mode;
    int P, TR, TN;            // anchors: TN images x TR rows x P columns = 128
    int tw_valid;             // output columns per tile
    int RI;                   // rows of the activation box
    int BN, BK, tb, n_taps, n_chunks;
    uint32_t a_bytes, b_bytes;
};

// a: the convolution as its kernel sees it (a gathered stem already reduced to 1x1).
// even_tiles: tiles must hold whole 2x2 windows (rows and valid columns even, at least two rows).
// bulk_out: the tile's output leaves by bulk stores (the workers' own copy-out needs every unit of the tile in place).
// ring: bytes of the operand ring, of which a slab stage needs two activation boxes and a weight box.  n_cta: the program's CTAs.
Geom choose_geom(const ConvArgs &a, int rows, bool even_tiles, bool bulk_out, uint32_t ring, int n_cta)
{
    Geom g{};
    g.BK = a.Cin % 64 == 0 ? 64 : (a.Cin % 32 == 0 ? 32 : 16);
    g.BN = 16;
    for (int bn = 128; bn >= 16; bn -= 16)
        if (a.Cout % bn == 0 && (bulk_out || bn / unit_channels(bn) <= WF_UNITS)) { g.BN = bn; break; }
    g.n_taps = a.kh * a.kw;
    g.n_chunks = a.Cin / g.BK;
    const uint32_t row_bytes = (uint32_t)g.BK * 2u;
    const bool pointwise = a.kh == 1 && a.kw == 1;
    const int halo_w = (a.kw - 1) * a.dw, halo_h = (a.kh - 1) * a.dh;
    bool slab = false;
    if (!pointwise && a.sh == 1 && a.sw == 1 && g.BK == 64) {
        // pitch P: the split of 128 anchors into rows of P pixels that needs the fewest tiles, then the smallest box
        long long best_tiles = -1, best_box = 0;
        for (int P = 16; P <= 128; P <<= 1) {
            const int twv = P - halo_w, TR = 128 / P, RI = TR + halo_h;
            if (twv < 8 || RI > 256 || (even_tiles && (TR < 2 || (twv & 1)))) continue;
            const uint32_t box = (uint32_t)RI * P * row_bytes;
            if (box > A_BOX_MAX || 2u * box + (uint32_t)(a.kw * g.BN) * row_bytes > ring) continue;
            const long long tiles = (long long)((a.Wo + twv - 1) / twv) * ((rows + TR - 1) / TR);
            if (best_tiles < 0 || tiles < best_tiles || (tiles == best_tiles && box < best_box)) {
                best_tiles = tiles; best_box = box;
                g.P = P; g.TR = TR; g.TN = 1; g.tw_valid = twv; g.RI = RI;
                slab = true;
            }
        }
    }
    g.mode = slab ? WF_SLAB : WF_TAP;
    if (!slab) {
        // dense tile: the (TW, TR, TN) split of 128 pixels that needs the fewest tiles
        int nmax = 1;
        while (nmax * 2 <= a.N) nmax *= 2;
        long long best = -1;
        g.P = 128; g.TR = 1; g.TN = 1;
        for (int tw = 128; tw >= 1; tw >>= 1)
            for (int tr = 128 / tw; tr >= 1; tr >>= 1) {
                const int tn = 128 / (tw * tr);
                if (tn > nmax || (even_tiles && (tw < 2 || tr < 2))) continue;
                const long long tiles = (long long)((a.Wo + tw - 1) / tw) * ((rows + tr - 1) / tr) * ((a.N + tn - 1) / tn);
                if (best < 0 || tiles < best) { best = tiles; g.P = tw; g.TR = tr; g.TN = tn; }
            }
        g.tw_valid = g.P; g.RI = g.TR;
    }
    // Output channels per tile: the widest tile reads its activations once and its MMAs do the most work each, but a layer
    // with few of them leaves SMs idle.  A tile half as wide takes about 1 / 1.4 of the time (an MMA with N = 64 costs the
    // issuing thread 48 cycles, one with N = 128 65; the epilogue 1.5 and 2.2 us), so the width follows from the number of
    // rounds the layer's tiles take on 148 SMs.  Not below 64: an MMA with N = 32 costs as much as one with N = 64.
    const long long pixel_tiles = (long long)((a.Wo + g.tw_valid - 1) / g.tw_valid) * ((a.Ho + g.TR - 1) / g.TR) * ((a.N + g.TN - 1) / g.TN);
    auto rounds = [&](int bn) { return (pixel_tiles * (a.Cout / bn) + n_cta - 1) / n_cta; };
    while (g.BN > 64 && g.BN % 32 == 0 && rounds(g.BN / 2) < 1.4 * rounds(g.BN)) g.BN /= 2;
    if (a.k_split > 1) g.BN = (int)WF_SPLIT_BN;
    g.a_bytes = (uint32_t)g.RI * g.P * g.TN * row_bytes;
    // (a shifted tap reads up to halo_w pixels past the box, into whatever follows it in shared memory: those rows of the
    // accumulator are the dropped anchors of the halo gap)
    g.tb = 1;
    if (slab) {
        // whole filter rows where one fits a box, else as many taps as do
        const uint32_t tap_bytes = (uint32_t)g.BN * row_bytes;
        const int cap = std::max(1, (int)(B_BOX_MAX / tap_bytes)), nblk = (g.n_taps + cap - 1) / cap;
        g.tb = a.kw * tap_bytes <= B_BOX_MAX ? a.kw : (g.n_taps + nblk - 1) / nblk;
    }
    g.b_bytes = (uint32_t)g.tb * g.BN * row_bytes;
    return g;
}

struct MapSet { int seg, layer, P, RI, TN, BN, BK, tb, base; };

// Five tensor maps of a convolution stage: the activation seen through the (row parity, column parity)
// classes of its stride, and the weights as [tap][cout][cin].
int encode_maps(const ConvArgs &a, const Geom &g, CUtensorMap *out, int *valid_mask)
{
    TensorMapEncodeFn enc = tensor_map_encoder();
    if (!enc) return LOP_ECUDA;
    const CUtensorMapSwizzle swz = g.BK == 64 ? CU_TENSOR_MAP_SWIZZLE_128B
                                   : (g.BK == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    const cuuint32_t ones[4] = {1, 1, 1, 1};
    int mask = 0;
    for (int ph = 0; ph < a.sh; ++ph)
        for (int pw = 0; pw < a.sw; ++pw) {
            const int idx = ph * a.sw + pw;
            if (idx >= 4) continue;
            const long long Hp = (a.Hin - ph + a.sh - 1) / a.sh, Wp = (a.Win - pw + a.sw - 1) / a.sw;
            if (a.Hin - ph <= 0 || a.Win - pw <= 0 || Hp <= 0 || Wp <= 0) continue;
            const cuuint64_t dims[4] = {(cuuint64_t)a.x_run, (cuuint64_t)Wp, (cuuint64_t)Hp, (cuuint64_t)a.N};
            const cuuint64_t strides[3] = {(cuuint64_t)a.sw * a.x_pixel * 2, (cuuint64_t)(a.sh * a.x_row * 2), (cuuint64_t)(a.Hin * a.x_row * 2)};
            const cuuint32_t box[4] = {(cuuint32_t)g.BK, (cuuint32_t)g.P, (cuuint32_t)g.RI, (cuuint32_t)g.TN};
            void *basep = (void *)(static_cast<const char *>(a.x) + (ph * a.x_row + (long long)pw * a.x_pixel) * 2);
            if (enc(&out[idx], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, basep, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return LOP_ECUDA;
            mask |= 1 << idx;
        }
    if (!mask) return LOP_ECUDA;
    for (int i = 0; i < 4; ++i)
        if (!((mask >> i) & 1))
            for (int j = 0; j < 4; ++j)
                if ((mask >> j) & 1) { out[i] = out[j]; break; }
    const cuuint64_t taps = (cuuint64_t)a.kh * a.kw;
    const cuuint64_t wd[3] = {(cuuint64_t)a.Cin, (cuuint64_t)a.Cout, taps};
    const cuuint64_t ws[2] = {taps * a.Cin * 2, (cuuint64_t)a.Cin * 2};
    const cuuint32_t wb[3] = {(cuuint32_t)g.BK, (cuuint32_t)g.BN, (cuuint32_t)g.tb};
    if (enc(&out[4], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(a.w), wd, ws, wb, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return LOP_ECUDA;
    *valid_mask = mask;
    return LOP_OK;
}

// Rows below oh_hi of an output-shaped tensor, in boxes of one output unit: `sub` channels of a tile's packed rows.
int encode_rows_map(const ConvArgs &a, const void *tensor, int sub, int tw, int tr, int tn, CUtensorMap *out)
{
    TensorMapEncodeFn enc = tensor_map_encoder();
    if (!enc) return LOP_ECUDA;
    const CUtensorMapSwizzle swz = sub == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (sub == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    const cuuint32_t ones[4] = {1, 1, 1, 1};
    const cuuint64_t dims[4] = {(cuuint64_t)a.Cout, (cuuint64_t)a.Wo, (cuuint64_t)a.oh_hi, (cuuint64_t)a.N};
    const cuuint64_t strides[3] = {(cuuint64_t)a.Cout * 2, (cuuint64_t)a.Wo * a.Cout * 2, (cuuint64_t)a.Ho * a.Wo * a.Cout * 2};
    const cuuint32_t box[4] = {(cuuint32_t)sub, (cuuint32_t)tw, (cuuint32_t)tr, (cuuint32_t)tn};
    return enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(tensor), dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? LOP_OK : LOP_ECUDA;
}

// Bulk stores go to device memory; a result tensor in mapped host memory is stored by the workers.
bool in_device_memory(const void *p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) { cudaGetLastError(); return false; }
    return at.type == cudaMemoryTypeDevice;
}

// Layer i is a tensor-core convolution whose output is read by nothing but a 2x2 stride-2 unpadded max pooling
// right behind it: the persistent kernel can then pool inside the convolution's epilogue.
bool pool_fusable(const lop_plan_t *pl, int i)
{
    const int L = (int)pl->layers.size();
    if (i + 1 >= L) return false;
    const LayerInfo &c = pl->layers[i], &q = pl->layers[i + 1];
    if (c.l.op != LOP_CONV2D || c.kernel != K_CONV_TC || q.l.op != LOP_MAXPOOL2D || q.l.input_from != i) return false;
    if (q.l.kh != 2 || q.l.kw != 2 || q.l.sh != 2 || q.l.sw != 2 || q.l.ph != 0 || q.l.pw != 0) return false;
    for (int j = i + 2; j < L; ++j)
        if (pl->layers[j].l.input_from == i || pl->layers[j].l.residual_from == i) return false;
    return true;
}

}  // namespace

// Item shape of a depth-wise stage in the persistent kernel (rows, columns and channels of one tile).
static bool dw_tile(const lop_plan_t *pl, const LayerInfo &li, rowop::DwTile *t)
{
    const lop_layer &l = li.l;
    rowop::DwTile tmp;
    if (!li.dw_transposed) return false;
    return rowop::dw_choose_tile(l.kh, l.kw, l.sh, l.sw, l.dh, l.dw, pl->N, li.Ho, li.Wo, l.cin, LOP_ROWOP_STAGING_BYTES, 32 * WF_WORKER_WARPS,
                                 t ? t : &tmp);
}

bool program_folds_pool(const lop_plan_t *pl, int layer) { return pool_fusable(pl, layer); }

bool program_supported(const lop_plan_t *pl)
{
    if (pl->dtype != LOP_BF16) return false;
    for (const auto &li : pl->layers) {
        if (li.l.op == LOP_CONV2D && li.kernel != K_CONV_TC) return false;
        // the worker warps move these in 16-byte vectors of eight channels
        if (li.l.op == LOP_DWCONV2D && !dw_tile(pl, li, nullptr)) return false;
        if (li.l.op == LOP_LAYERNORM && (li.l.cin % 8 != 0 || li.l.cin > 1024)) return false;     // a lane keeps at most four vectors
        if (li.l.op == LOP_CONCAT && (li.l.cin % 8 != 0 || li.l.cout % 8 != 0)) return false;
        if (li.l.op == LOP_MAXPOOL2D && li.l.cin % 8 != 0) return false;
    }
    return true;
}

namespace {

// What a request reads: rows of tensors produced inside the program, and whether it touches the raw chain input
// (only plan 0 can: a later plan's "input" is the previous plan's last layer).
struct Need { int tensor, lo, hi; bool same_seg; };
struct Reads { Need need[3]; int n = 0; bool raw = false; };

struct Ctx {
    const std::vector<SegBind> &segs;
    std::vector<int> base;              // first tensor id of each plan; id base+layer, base+L = the stem's patches
    int raw = -1;                       // tensor id of the chain input when the program fetches it itself, else -1
    int tensor_id(int seg, int layer) const { return base[seg] + layer; }
    int patches_id(int seg) const { return base[seg] + (int)segs[seg].pl->layers.size(); }
    int input_id(int seg) const { return tensor_id(seg - 1, (int)segs[seg - 1].pl->layers.size() - 1); }
};

// A convolution's shortcut, a concatenation's second tensor: read at the rows that are computed.
bool has_second_input(const lop_layer &l)
{
    return (l.op == LOP_CONV2D || l.op == LOP_DWCONV2D || l.op == LOP_CONCAT) && l.residual_from != LOP_NO_RESIDUAL;
}

// Rows [o0, o1) of request rq: the tensors and rows they are computed from (Sec. IV-B: a dependency exists as soon as
// any part of a producer's output is used).
Reads reads_of(const Ctx &cx, const StageReq &rq, int o0, int o1)
{
    Reads r;
    const lop_plan_t *pl = cx.segs[rq.seg].pl;
    const LayerInfo &li = pl->layers[rq.layer];
    const lop_layer &l = li.l;
    auto window = [&](int &a_out, int &b_out) {
        long long a = (long long)o0 * l.sh - l.ph, b = (long long)(o1 - 1) * l.sh - l.ph + (long long)(l.kh - 1) * l.dh;
        a = std::max(a, 0LL); b = std::min(b, (long long)li.Hin - 1);
        a_out = (int)a; b_out = (int)b + 1;
        return a <= b;
    };
    int a = 0, b = 0;
    if (rq.fetch) return r;                                                   // reads host memory only
    if (rq.gather || (l.input_from == LOP_INPUT && !li.stem_gather)) {
        if (rq.seg == 0) {
            r.raw = true;
            if (cx.raw >= 0 && window(a, b)) r.need[r.n++] = Need{cx.raw, a, b, false};     // whichever band fetched them
        } else if (window(a, b)) r.need[r.n++] = Need{cx.input_id(rq.seg), a, b, false};
    } else if (li.stem_gather) {
        r.need[r.n++] = Need{cx.patches_id(rq.seg), o0, o1, true};            // the patches of exactly these rows
    } else if (window(a, b)) {
        r.need[r.n++] = Need{cx.tensor_id(rq.seg, l.input_from), a, b, true};
    }
    if (!rq.gather && has_second_input(l)) {
        if (l.residual_from >= 0) r.need[r.n++] = Need{cx.tensor_id(rq.seg, l.residual_from), o0, o1, true};
        else if (rq.seg == 0) {
            r.raw = true;
            if (cx.raw >= 0) r.need[r.n++] = Need{cx.raw, o0, o1, false};
        } else r.need[r.n++] = Need{cx.input_id(rq.seg), o0, o1, false};
    }
    return r;
}

// Puts the requests into ascending priority as far as dependencies allow (a stable topological order).
int order_requests(const Ctx &cx, std::vector<StageReq> &reqs, bool reuse)
{
    const size_t n = reqs.size();
    std::vector<int> produces(n);
    for (size_t i = 0; i < n; ++i)
        produces[i] = reqs[i].fetch ? cx.raw : (reqs[i].gather ? cx.patches_id(reqs[i].seg) : cx.tensor_id(reqs[i].seg, reqs[i].layer));
    bool sorted_already = true;
    for (size_t i = 1; i < n; ++i)
        if (reqs[i].prio < reqs[i - 1].prio) sorted_already = false;
    std::vector<std::vector<int>> users(n);
    std::vector<int> pending(n, 0), heap;
    for (size_t i = 0; i < n; ++i) {
        const Reads r = reads_of(cx, reqs[i], reqs[i].lo, reqs[i].hi);
        for (int q = 0; q < r.n; ++q)
            for (size_t j = 0; j < n; ++j) {
                if (j == i || produces[j] != r.need[q].tensor) continue;
                if (!reuse && r.need[q].same_seg && reqs[j].band != reqs[i].band) continue;
                if (std::max(r.need[q].lo, reqs[j].lo) >= std::min(r.need[q].hi, reqs[j].hi)) continue;
                users[j].push_back((int)i);
                ++pending[i];
                if (j > i) sorted_already = false;
            }
    }
    if (sorted_already) return LOP_OK;
    auto later = [&](int x, int y) { return reqs[x].prio != reqs[y].prio ? reqs[x].prio > reqs[y].prio : x > y; };
    for (size_t i = 0; i < n; ++i)
        if (!pending[i]) heap.push_back((int)i);
    std::make_heap(heap.begin(), heap.end(), later);
    std::vector<StageReq> out;
    while (!heap.empty()) {
        std::pop_heap(heap.begin(), heap.end(), later);
        const int i = heap.back();
        heap.pop_back();
        out.push_back(reqs[i]);
        for (int u : users[i])
            if (--pending[u] == 0) { heap.push_back(u); std::push_heap(heap.begin(), heap.end(), later); }
    }
    if (out.size() != n) { set_error("the stage requests depend on each other in a cycle"); return LOP_EINVAL; }
    reqs.swap(out);
    return LOP_OK;
}

// A row group of a stage: consecutive items that wait for the same producers and count as one dependency, its counter
// being counters[WF_CTR_FIRST + its index].
struct Unit {
    int first_item, items, first_dep, deps;
    double item_us, tail_us;      // a CTA's time for one item; from an item's end on its CTA to its result being visible
    double fetch_us;              // time on the host link (a fetch unit: no items), else 0
};

// Order in which the units' items are dealt out: that in which a model of the machine could start them.  Items go
// round-robin to the CTAs and each CTA takes its items in order, waiting for an item's unit to be ready; fetches queue
// on the host link.  A list of units in stage order (layer by layer, operation batching of Sec. IV-C) is right while
// every layer fills the machine; where the input is still arriving, or layers are too small to fill it, units of later
// layers over early rows have to come in between (the pipeline of Sec. IV-B). Dealing out, whenever
// a CTA is free, the ready unit with the longest chain of readers behind it does either: while the machine waits the
// order follows the rows down the layers, and once it is saturated it turns layer by layer by itself.
// arrival_us: expected arrival of each band a negative dependency names.  n_cta: how many CTAs there will be.
void schedule_units(const std::vector<Unit> &units, const std::vector<int2> &deps, const std::vector<double> *arrival_us, int n_cta, std::vector<int> &order)
{
    const int n = (int)units.size();
    // producer's last store -> consumer sees the counter: about 1 us, and a margin, because a unit dealt out too early makes
    // a CTA wait with everything behind it, one dealt out too late costs next to nothing (1 -> 4: a ResNet-50 of batch 32
    // 1091 -> 1063 us, a 1024x1024 stack streamed 314 -> 302)
    const double hop_us = 4.0;
    std::vector<int> pending(n, 0), start(n + 1, 0), users, heap;
    std::vector<double> ready(n, 0.0);
    for (int i = 0; i < n; ++i)
        for (int d = units[i].first_dep; d < units[i].first_dep + units[i].deps; ++d) {
            if (deps[d].x >= WF_CTR_FIRST) { ++start[deps[d].x - WF_CTR_FIRST + 1]; ++pending[i]; }
            else if (arrival_us && -1 - deps[d].x < (int)arrival_us->size()) ready[i] = std::max(ready[i], (*arrival_us)[-1 - deps[d].x]);
        }
    for (int i = 0; i < n; ++i) start[i + 1] += start[i];
    users.resize(start[n]);
    {
        std::vector<int> at(start.begin(), start.end() - 1);
        for (int i = 0; i < n; ++i)
            for (int d = units[i].first_dep; d < units[i].first_dep + units[i].deps; ++d)
                if (deps[d].x >= WF_CTR_FIRST) users[at[deps[d].x - WF_CTR_FIRST]++] = i;
    }
    // time from a unit's start to the end of the longest chain behind it (producers come before their readers in `units`)
    std::vector<double> path(n, 0.0);
    for (int i = n - 1; i >= 0; --i) {
        double behind = 0.0;
        for (int u = start[i]; u < start[i + 1]; ++u) behind = std::max(behind, path[users[u]]);
        path[i] = behind + hop_us + units[i].item_us + units[i].tail_us;
    }
    auto later = [&](int x, int y) { return ready[x] != ready[y] ? ready[x] > ready[y] : x > y; };
    auto shorter = [&](int x, int y) { return path[x] != path[y] ? path[x] < path[y] : x > y; };
    for (int i = 0; i < n; ++i)
        if (!pending[i]) heap.push_back(i);
    std::make_heap(heap.begin(), heap.end(), later);        // by the time they are ready
    std::vector<int> now;                                   // ready when the next CTA is free: longest chain first
    std::vector<double> cta_free(n_cta, 0.0);
    double link_free = 0.0;
    size_t rr = 0;                                          // items placed so far: the round-robin position
    order.clear();
    while (!heap.empty() || !now.empty()) {
        while (!heap.empty() && (now.empty() || ready[heap.front()] <= cta_free[rr % n_cta])) {
            now.push_back(heap.front());
            std::pop_heap(heap.begin(), heap.end(), later);
            heap.pop_back();
            std::push_heap(now.begin(), now.end(), shorter);
        }
        std::pop_heap(now.begin(), now.end(), shorter);
        const int i = now.back();
        now.pop_back();
        order.push_back(i);
        double fin = ready[i];
        if (units[i].items == 0) {
            link_free = std::max(link_free, fin) + units[i].fetch_us;
            fin = link_free + 3.0;                          // + the link's latency
        }
        for (int it = 0; it < units[i].items; ++it) {
            double &f = cta_free[rr++ % n_cta];
            f = std::max(f, ready[i]) + units[i].item_us;
            fin = std::max(fin, f + units[i].tail_us);
        }
        for (int u = start[i]; u < start[i + 1]; ++u) {
            ready[users[u]] = std::max(ready[users[u]], fin + hop_us);
            if (--pending[users[u]] == 0) { heap.push_back(users[u]); std::push_heap(heap.begin(), heap.end(), later); }
        }
    }
}

}  // namespace

int program_build(const std::vector<SegBind> &segs, std::vector<StageReq> reqs, Program **result, const std::vector<double> *arrival_us,
                  const void *fetch_src)
{
    *result = nullptr;
    if (segs.empty()) { set_error("program_build: no plan"); return LOP_EINVAL; }
    const bool reuse = (segs[0].pl->flags & LOP_FLAG_REUSE_HALO) != 0;
    Ctx cx{segs, {}};
    int n_tensors = 0;
    for (const SegBind &sb : segs) { cx.base.push_back(n_tensors); n_tensors += (int)sb.pl->layers.size() + 1; }
    for (const StageReq &rq : reqs)
        if (rq.fetch && rq.hi > rq.lo) cx.raw = n_tensors;
    if (cx.raw >= 0) {
        ++n_tensors;
        if (!fetch_src) { set_error("program_build: fetch requests without a source"); return LOP_EINVAL; }
        if ((reinterpret_cast<uintptr_t>(fetch_src) & 15) != (reinterpret_cast<uintptr_t>(segs[0].in) & 15) ||
            (reinterpret_cast<uintptr_t>(fetch_src) & 1)) {
            set_error("host input and staging tensor must agree in their address modulo 16");
            return LOP_EUNSUPPORTED;
        }
    }
    {
        std::vector<StageReq> live;
        for (const StageReq &rq : reqs)
            if (rq.hi > rq.lo) live.push_back(rq);
        reqs.swap(live);
    }
    int orc = order_requests(cx, reqs, reuse);
    if (orc != LOP_OK) return orc;

    std::vector<WfStage> stages;
    std::vector<int> stage_band, stage_rows_per_group;
    std::vector<int4> items, fetch_items;
    std::vector<CUtensorMap> maps;
    std::vector<MapSet> mapsets;
    std::vector<int2> deps;
    std::vector<std::vector<int>> by_tensor(n_tensors);   // stage indices per produced tensor
    std::vector<int> expected;                         // completions per row group, per stage
    std::vector<Unit> units;
    int n_ctr = WF_CTR_FIRST;
    bool uses_flags = false;
    uint32_t unit_bytes = 1024, stg_bytes = 0;
    // scratch of the SIMT items, and with it what the operand ring has at least
    // Rows of one gather or pooling item: an item's fixed cost (about 1.5 us: its dependencies, the loads' latency, the
    // hand-over) is shared by its rows, and the rows of a window are loaded fewer times, but the items have to go round 148
    // SMs.  A row costs about 1 us per 600 vectors of 16 bytes written (measured at 32 images of 112x230x24).  Where the
    // input is still arriving, larger items hold up the rows behind them: several rows only where there are many items
    // (a ResNet-50 of batch 8 streamed: 490 us so, 527 with four rows).
    bool arriving = cx.raw >= 0;
    for (const StageReq &rq : reqs) arriving = arriving || rq.wait_arrival;
    auto rows_per_item = [arriving](long long all, double row_us) {
        if (arriving) return all >= 8 * 148 ? 4 : (all >= 4 * 148 ? 2 : 1);
        int best = 1;
        auto time = [&](int r) { return (double)((all + 148LL * r - 1) / (148LL * r)) * (1.5 + row_us * r); };
        for (int r = 2; r <= 4; r *= 2)
            if (time(r) < time(best)) best = r;
        return best;
    };
    auto row_us = [](long long w, long long c) { return (double)(w * c / 8) / 600.0; };
    auto gather_scratch = [&](const lop_plan_t *pl, int layer, int *rows) {
        const GatherGeom g = gather_geom(pl, layer);
        *rows = rows_per_item((long long)g.N * g.Ho, row_us(g.Wo, g.Kcol));
        // the image rows they read are staged in shared memory when they fit, else read in place
        auto bytes = [&](int r) { return (long long)gather_rows_in(g, r) * gather_pitch(g) + 4 * g.kh * g.kw * g.C; };
        while (*rows > 1 && bytes(*rows) > 20 * 1024) *rows /= 2;
        return bytes(*rows) <= 48 * 1024 ? round_up_u32((uint32_t)bytes(*rows), 1024u) : 0u;
    };
    for (const StageReq &rq : reqs) {
        const lop_plan_t *pl = segs[rq.seg].pl;
        const LayerInfo &li = pl->layers[rq.layer];
        rowop::DwTile t{1, 1, 8};
        int gr = 1;
        if (rq.gather) stg_bytes = std::max(stg_bytes, gather_scratch(pl, rq.layer, &gr));
        else if (!rq.fetch && li.l.op == LOP_DWCONV2D && dw_tile(pl, li, &t))
            stg_bytes = std::max(stg_bytes, round_up_u32((uint32_t)rowop::dw_tile_bytes(li.l.kh, li.l.kw, li.l.sh, li.l.sw, li.l.dh, li.l.dw, t), 1024u));
    }
    // CTAs per cluster: as many as the most finely split tile has parts.  Clusters of four leave some SMs out (33 of them fit).
    int cluster = 1;
    for (const StageReq &rq : reqs)
        if (!rq.fetch && !rq.gather) cluster = std::max(cluster, segs[rq.seg].pl->layers[rq.layer].k_split);
    const int n_cta = cluster == 4 ? 132 : 148;
    if (cluster > 1) unit_bytes = std::max(unit_bytes, WF_SPLIT_UNIT);
    const uint32_t ring_least = (227u * 1024u - 1024u - WF_FIXED_SMEM - stg_bytes - WF_UNITS * 16u * 1024u) & ~1023u;
    std::vector<char> out_on_device(segs.size());
    for (size_t i = 0; i < segs.size(); ++i) out_on_device[i] = in_device_memory(segs[i].out);

    std::vector<char> consumed(reqs.size(), 0);            // pooling requests folded into their convolution's stage
    std::vector<int> prod_lo, prod_hi;                     // per stage: rows of the tensor it produces
    for (size_t ri = 0; ri < reqs.size(); ++ri) {
        const StageReq &rq = reqs[ri];
        if (consumed[ri]) continue;
        if (stages.size() >= 65535) { set_error("program has too many stages"); return LOP_EUNSUPPORTED; }
        lop_plan_t *pl = segs[rq.seg].pl;
        const void *in = segs[rq.seg].in;
        void *out = segs[rq.seg].out, *ws = segs[rq.seg].ws;
        char *wsb = static_cast<char *>(ws);
        const LayerInfo &li = pl->layers[rq.layer];
        const lop_layer &l = li.l;
        WfStage st{};
        st.oh_lo = rq.lo; st.oh_hi = rq.hi;
        const int rows = rq.hi - rq.lo;
        int group_rows = 1, tiles_r = rows, tiles_w = 1, tiles_n = pl->N, cout_tiles = 1;
        int produces = rq.fetch ? cx.raw : (rq.gather ? cx.patches_id(rq.seg) : cx.tensor_id(rq.seg, rq.layer));
        int out_lo = rq.lo, out_hi = rq.hi;                    // rows of the produced tensor
        double item_us = 4.0, tail_us = 0.5;                   // for the schedule (measured, microseconds)
        if (rq.fetch) {
            // a stage only in the book-keeping sense (row-group counters its readers wait for): its work goes to the
            // fetch list.  Entries of about 3 KB, whole rows: a warp has that much in flight at a time.
            const long long row_b = (long long)pl->W * pl->C * 2;
            st.kind = WF_FETCH;
            st.x = fetch_src; st.y = const_cast<void *>(in);
            st.N = pl->N; st.Hin = pl->H; st.Win = pl->W; st.Cin = pl->C;
            group_rows = (int)std::max(1LL, std::min<long long>(rows, LOP_FETCH_ENTRY_BYTES / row_b));
            tiles_r = (rows + group_rows - 1) / group_rows;
            if (row_b * group_rows > 0x7fffffffLL) { set_error("input rows too long to fetch"); return LOP_EUNSUPPORTED; }
        } else if (rq.gather) {
            st.kind = WF_GATHER;
            st.x = in; st.y = wsb + pl->col_off;
            const GatherGeom gg = gather_geom(pl, rq.layer);
            st.N = gg.N; st.Hin = gg.H; st.Win = gg.W; st.Cin = gg.C; st.Ho = gg.Ho; st.Wo = gg.Wo; st.Cout = gg.Kcol;
            st.kh = gg.kh; st.kw = gg.kw; st.sh = gg.sh; st.sw = gg.sw; st.ph = gg.ph; st.pw = gg.pw; st.dh = gg.dh; st.dw = gg.dw;
            st.mode = gather_scratch(pl, rq.layer, &group_rows) ? 0 : 1;
            st.tr_log = ilog2i(group_rows);
            item_us = 1.5 + group_rows * row_us(gg.Wo, gg.Kcol);
            tiles_r = (rows + group_rows - 1) / group_rows;
        } else if (l.op == LOP_MAXPOOL2D) {
            const PoolArgs a = pool_args(pl, rq.layer, in, out, ws, rq.lo, rq.hi);
            st.kind = WF_POOL;
            // 3x3 windows: several rows per item where they leave two items per SM (a window's rows are loaded fewer times, and
            // an item's fixed cost is shared); st.mode says which of the two pooling routines runs
            st.mode = a.kh == 3 && a.kw == 3 && a.dh == 1 && a.dw == 1;
            if (st.mode) group_rows = rows_per_item((long long)a.N * a.Ho, row_us(a.Wo, a.C));
            st.tr_log = ilog2i(group_rows);
            tiles_r = (rows + group_rows - 1) / group_rows;
            item_us = st.mode ? 1.5 + group_rows * row_us(a.Wo, a.C) : 3.4;
            st.x = a.x; st.y = a.y;
            st.N = a.N; st.Hin = a.Hin; st.Win = a.Win; st.Cin = a.C; st.Ho = a.Ho; st.Wo = a.Wo; st.Cout = a.C;
            st.kh = a.kh; st.kw = a.kw; st.sh = a.sh; st.sw = a.sw; st.ph = a.ph; st.pw = a.pw; st.dh = a.dh; st.dw = a.dw;
        } else if (l.op == LOP_DWCONV2D || l.op == LOP_LAYERNORM || l.op == LOP_CONCAT) {
            const ConvArgs a = conv_args(pl, rq.layer, in, out, ws, rq.lo, rq.hi);
            st.kind = l.op == LOP_DWCONV2D ? WF_DWCONV : (l.op == LOP_LAYERNORM ? WF_LAYERNORM : WF_CONCAT);
            st.x = a.x; st.res = a.res; st.scale = a.scale; st.shift = a.shift; st.y = a.y;
            st.N = a.N; st.Hin = a.Hin; st.Win = a.Win; st.Cin = a.Cin; st.Ho = a.Ho; st.Wo = a.Wo; st.Cout = a.Cout;
            st.kh = a.kh; st.kw = a.kw; st.sh = a.sh; st.sw = a.sw; st.ph = a.ph; st.pw = a.pw; st.dh = a.dh; st.dw = a.dw;
            st.act = a.act; st.res_pos = a.res_pos;
            if (l.op == LOP_DWCONV2D) {
                rowop::DwTile t{1, 1, 8};
                if (!dw_tile(pl, li, &t)) { set_error("layer %d: depth-wise window does not fit the staging tile", rq.layer); return LOP_EUNSUPPORTED; }
                st.BN = t.cc; st.tw_valid = t.tw; st.tr_log = ilog2i(t.R);
                st.w_taps = wsb + li.wpad_off;
                group_rows = t.R;
                tiles_r = (rows + t.R - 1) / t.R;
                tiles_w = (li.Wo + t.tw - 1) / t.tw;
                cout_tiles = l.cin / t.cc;
            }
        } else {
            const ConvArgs a = conv_args(pl, rq.layer, in, out, ws, rq.lo, rq.hi);
            // a 2x2 pooling that is this convolution's only reader, asked for exactly the rows this stage feeds it
            size_t rj = reqs.size();
            if (pool_fusable(pl, rq.layer))
                for (size_t k = 0; k < reqs.size(); ++k)
                    if (!consumed[k] && !reqs[k].gather && reqs[k].seg == rq.seg && reqs[k].band == rq.band &&
                        reqs[k].layer == rq.layer + 1 && rq.lo == 2 * reqs[k].lo && rq.hi == 2 * reqs[k].hi) { rj = k; break; }
            const bool fuse = rj < reqs.size();
            const bool bulk_out = !fuse && (rq.layer + 1 < (int)pl->layers.size() || out_on_device[rq.seg]);
            const Geom g = choose_geom(a, rows, fuse, bulk_out, ring_least, n_cta);
            st.kind = WF_CONV;
            st.mode = g.mode;
            st.x = a.x; st.res = a.res; st.scale = a.scale; st.shift = a.shift; st.y = a.y;
            st.N = a.N; st.Hin = a.Hin; st.Win = a.Win; st.Cin = a.Cin; st.Ho = a.Ho; st.Wo = a.Wo; st.Cout = a.Cout;
            st.kh = a.kh; st.kw = a.kw; st.sh = a.sh; st.sw = a.sw; st.ph = a.ph; st.pw = a.pw; st.dh = a.dh; st.dw = a.dw;
            st.act = a.act; st.res_pos = a.res_pos;
            int base = -1;
            for (const MapSet &m : mapsets)
                if (m.seg == rq.seg && m.layer == rq.layer && m.P == g.P && m.RI == g.RI && m.TN == g.TN && m.BN == g.BN && m.BK == g.BK &&
                    m.tb == g.tb)
                    base = m.base;
            CUtensorMap cm[5];
            int mask = 0;
            const int rc = encode_maps(a, g, cm, &mask);            // also tells which parity classes exist
            if (rc != LOP_OK) { set_error("layer %d: tensor-map encoding failed", rq.layer); return rc; }
            if (base < 0) {
                base = (int)maps.size();
                for (int i = 0; i < 5; ++i) maps.push_back(cm[i]);
                mapsets.push_back(MapSet{rq.seg, rq.layer, g.P, g.RI, g.TN, g.BN, g.BK, g.tb, base});
            }
            st.map_base = base;
            st.a_valid_mask = mask;
            st.p_log = ilog2i(g.P); st.tr_log = ilog2i(g.TR); st.tw_valid = g.tw_valid;
            st.BN = g.BN; st.BK = g.BK; st.n_chunks = g.n_chunks; st.n_taps = g.n_taps; st.tb = g.tb;
            st.a_bytes = g.a_bytes; st.b_bytes = g.b_bytes;
            st.row_bytes = (uint32_t)g.BK * 2u;
            st.layout_code = g.BK == 64 ? 2u : (g.BK == 32 ? 4u : 6u);
            st.sbo_bytes = 8u * st.row_bytes;
            // instruction descriptor: fp32 accumulate, bf16 x bf16, both operands K-major, N = BN, M = 128
            st.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.BN >> 3) << 17) | ((128u >> 4) << 24);
            // a split tile's items: each walks its share of the chunks and finishes its slice of the channels
            st.s_log = ilog2i(a.k_split);
            st.n_chunks = g.n_chunks >> st.s_log;
            const int out_channels = g.BN >> st.s_log;
            const int sub = unit_channels(out_channels);
            st.sub_log = ilog2i(sub);
            unit_bytes = std::max(unit_bytes, round_up_u32((uint32_t)((128 >> st.p_log) * g.tw_valid * sub * 2), 1024u));
            st.out_map = st.res_map = -1;
            CUtensorMap rm;
            if (a.res) {
                if (encode_rows_map(a, a.res, sub, g.tw_valid, g.TR, g.TN, &rm) != LOP_OK) { set_error("layer %d: residual map encoding failed", rq.layer); return LOP_ECUDA; }
                st.res_map = (int)maps.size();
                maps.push_back(rm);
            }
            if (bulk_out) {
                if (encode_rows_map(a, a.y, sub, g.tw_valid, g.TR, g.TN, &rm) != LOP_OK) { set_error("layer %d: output map encoding failed", rq.layer); return LOP_ECUDA; }
                st.out_map = (int)maps.size();
                maps.push_back(rm);
            }
            if (fuse) {
                const LayerInfo &pool = pl->layers[rq.layer + 1];
                consumed[rj] = 1;
                st.fuse_pool = 1; st.pool_Ho = pool.Ho; st.pool_Wo = pool.Wo;
                st.y = const_cast<void *>(tensor_of(pl, rq.layer + 1, in, out, ws));
                produces = cx.tensor_id(rq.seg, rq.layer + 1);
                out_lo = reqs[rj].lo; out_hi = reqs[rj].hi;
            }
            // an MMA costs the issuing thread 0.05 to 0.09 us with its share of the waits, the epilogue runs beside the next tile's
            item_us = std::max(g.BN > 64 ? 2.2 : 1.5, 0.6 + 0.07 * st.n_chunks * g.n_taps * (g.BK / 16)) + (st.s_log ? 0.9 : 0.0);
            tail_us = 3.0;
            group_rows = g.TR;
            tiles_r = (rows + g.TR - 1) / g.TR;
            tiles_w = (a.Wo + g.tw_valid - 1) / g.tw_valid;
            tiles_n = (a.N + g.TN - 1) / g.TN;
            cout_tiles = a.Cout / out_channels;
        }
        if (tiles_w > 65535 || tiles_n > 65535 || cout_tiles > 65535 || tiles_r >= (1 << 20)) {
            set_error("layer %d: too many tiles for one stage", rq.layer);
            return LOP_EUNSUPPORTED;
        }
        st.ctr_base = n_ctr;
        n_ctr += tiles_r;
        const int exp_here = tiles_w * tiles_n * cout_tiles;
        const int sidx = (int)stages.size();

        // ---- dependencies of every row group of this stage on earlier stages of this program
        for (int tr = 0; tr < tiles_r; ++tr) {
            const int o0 = rq.lo + tr * group_rows, o1 = std::min(o0 + group_rows, rq.hi);
            const Reads rd = reads_of(cx, rq, o0, o1);
            const int first = (int)deps.size();
            if (rq.wait_arrival && rd.raw) {
                // every band whose transfer brings rows these output rows read (a request may span several bands where
                // thin bands were joined); no assumption is made about the order in which arrivals become visible
                long long a = (long long)o0 * l.sh - l.ph, b = (long long)(o1 - 1) * l.sh - l.ph + (long long)(l.kh - 1) * l.dh + 1;
                const bool main_raw = rq.gather || (l.input_from == LOP_INPUT && !li.stem_gather);
                if (!main_raw) { a = o0; b = o1; }                          // only the residual reads the chain input: its own rows
                else if (!rq.gather && has_second_input(l) && l.residual_from == LOP_INPUT) { a = std::min<long long>(a, o0); b = std::max<long long>(b, o1); }
                a = std::max(a, 0LL); b = std::min<long long>(b, pl->H);
                int last_leader = -1;
                for (int b2 = 0; b2 < pl->n_bands; ++b2) {
                    const lop_range &o = pl->in_need[b2];
                    if (o.out_hi <= o.new_lo || o.out_hi <= a || o.new_lo >= b) continue;
                    // the bands of one copy arrive together: the flag of the copy's last band stands for all of them
                    const int leader = std::min(pl->n_bands - 1, (b2 / pl->copy_group) * pl->copy_group + pl->copy_group - 1);
                    if (leader == last_leader) continue;
                    last_leader = leader;
                    deps.push_back(make_int2(-1 - leader, -1));         // patched below
                }
                uses_flags = true;
            }
            for (int q = 0; q < rd.n; ++q)
                for (int ps : by_tensor[rd.need[q].tensor]) {
                    if (!reuse && rd.need[q].same_seg && stage_band[ps] != rq.band) continue;
                    const WfStage &p = stages[ps];
                    const int lo = std::max(rd.need[q].lo, prod_lo[ps]), hi = std::min(rd.need[q].hi, prod_hi[ps]);
                    if (lo >= hi) continue;
                    const int gr = stage_rows_per_group[ps];
                    for (int g = (lo - prod_lo[ps]) / gr; g <= (hi - 1 - prod_lo[ps]) / gr; ++g)
                        deps.push_back(make_int2(p.ctr_base + g, expected[ps]));
                }
            const int count = (int)deps.size() - first;
            if (count > WF_MAX_DEPS) { set_error("layer %d: a tile depends on too many row groups", rq.layer); return LOP_EUNSUPPORTED; }
            units.push_back(Unit{(int)items.size(), rq.fetch ? 0 : exp_here, first, count, item_us, tail_us, 0.0});
            if (rq.fetch) {
                const long long row_b = (long long)pl->W * pl->C * 2;
                units.back().fetch_us = (double)(o1 - o0) * row_b * pl->N / 48e3;      // ~48 GB/s measured for SM-issued reads
                for (int n = 0; n < pl->N; ++n) {
                    const unsigned long long off = (unsigned long long)(((long long)n * pl->H + o0) * row_b);
                    fetch_items.push_back(make_int4((int)(unsigned)(off & 0xffffffffu), (int)(unsigned)(off >> 32), (int)((o1 - o0) * row_b),
                                                    st.ctr_base + tr));
                }
                continue;
            }
            for (int tn = 0; tn < tiles_n; ++tn)
                for (int tw = 0; tw < tiles_w; ++tw)
                    for (int ct = 0; ct < cout_tiles; ++ct)
                        items.push_back(make_int4(sidx | (ct << 16), tw | (tn << 16), tr | (count << 20), first));
        }
        by_tensor[produces].push_back(sidx);
        stages.push_back(st);
        stage_band.push_back(rq.band);
        stage_rows_per_group.push_back(st.fuse_pool ? group_rows / 2 : group_rows);    // in rows of the produced tensor
        prod_lo.push_back(out_lo);
        prod_hi.push_back(out_hi);
        expected.push_back(exp_here);
    }

    if (arrival_us || cx.raw >= 0) {
        std::vector<int> order;
        schedule_units(units, deps, arrival_us, n_cta, order);
        if (order.size() != units.size()) { set_error("the stages depend on each other in a cycle"); return LOP_EINVAL; }
        std::vector<int4> dealt;
        dealt.reserve(items.size());
        for (int u : order) dealt.insert(dealt.end(), items.begin() + units[u].first_item, items.begin() + units[u].first_item + units[u].items);
        items.swap(dealt);
    }
    if (cluster > 1) {
        // a split tile's items start at the first CTA of its part of a cluster: items without work fill what is missing
        std::vector<int4> placed;
        placed.reserve(items.size() + items.size() / 8);
        for (size_t i = 0; i < items.size();) {
            const size_t parts = (size_t)1 << stages[items[i].x & 0xFFFF].s_log;
            while (placed.size() % parts) placed.push_back(make_int4((int)stages.size(), 0, 0, 0));
            for (size_t e = i + parts; i < e; ++i) placed.push_back(items[i]);
        }
        items.swap(placed);
        if (stages.size() >= 65535) { set_error("program has too many stages"); return LOP_EUNSUPPORTED; }
        WfStage none{};
        none.kind = WF_NONE;
        none.kh = none.kw = none.sh = none.sw = none.tb = 1;
        stages.push_back(none);
    }
    lop_plan_t *pl0 = segs[0].pl;
    Program *p = new (std::nothrow) Program();
    if (!p) { set_error("out of host memory"); return LOP_ENOMEM; }
    if (uses_flags) {                                        // arrival flags live after the row-group counters
        p->flag_base = n_ctr;
        p->n_flags = pl0->n_bands;
        for (int2 &d : deps)
            if (d.x < 0) d.x = p->flag_base + (-1 - d.x);
        n_ctr += p->n_flags;
    }
    const int n_items = (int)items.size();
    if (n_items == 0 && fetch_items.empty()) { *result = p; return LOP_OK; }          // nothing to do: an empty program

    std::map<int, long long> tiles_of;                            // convolution tiles per weight map: the layer's stages together
    for (const int4 &it : items)
        if (stages[it.x & 0xFFFF].kind == WF_CONV) ++tiles_of[stages[it.x & 0xFFFF].map_base];
    // ---- shared memory: the operand ring takes what the output units and the SIMT scratch leave.  Without a convolution
    // there is none: what is not asked for stays L1, which the loads of the memory-bound items go through (8x224x224x64 with
    // the whole of it asked for and without: depth-wise 7x7 289 and 238 us, normalisation 115 and 98, concatenation 260 and 222).
    const uint32_t ring_bytes = tiles_of.empty() ? 0u : (227u * 1024u - 1024u - WF_FIXED_SMEM - stg_bytes - WF_UNITS * unit_bytes) & ~1023u;
    auto slot = [](uint32_t bytes) { return round_up_u32(bytes, 1024u); };
    std::map<uint32_t, uint32_t> box_step;                        // slab stages that share a cut of the ring: divisor of their weight boxes
    for (WfStage &st : stages) {
        if (st.kind != WF_CONV) continue;
        const uint32_t a_sz = slot(st.a_bytes), b_sz = slot(st.b_bytes);
        // Weights stay in shared memory from tile to tile where every CTA gets at least two tiles of the layer, always of
        // the same output channels (items go round-robin), and they leave room for two activation boxes and a full entry (a
        // ResNet-50 of four 640x1152 images, whose gather leaves the ring 112 KB: 1602 us so, 1611 with 64 KB of weights kept
        // beside entries of two boxes).
        const uint32_t boxes = (uint32_t)st.n_chunks * ((st.n_taps + st.tb - 1) / st.tb);
        const uint32_t beside = std::max(2u * a_sz, st.mode == WF_TAP ? LOP_ENTRY_BYTES / a_sz * a_sz : 0u);
        const int cout_tiles = st.Cout / st.BN;
        if (st.s_log == 0 && boxes * b_sz <= LOP_KEEP_BYTES && boxes * b_sz + beside <= ring_bytes && n_cta % cout_tiles == 0 && tiles_of[st.map_base] >= 2 * n_cta)
            st.keep_bytes = (int)(boxes * b_sz);
        if (2u * a_sz + b_sz > ring_bytes) { delete p; set_error("tile buffers do not fit shared memory"); return LOP_EUNSUPPORTED; }
        if (st.mode == WF_SLAB && !st.keep_bytes) box_step[a_sz] = std::gcd(box_step[a_sz], b_sz);
    }
    for (WfStage &st : stages) {
        st.cps = 1;
        if (st.kind != WF_CONV) continue;
        const uint32_t a_sz = slot(st.a_bytes), b_sz = slot(st.b_bytes);
        // what the stage's entries share: the ring without the kept weights, or without a slab stage's activation boxes
        const uint32_t lim = ring_bytes - (st.keep_bytes ? (uint32_t)st.keep_bytes : (st.mode == WF_SLAB ? 2u * a_sz : 0u));
        if (st.mode == WF_SLAB && !st.keep_bytes) {
            // weight boxes per full barrier: the issuing thread stalls at every wait, so it waits once per chunk where the
            // chunk's weights fit the ring with room for part of the next chunk's
            const int per_chunk = (st.n_taps + st.tb - 1) / st.tb;
            const uint32_t most = std::max(b_sz, lim * 7u / 10u);
            const int groups = (int)((per_chunk * b_sz + most - 1) / most);
            st.cps = std::min({(per_chunk + groups - 1) / groups, (int)(most / b_sz), WF_ENTRIES});
            // The loader places a group's boxes before any of them can be consumed.  A box does not straddle the ring's end,
            // and boxes start at multiples of the divisor of all sizes in this cut: what is skipped there and the group
            // have to fit together.
            while (st.cps > 1 && (st.cps + 1) * b_sz - box_step[a_sz] > lim) --st.cps;
        }
        if (st.mode == WF_TAP) {
            const uint32_t step = st.keep_bytes ? a_sz : a_sz + b_sz;
            st.cps = (int)std::max(1u, std::min<uint32_t>(LOP_ENTRY_BYTES, lim) / step);
        }
        // (an entry larger than its ring would be waited for in vain)
        const uint32_t entry = st.keep_bytes ? (st.mode == WF_TAP ? (uint32_t)st.cps * a_sz : a_sz)
                                             : (uint32_t)st.cps * (st.mode == WF_TAP ? a_sz + b_sz : b_sz);
        if (entry > lim) { delete p; set_error("an operand ring entry of %u bytes does not fit %u", entry, lim); return LOP_EUNSUPPORTED; }
    }

#ifdef LOP_WF_TRACE
    fprintf(stderr, "program: %zu stages, %d items, ring %u B, units %u B, scratch %u B\n", stages.size(), n_items, ring_bytes, unit_bytes, stg_bytes);
#endif
    // ---- one device allocation for all tables
    auto al = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t o_stages = 0;
    const size_t o_items = o_stages + al(stages.size() * sizeof(WfStage));
    const size_t o_maps = o_items + al(items.size() * sizeof(int4));
    const size_t o_deps = o_maps + al(std::max<size_t>(maps.size(), 1) * sizeof(CUtensorMap));
    const size_t o_fetch = o_deps + al(std::max<size_t>(deps.size(), 1) * sizeof(int2));
    const size_t o_ctr = o_fetch + al(fetch_items.size() * sizeof(int4));
    const size_t total = o_ctr + al((size_t)n_ctr * sizeof(unsigned));
    cudaError_t e = cudaMalloc(&p->dev, total);
    if (e != cudaSuccess) { delete p; set_error("cudaMalloc(%zu) failed: %s", total, cudaGetErrorString(e)); return LOP_ECUDA; }
    char *d = static_cast<char *>(p->dev);
    auto up = [&](size_t off, const void *src, size_t bytes) {
        return bytes ? cudaMemcpy(d + off, src, bytes, cudaMemcpyHostToDevice) : cudaSuccess;
    };
    if ((e = cudaMemset(d, 0, total)) != cudaSuccess || (e = up(o_stages, stages.data(), stages.size() * sizeof(WfStage))) != cudaSuccess ||
        (e = up(o_items, items.data(), items.size() * sizeof(int4))) != cudaSuccess ||
        (e = up(o_maps, maps.data(), maps.size() * sizeof(CUtensorMap))) != cudaSuccess ||
        (e = up(o_deps, deps.data(), deps.size() * sizeof(int2))) != cudaSuccess ||
        (e = up(o_fetch, fetch_items.data(), fetch_items.size() * sizeof(int4))) != cudaSuccess) {
        program_destroy(p);
        set_error("program upload failed: %s", cudaGetErrorString(e));
        return LOP_ECUDA;
    }
    p->counters = reinterpret_cast<unsigned *>(d + o_ctr);
    WfParams &P = p->params;
    P.stages = reinterpret_cast<const WfStage *>(d + o_stages);
    P.items = reinterpret_cast<const int4 *>(d + o_items);
    P.maps = reinterpret_cast<const CUtensorMap *>(d + o_maps);
    P.deps = reinterpret_cast<const int2 *>(d + o_deps);
    P.counters = p->counters;
    P.status = reinterpret_cast<unsigned *>(static_cast<char *>(segs[0].ws) + pl0->status_off);
    P.flag_base = p->flag_base; P.n_flags = p->n_flags;
    P.n_stages = (int)stages.size();
    P.n_items = n_items;
    P.ring_bytes = ring_bytes; P.unit_bytes = unit_bytes; P.simt_bytes = stg_bytes;
    P.fetch_items = reinterpret_cast<const int4 *>(d + o_fetch);
    P.fetch_src = fetch_src;
    P.fetch_dst = const_cast<void *>(segs[0].in);
    P.n_fetch = (int)fetch_items.size();
    P.cluster = cluster;
    P.row_ops = P.smooth = 0;
    for (const WfStage &st : stages)
        if (st.kind == WF_DWCONV || st.kind == WF_LAYERNORM || st.kind == WF_CONCAT) P.row_ops = 1;
        else if (st.kind == WF_CONV && (st.act == LOP_ACT_SILU || st.act == LOP_ACT_GELU)) P.smooth = 1;
    // entries in flight: about the link's bandwidth-delay product (some 25 GB/s x 3 us), at least a few warps' worth
    long long bytes = 0;
    for (const int4 &f : fetch_items) bytes += f.z;
    P.fetch_bytes = bytes;
    if (P.n_fetch > 0) {
        // (a small input keeps the short window, which keeps its few bands in order; an input of megabytes is bound by
        // the link's rate, which needs more bytes on their way: measured 597 -> 577 us on a 2.4 MB batch)
        const long long window_bytes = std::min<long long>(LOP_FETCH_WINDOW_MAX_BYTES, std::max<long long>(LOP_FETCH_WINDOW_BYTES, bytes / 8));
        P.fetch_window = (int)std::max(8LL, window_bytes * P.n_fetch / std::max(1LL, bytes));
    }
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    p->owner = pl0;
    p->grid = n_items > 0 ? std::min(n_items, sms) : std::min((int)fetch_items.size(), sms);   // (a fetch-only program: its fetch warps)
    // every CTA of a launch must be resident (see the kernel's deadlock-freedom argument); what the device can hold
    // with this kernel's shared memory and registers says whether that is possible at all -- whether the SMs are free
    // at launch time is the caller's business: the stream must have the GPU to itself while the kernel runs
    int resident = 0;
    e = wavefront_resident_ctas(P, &resident);
    if (e != cudaSuccess) { program_destroy(p); set_error("occupancy query failed: %s", cudaGetErrorString(e)); return LOP_ECUDA; }
    if (cluster > 1) p->grid = std::min((n_items + cluster - 1) / cluster * cluster, resident / cluster * cluster);
    if (resident < p->grid || p->grid == 0) {
        program_destroy(p);
        set_error("the device holds %d CTAs of the persistent kernel at a time, the program needs %d", resident, p->grid);
        return LOP_EUNSUPPORTED;
    }
    *result = p;
    return LOP_OK;
}

int program_launch(Program *p, cudaStream_t s)
{
    if (!p || p->grid == 0) return LOP_OK;
    p->params.spin_limit = (p->owner && p->owner->wait_limit) ? p->owner->wait_limit : WF_SPIN_LIMIT_DEFAULT;
    cudaError_t e = launch_wavefront(p->params, p->grid, s);
    if (e != cudaSuccess) { set_error("wavefront launch failed: %s", cudaGetErrorString(e)); return LOP_ECUDA; }
    return LOP_OK;
}

bool program_empty(const Program *p) { return !p || p->grid == 0; }

unsigned *program_arrival_flag(Program *p, int band)
{
    if (!p || !p->counters || band < 0 || band >= p->n_flags) return nullptr;
    return p->counters + p->flag_base + band;
}

}  // namespace lop
