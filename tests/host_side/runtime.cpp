// Stand-ins for the CUDA runtime and for the library's kernel launches, so that its host side (planner, executors, program
// builder) runs without a GPU: device allocations are host memory, stream commands and launches only append a line to a log,
// and the tables of the last persistent launch can be read back.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "lop_internal.h"
#include "lop_kernels.cuh"
#include "lop_wavefront.cuh"

namespace {
std::string g_log;
std::map<uintptr_t, size_t> g_pinned;                  // page-locked host buffers
lop::WfParams g_last{};
uintptr_t g_handle = 0x100;                            // streams and events: 0x110, 0x120, ...
constexpr uintptr_t DEVICE_LO = uintptr_t(1) << 46;     // addresses from here on are device memory

template <typename... A>
cudaError_t note(const char *fmt, A... a)
{
    char line[256];
    std::snprintf(line, sizeof line, fmt, a...);
    g_log += line;
    g_log += '\n';
    return cudaSuccess;
}
unsigned long long id(const void *p) { return (unsigned long long)reinterpret_cast<uintptr_t>(p); }
template <typename T>
cudaError_t fresh(T *out) { g_handle += 0x10; *out = reinterpret_cast<T>(g_handle); return cudaSuccess; }

CUresult encode(CUtensorMap *m, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill)
{
    std::memset(m, 0, sizeof *m);
    return CUDA_SUCCESS;
}
CUresult write_value(CUstream s, CUdeviceptr, cuuint32_t, unsigned) { note("flag %llx", id(s)); return CUDA_SUCCESS; }
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { *p = std::calloc(1, n); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t n, cudaStream_t s) { return note("memset %llx %zu", id(s), n); }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t n, cudaMemcpyKind, cudaStream_t s) { return note("copy %llx %zu", id(s), n); }
cudaError_t cudaMemcpy2DAsync(void *, size_t, const void *, size_t, size_t w, size_t h, cudaMemcpyKind, cudaStream_t s)
{
    return note("copy %llx %zu", id(s), w * h);
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return fresh(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return note("wait %llx %llx", id(s), id(e)); }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return fresh(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return fresh(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return note("record %llx %llx", id(s), id(e)); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "(no runtime)"; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char *, void **fn, unsigned long long, cudaDriverEntryPointQueryResult *q)
{
    *fn = reinterpret_cast<void *>(write_value);
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p)
{
    std::memset(a, 0, sizeof *a);
    const uintptr_t v = reinterpret_cast<uintptr_t>(p);
    if (v >= DEVICE_LO) { a->type = cudaMemoryTypeDevice; a->devicePointer = const_cast<void *>(p); return cudaSuccess; }
    for (const auto &b : g_pinned)
        if (v >= b.first && v < b.first + b.second) {
            a->type = cudaMemoryTypeHost;
            a->devicePointer = a->hostPointer = const_cast<void *>(p);
            return cudaSuccess;
        }
    a->type = cudaMemoryTypeUnregistered;
    return cudaSuccess;
}

// (the object files register no device code: there is none to register it with)
void **__cudaRegisterFatBinary(void *) { static void *none; return &none; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}

// what a test sets and reads
void host_side_pin(uintptr_t p, size_t n) { if (n) g_pinned[p] = n; else g_pinned.erase(p); }
void host_side_clear() { g_log.clear(); g_last = lop::WfParams{}; }
const char *host_side_log() { return g_log.c_str(); }

// The operand rings of the last persistent launch, walked CTA by CTA as the kernel's loader fills them and its MMA issuer
// follows: 0 when every entry fits its ring, no entry overlaps a live one, every wait for a place is for a group of boxes
// that is complete, and both sides agree on the places; else the number of the stage where that fails, plus one.
int host_side_walk_rings()
{
    using namespace lop;
    const WfParams &P = g_last;
    auto up = [](uint32_t v) { return (v + 1023u) & ~1023u; };
    const int grid = P.n_items < 148 ? P.n_items : 148;
    for (int cta = 0; cta < grid; ++cta) {
        struct Entry { uint32_t at, size, head; bool complete; };
        std::vector<Entry> es;
        uint32_t lim = 0, head = 0, pos = 0, tail_at = 0, n_freed = 0, slab_end0 = 0, slab_end1 = 0, issuer_pos = 0;
        long long cut_key = 0;
        bool first = true;
        for (int item = cta; item < P.n_items; item += grid) {
            const int4 rec = P.items[item];
            const int sidx = rec.x & 0xFFFF;
            const WfStage &s = P.stages[sidx];
            if (s.kind != WF_CONV) continue;
            const uint32_t a = up(s.a_bytes), b = up(s.b_bytes);
            const bool kept = s.keep_bytes != 0, slab = s.mode == WF_SLAB;
            const long long key = kept ? (((long long)s.map_base << 16) | (int)((unsigned)rec.x >> 16)) + 1 : (slab ? -(long long)a : 0);
            if (first || key != cut_key) {
                first = false;
                cut_key = key;
                const uint32_t cut = key < 0 ? 2u * a : (uint32_t)s.keep_bytes;
                if (cut >= P.ring_bytes) return sidx + 1;
                lim = P.ring_bytes - cut;
                n_freed = slab_end0 = slab_end1 = (uint32_t)es.size();
                head = pos = tail_at = issuer_pos = 0;
            }
            auto free_oldest = [&]() {
                if (n_freed == es.size() || !es[n_freed].complete) return false;       // the kernel would wait for good
                ++n_freed;
                tail_at = n_freed == es.size() ? head : es[n_freed].head;
                return true;
            };
            auto place = [&](uint32_t size) {
                if (pos + size > lim) { head += lim - pos; pos = 0; }
                if (n_freed == es.size()) tail_at = head;
                while (head + size - tail_at > lim || es.size() - n_freed == (size_t)WF_ENTRIES)
                    if (!free_oldest()) return false;
                for (size_t e = n_freed; e < es.size(); ++e)
                    if (pos < es[e].at + es[e].size && es[e].at < pos + size) return false;
                if (issuer_pos + size > lim) issuer_pos = 0;
                if (issuer_pos != pos || pos + size > lim) return false;
                es.push_back(Entry{pos, size, head, false});
                head += size; pos += size; issuer_pos += size;
                return true;
            };
            auto complete = [&](size_t n) { for (size_t e = es.size() - n; e < es.size(); ++e) es[e].complete = true; };
            if (slab && !kept) {
                const int per_chunk = (s.n_taps + s.tb - 1) / s.tb;
                for (int ch = 0; ch < s.n_chunks; ++ch) {
                    while ((int)(n_freed - slab_end0) < 0)
                        if (!free_oldest()) return sidx + 1;
                    for (int i = 0, n = 0; i < per_chunk; ++i) {
                        if (!place(b)) return sidx + 1;
                        if (++n == s.cps || i == per_chunk - 1) { complete((size_t)n); n = 0; }
                    }
                    slab_end0 = slab_end1; slab_end1 = (uint32_t)es.size();
                }
            } else {
                const int steps = slab ? s.n_chunks : s.n_chunks * s.n_taps, cps = slab ? 1 : s.cps;
                for (int st = 0; st < steps; st += cps) {
                    if (!place((uint32_t)(steps - st < cps ? steps - st : cps) * (kept ? a : a + b))) return sidx + 1;
                    complete(1);
                }
            }
        }
    }
    return 0;
}
}

namespace lop {
cudaError_t launch_conv_simt(const ConvArgs &a, int, cudaStream_t s) { return note("conv %llx rows %d %d", id(s), a.oh_lo, a.oh_hi); }
cudaError_t launch_maxpool(const PoolArgs &a, int, cudaStream_t s) { return note("pool %llx rows %d %d", id(s), a.oh_lo, a.oh_hi); }
cudaError_t launch_dwconv(const ConvArgs &a, int, const void *, cudaStream_t s) { return note("dwconv %llx rows %d %d", id(s), a.oh_lo, a.oh_hi); }
cudaError_t launch_layernorm(const ConvArgs &a, int, cudaStream_t s) { return note("layernorm %llx rows %d %d", id(s), a.oh_lo, a.oh_hi); }
cudaError_t launch_concat(const ConvArgs &a, int, cudaStream_t s) { return note("concat %llx rows %d %d", id(s), a.oh_lo, a.oh_hi); }
cudaError_t launch_dw_transpose(const void *, void *, int, int, cudaStream_t s) { return note("weights %llx", id(s)); }
cudaError_t launch_stem_weights(const StemWeights &, cudaStream_t s) { return note("weights %llx", id(s)); }
cudaError_t launch_stem_gather(const void *, void *, const GatherGeom &, int lo, int hi, cudaStream_t s, unsigned *, const StemWeights &)
{
    return note("gather %llx rows %d %d", id(s), lo, hi);
}
cudaError_t launch_fetch_rows(const void *, void *, int, int, long long, int lo, int hi, cudaStream_t s) { return note("fetch %llx rows %d %d", id(s), lo, hi); }
ConvTcGeom conv_tc_geometry(const ConvArgs &, int, bool) { return ConvTcGeom{}; }
int conv_tc_encode(const ConvArgs &, const ConvTcGeom &, ConvTcMaps *) { return LOP_OK; }
cudaError_t launch_conv_tc(const ConvArgs &a, const ConvTcGeom &, const ConvTcMaps &, unsigned *, cudaStream_t s)
{
    return note("conv %llx rows %d %d", id(s), a.oh_lo, a.oh_hi);
}
TensorMapEncodeFn tensor_map_encoder() { return encode; }
size_t wavefront_smem_bytes(const WfParams &p) { return 1024 + (size_t)p.ring_bytes + (size_t)WF_UNITS * p.unit_bytes + p.simt_bytes + WF_FIXED_SMEM; }
cudaError_t wavefront_resident_ctas(const WfParams &, int *ctas) { *ctas = 148; return cudaSuccess; }
cudaError_t launch_wavefront(const WfParams &p, int, cudaStream_t s) { g_last = p; return note("persistent %llx %zu", id(s), wavefront_smem_bytes(p)); }
}  // namespace lop

extern "C" int lop_run_whole_static(lop_plan_t *, const void *, void *, unsigned *, void *) { return LOP_EUNSUPPORTED; }
