// PTX wrappers for sm_100a shared by the tensor-core kernels: mbarrier, TMA (cp.async.bulk.tensor),
// tcgen05 (alloc / mma / commit / ld) and the shared-memory matrix descriptor.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "lop.h"
#include "lop_rowops.cuh"

namespace lop {
namespace ptx {

constexpr uint32_t WAIT_LIMIT = 1u << 23;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// True in one lane of a converged warp, the same one every time.  The single-thread roles are entered by this and not by a
// comparison with a lane number: the compiler knows then that one thread is active, and hands addresses and descriptors to
// the TMA and tensor-core instructions without a loop over the warp's active lanes.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "elect.sync _|p, 0xffffffff;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(p));
    return p != 0u;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Distributed shared memory: an address of this CTA's shared memory in CTA `rank` of the cluster; stores there whose bytes
// count on one of that CTA's barriers.
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ uint32_t cta_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void st_async(uint32_t remote, uint32_t value, uint32_t remote_bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(remote), "r"(value), "r"(remote_bar) : "memory");
}
__device__ __forceinline__ void st_async4(uint32_t remote, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t remote_bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(remote), "r"(a), "r"(b), "r"(c), "r"(d),
                 "r"(remote_bar)
                 : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t remote, uint32_t value)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote), "r"(value) : "memory");
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive;" ::: "memory");
    asm volatile("barrier.cluster.wait;" ::: "memory");
}

// Bounded wait on an mbarrier phase; false when the limit ran out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i) {
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
    }
    return false;
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2,
                                            int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

// A box's lines on their way to L2; a tensor map's 128 bytes on their way to the descriptor cache.
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap *map, int c0, int c1, int c2)
{
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// Bulk tensor store of one box, shared -> global; elements outside the map's extents are not written.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, uint32_t src, int c0, int c1, int c2, int c3)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(reinterpret_cast<uint64_t>(map)),
                 "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }

// Shared-memory matrix descriptor of a K-major operand tile (rows of `row bytes` = swizzle span).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t sbo_bytes, uint32_t layout_code)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);               // start address, 16-byte units
    d |= (uint64_t)1 << 16;                                // leading-dimension offset: unused for swizzled K-major
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;      // stride between 8-row groups
    d |= (uint64_t)1 << 46;                                // descriptor version of this architecture
    // base-offset field (bits 49-51) stays 0: the swizzle is a function of the shared-memory address itself, so
    // an operand may start at any row of a 1024-byte-aligned box (the slab convolution's shifted taps rely on it)
    d |= (uint64_t)layout_code << 61;                      // swizzle mode
    return d;
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float exp2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// GELU, t * Phi(t) with the exact normal distribution function, of two values.  The upper tail Q(u) = Phi(-u) is R(v) *
// exp(-u^2 / 2) with v = 0.33 u / (1 + 0.33 u), after the form of Abramowitz and Stegun 7.1.26; R is of degree seven with R(0) = 1/2,
// fitted for this purpose (least squares reweighted towards the largest relative error, which is 3e-8 up to u = 3 before
// rounding, 1e-6 at 5, 1e-5 at 9).  In v, which is small where u is, and not in 1 - v, whose rounding would weigh twice its
// size in Q(0).  Norm of the error over the result's against 64 bits, for normal t of deviation 1, 2, 3: 3.5, 3.1, 2.6e-8;
// 0.5 t (1 + erf(t / sqrt 2)) in fp32 has 3.8, 3.7, 3.1e-8; relative to a single value of |t| < 1 at most 3.1e-7 and 2.2e-7.
// It keeps its relative accuracy in the lower tail, where that form cancels.  It has neither branches nor the library
// erf's two polynomials, which took 5.5 us of a 128x128 tile's epilogue (a ConvNeXt block 45.0 -> 41.0 us).
// u is clamped at 16, where Q is 0 in fp32, so that an infinite t has no 0 * infinity on the way.
__device__ __forceinline__ float2 gelu2(float t0, float t1)
{
    using rowop::f32x2;
    auto both = [](float c) { return rowop::pack2(c, c); };
    auto mul2 = [](f32x2 a, f32x2 b) { f32x2 d; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; };
    const f32x2 u = rowop::pack2(fminf(fabsf(t0), 16.0f), fminf(fabsf(t1), 16.0f));
    f32x2 den = both(1.0f);
    rowop::fma2(den, u, both(0.33f));
    float d0, d1;
    rowop::unpack2(den, d0, d1);
    const f32x2 v = mul2(mul2(u, both(0.33f)), rowop::pack2(rcp_approx(d0), rcp_approx(d1)));
    const float coeff[7] = {0.10439056158065796f, 0.030913464725017548f, -0.145896777510643f, -0.3189733922481537f,
                            1.086843490600586f, -1.2089178562164307f, 0.5f};
    f32x2 r = both(-0.04851029813289642f);
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        f32x2 next = both(coeff[i]);
        rowop::fma2(next, r, v);
        r = next;
    }
    float a0, a1, q0, q1;
    rowop::unpack2(mul2(mul2(u, both(-0.72134752f)), u), a0, a1);              // -u^2 / (2 ln 2)
    rowop::unpack2(mul2(r, rowop::pack2(exp2_approx(a0), exp2_approx(a1))), q0, q1);
    return make_float2(t0 * (t0 < 0.0f ? q0 : 1.0f - q0), t1 * (t1 < 0.0f ? q1 : 1.0f - q1));
}

// Activation with the kind fixed at compile time: selected once per tile, outside the per-element loops (a
// run-time `act` inside them makes the compiler evaluate the SiLU division for every element of every kind).
template <int ACT>
__device__ __forceinline__ float2 activate2_t(float t0, float t1)
{
    if (ACT == LOP_ACT_RELU) return make_float2(fmaxf(t0, 0.0f), fmaxf(t1, 0.0f));
    if (ACT == LOP_ACT_SILU) return make_float2(__fdividef(t0, 1.0f + __expf(-t0)), __fdividef(t1, 1.0f + __expf(-t1)));
    if (ACT == LOP_ACT_GELU) return gelu2(t0, t1);
    return make_float2(t0, t1);
}
template <int ACT, int N>
__device__ __forceinline__ void activate_n(float (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const float2 f = activate2_t<ACT>(v[i], v[i + 1]);
        v[i] = f.x; v[i + 1] = f.y;
    }
}

template <int ACT, int N>
__device__ __forceinline__ void finish_n_t(float (&v)[N], const float (&rv)[N], int res_pos)
{
    if (res_pos == LOP_RES_PRE_ACT) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = __fadd_rn(v[i], rv[i]);
    }
    activate_n<ACT>(v);
    if (res_pos == LOP_RES_POST_ACT) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = __fadd_rn(v[i], rv[i]);
    }
}
// Last step of the fused epilogue on N channels: v = scale*acc + shift already; rv = residual values.
// res_pos must be LOP_RES_NONE when there is no residual (rv is then not read).  FORM: 0 has neither SiLU nor GELU, 1 has
// both (the persistent kernel, whose roles compete for registers and instruction cache), 2 has a copy of the whole for each
// activation (a stand-alone kernel: 51.3 us for a VGG block where form 1 takes 54.2).
// The additions are kept from being contracted into an activation's last product: both forms give the same bits.
template <int FORM, int N>
__device__ __forceinline__ void finish_n(float (&v)[N], const float (&rv)[N], int res_pos, int act)
{
    if (FORM == 2) {
        if (act == LOP_ACT_RELU) finish_n_t<LOP_ACT_RELU>(v, rv, res_pos);
        else if (act == LOP_ACT_SILU) finish_n_t<LOP_ACT_SILU>(v, rv, res_pos);
        else if (act == LOP_ACT_GELU) finish_n_t<LOP_ACT_GELU>(v, rv, res_pos);
        else finish_n_t<LOP_ACT_NONE>(v, rv, res_pos);
        return;
    }
    if (res_pos == LOP_RES_PRE_ACT) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = __fadd_rn(v[i], rv[i]);
    }
    if (act == LOP_ACT_RELU) {
        activate_n<LOP_ACT_RELU>(v);
    } else if (FORM > 0 && act == LOP_ACT_SILU) {
        activate_n<LOP_ACT_SILU>(v);
    } else if (FORM > 0 && act == LOP_ACT_GELU) {
        activate_n<LOP_ACT_GELU>(v);
    }
    if (res_pos == LOP_RES_POST_ACT) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = __fadd_rn(v[i], rv[i]);
    }
}

__device__ __forceinline__ int floor_div_i(int a, int b) { int q = a / b; return (a % b != 0 && a < 0) ? q - 1 : q; }


}  // namespace ptx
}  // namespace lop
