// What the two TMA + tcgen05 attention kernels (attn_tc5.cu, attn_tc5_wide.cu) share: PTX wrappers, the exponential on the FMA
// pipe, the work schedule every CTA derives from kv_len, the paged producer, and the merge of split-KV partials.
#pragma once
#include <cuda_bf16.h>
#include <cstdint>
#include <type_traits>

#include "launch.cuh"
#include "vispec_internal.h"

namespace vispec {
namespace tc5 {

constexpr int D = 128;                         // head size of the paged and fused-rotary forms; the plain one also takes 64
constexpr int kMaxB = 32;                      // sequences per call these kernels take
constexpr float kRescaleGap = 8.0f;            // log2 units
constexpr long long kWaitCycles = 1500000000LL;   // ~0.8 s at 1.9 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Has the phase with parity `parity` completed?  One non-blocking test; its result can be left unused for a while.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait for the completion of the phase with parity `parity`.  Returns false after ~limit cycles
// or as soon as another role has raised the abort flag.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          long long limit = kWaitCycles) {
    long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
        if ((it & 63) == 63) {
            if (*abort_flag) return false;
            const long long now = clock64();
            if (t0 == 0) t0 = now;
            else if (now - t0 > limit) { *abort_flag = 1; return false; }
        }
    }
}
// The same wait for a barrier that threads of other CTAs of the cluster arrive on (acquire at cluster scope).
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                  long long limit = kWaitCycles) {
    long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
        if ((it & 63) == 63) {
            if (*abort_flag) return false;
            const long long now = clock64();
            if (t0 == 0) t0 = now;
            else if (now - t0 > limit) { *abort_flag = 1; return false; }
        }
    }
}
// Same, with a warp-uniform result (every lane of a converged warp calls it): the warp-collective
// tcgen05.ld/st that follow must never be reached by only part of a warp.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag));
}
// The K/V tiles are read once per call: they are marked evict-first in L2 so that the stream does not push out
// what is read again soon (q, masks, partial results, the next kernels' operands).
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "l"(pol) : "memory");
}
// Untiled copy of `bytes` (a multiple of 16, both addresses on 16 bytes) from global to shared memory.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// Thread-block cluster helpers (distributed shared memory).
__device__ __forceinline__ uint32_t cluster_ctarank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of the same shared-memory location in the CTA of rank `rank` of this cluster.
__device__ __forceinline__ uint32_t dsmem_addr(uint32_t local, uint32_t rank) {
    uint32_t r; asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank)); return r;
}
__device__ __forceinline__ float4 dsmem_ld4(uint32_t a) {
    float4 v; asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory"); return v;
}
__device__ __forceinline__ float4 smem_ld4(uint32_t a) {
    float4 v; asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory"); return v;
}
__device__ __forceinline__ float2 smem_ld2(uint32_t a) {
    float2 v; asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory"); return v;
}
__device__ __forceinline__ float2 dsmem_ld2(uint32_t a) {
    float2 v; asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory"); return v;
}
// The hardware cluster barrier in two halves: a warp arrives once and waits once per phase, all its lanes together
// (a wait taken by one lane and later by the other 31 never returns); the wait may sit anywhere later in the warp's
// path.  Relaxed arrival: what the peers must see, the initialised barriers, is published by fence.mbarrier_init.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// One arrival on an mbarrier of another CTA of the cluster (address from dsmem_addr), ordered after this thread's
// earlier accesses at cluster scope.
__device__ __forceinline__ void mbar_arrive_peer(uint32_t peer_bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(peer_bar) : "memory");
}
// One lane of a converged warp, the same one every time.
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0;
}
// One tcgen05.mma (cta_group::1, kind::f16) with the A operand in TMEM and B described in shared memory.
// The 64-bit descriptor is passed as 32-bit halves: the high half is constant, the low half carries the address.
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi,
                                          uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate) : "memory");
}
// The same with both operands described in shared memory.
__device__ __forceinline__ void tc_mma_ss(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                          uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate) : "memory");
}
// 32 lanes x 32 bit, 32 consecutive columns: thread i of the warp accesses lane (base lane + i).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr),
          "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr),
          "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor (sm_100 format), split in halves.  Low: start address and leading byte
// offset, both in 16-byte units.  High: stride byte offset (16-byte units), descriptor version 1 (bit 46),
// 128-byte swizzle (value 2 in bits 61-63).  Tile bases are 1024-byte aligned (base offset 0).
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo_bytes) {
    return ((addr >> 4) & 0x3FFFu) | ((lbo_bytes >> 4) << 16);
}
__host__ __device__ constexpr uint32_t desc_hi(uint32_t sbo_bytes) {
    return (sbo_bytes >> 4) | (1u << 14) | (2u << 29);
}
// Instruction descriptor, kind::f16: D fp32, A and B bf16, A K-major, M = 128, N = n; b_mn = 1 if B is MN-major.
__host__ __device__ constexpr uint32_t instr_desc(int b_mn, int n = 128) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn << 16) | (((uint32_t)n >> 3) << 17) | ((128u >> 4) << 24);
}
// 128-bit shifts on (lo, hi) pairs; any shift count >= 0.
__device__ __forceinline__ void shr128(uint64_t lo, uint64_t hi, int s, uint64_t& rlo, uint64_t& rhi) {
    if (s >= 128) { rlo = 0; rhi = 0; }
    else if (s >= 64) { rlo = hi >> (s - 64); rhi = 0; }
    else if (s == 0) { rlo = lo; rhi = hi; }
    else { rlo = (lo >> s) | (hi << (64 - s)); rhi = hi >> s; }
}
__device__ __forceinline__ void shl128_fill(uint64_t lo, uint64_t hi, int s, uint64_t& rlo, uint64_t& rhi) {
    // shift left by s in (0, 128) and set the s vacated low bits
    if (s >= 64) { rlo = ~0ull; rhi = (lo << (s - 64)) | (s == 64 ? 0ull : ((1ull << (s - 64)) - 1)); }
    else { rlo = (lo << s) | ((1ull << s) - 1); rhi = (hi << s) | (lo >> (64 - s)); }
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// ---- two fp32 lanes per instruction
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
    uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi)); return r;
}
__device__ __forceinline__ void up2(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r; asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r; asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r;
}
// The largest, NaN if any of them is (fmaxf drops it).
__device__ __forceinline__ float max_nan(float a, float b) {
    float r; asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
    float r; asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r;
}
// 1 / l for a row's sum l >= 0; a row that saw nothing (l = 0) is scaled to zeros, one that saw a NaN or an infinite score
// (the softmax makes its l NaN, whatever the exponentials gave) to NaN.
__device__ __forceinline__ float inv_sum(float l) { return l > 0.f ? 1.f / l : l; }
// 2^x on the FMA pipe (x <= 120, not NaN; -inf gives exactly 0, below -126 a denormal or 0 comes out): nearest integer by the
// 1.5 * 2^23 trick, a polynomial of degree 5 on the remainder f in [-0.5, 0.5], the integer added into the exponent field (at the
// clamp the remainder is not negative, so 2^-127 p(f) >= 2^-127 stays a positive pattern, and 0 at f = 0).  The polynomial is
// 1 + C1 f + ... + C5 f^5 with the largest relative error made smallest: 9.2e-8, 1.7e-7 with the roundings of its fp32
// evaluation, which is within exp2f's own 2 ulp, so that a row's sum and its lse do not depend on which columns come through
// here (a cubic, 7.5e-5, showed in lse).
constexpr float kExp2C1 = 0.693147f, kExp2C2 = 0.24022242f, kExp2C3 = 0.055507336f, kExp2C4 = 0.009671513f, kExp2C5 = 0.0013264727f;
__device__ __forceinline__ float exp2_fma(float x) {
    x = fmaxf(x, -127.f);
    const float z = x + 12582912.f;
    const float f = x - (z - 12582912.f);
    float p = fmaf(f, kExp2C5, kExp2C4);
    p = fmaf(p, f, kExp2C3);
    p = fmaf(p, f, kExp2C2);
    p = fmaf(p, f, kExp2C1);
    p = fmaf(p, f, 1.f);
    return __int_as_float(__float_as_int(p) + (__float_as_int(z) << 23));
}
__device__ __forceinline__ void exp2_fma_pair(float x0, float x1, float& e0, float& e1) {
    const uint64_t x = pk2(fmaxf(x0, -127.f), fmaxf(x1, -127.f));
    const uint64_t z = add2(x, pk2(12582912.f, 12582912.f));
    const uint64_t f = fma2(add2(z, pk2(-12582912.f, -12582912.f)), pk2(-1.f, -1.f), x);
    uint64_t p = fma2(f, pk2(kExp2C5, kExp2C5), pk2(kExp2C4, kExp2C4));
    p = fma2(p, f, pk2(kExp2C3, kExp2C3));
    p = fma2(p, f, pk2(kExp2C2, kExp2C2));
    p = fma2(p, f, pk2(kExp2C1, kExp2C1));
    p = fma2(p, f, pk2(1.f, 1.f));
    float p0, p1, z0, z1;
    up2(p, p0, p1); up2(z, z0, z1);
    e0 = __int_as_float(__float_as_int(p0) + (__float_as_int(z0) << 23));
    e1 = __int_as_float(__float_as_int(p1) + (__float_as_int(z1) << 23));
}

struct Tc5Params {
    const __nv_bfloat16* q; const int32_t* kv_len; const uint64_t* mask;
    __nv_bfloat16* out; float* lse;
    float4* part_o;            // [slot][D/4 col4][ROWS]: column-of-4 major, so that a warp's 32 rows are contiguous
    float2* part_ml;           // [slot][ROWS]: (m in log2 units or -inf, l)
    int B, N, Hq, Hkv, S_max, n_mblocks;
    int grid_attn;             // CTAs of the attention kernel (the merge kernel needs it for the schedule)
    int min_steps;             // a CTA is given at least this many steps (fewer CTAs work on small problems)
    int early;                 // stream committed-prefix tiles before waiting for the preceding kernel
    float scale_log2;
    int* status;
    int step;                  // cached tokens per pipeline step (rows of one K or V stage)
    short seg_cost;            // even split: steps that a segment's start is counted as when the line is cut (see SegIter)
    short lock;                // even split by groups of n_mblocks CTAs: CTA c works for group c / n_mblocks on row block c % n_mblocks
};
// Two descriptors, this and PagedArgs are 416 bytes of kernel parameters.  With more of them a launch takes 0.35 us of host time longer
// (424 or 488 bytes: 7.65 and 7.8 us a call of vispec_tree_verify_attn_static on 4 heads of size 64, 1 x 8 nodes on 256 tokens, against
// 7.3), and that is what bounds the shortest calls.
static_assert(sizeof(Tc5Params) <= 112, "a larger parameter block makes every launch slower");

// The schedule every CTA (and the merge kernel) derives from kv_len.
struct Sched {
    int base[kMaxB + 1];   // where sequence b starts on the line (see SegIter); base[B] = T
    int steps[kMaxB];      // steps of one unit of sequence b (0: sequence rejected or empty)
    int len[kMaxB];        // committed length S of sequence b
    int units;             // units with at least one step
};

// ---- schedule ---------------------------------------------------------------------------------------
// Built by one full warp.  Reads kv_len only.
static __device__ void sched_build(Sched& s, const Tc5Params& p, int lane, int kv_first) {   // kv_first: kv_len[lane], fetched by the caller

    const int upb = p.lock ? p.Hkv : p.Hkv * p.n_mblocks;        // units (lock: kv heads) per sequence
    int carry = 0;
    for (int b0 = 0; b0 < p.B; b0 += 32) {
        const int b = b0 + lane;
        int st = 0, S = 0;
        if (b < p.B) {
            S = b0 == 0 ? kv_first : p.kv_len[b];
            const bool ok = (S >= 0 && S + p.N <= p.S_max);
            st = ok ? (S + p.N + p.step - 1) / p.step : 0;
            s.steps[b] = st;
            s.len[b] = S;
        }
        const int len = st > 0 ? (st + p.seg_cost) * upb : 0;
        int x = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (b < p.B) s.base[b] = carry + x - len;
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) s.base[p.B] = carry;
    __syncwarp();
    int live = 0;
    for (int b0 = 0; b0 < p.B; b0 += 32) {
        const int b = b0 + lane;
        live += __popc(__ballot_sync(0xffffffffu, b < p.B && s.steps[b] > 0));
    }
    if (lane == 0) s.units = live * upb;
}
// Number of CTAs that get a range: each at least min_steps places of the line (see SegIter; with segments' starts counted a range may hold
// one step or none); a multiple of the unit count when
// the units are fewer than the CTAs (equally long units then never share a CTA) - unless the CTAs left out cost more
// steps than a second segment's Q tile and epilogue in every CTA (round_steps).  Unaligned ranges put the row blocks of a
// kv head, where they are units of their own, at different places of the cache, which is then read once per row block
// (qwen3b_S32768_N128_B8 345 -> 417 us): those are always aligned.
__device__ __forceinline__ int sched_round_steps(const Tc5Params& p) { return p.lock || p.n_mblocks == 1 ? 3 : 1 << 30; }
__device__ __forceinline__ int sched_ctas(int T, int units, int grid, int min_steps, int round_steps) {
    int g = T / min_steps;
    g = g < 1 ? 1 : g;
    g = g < grid ? g : grid;
    if (units <= g) {
        const int r = (g / units) * units;
        if (r != g && (T + r - 1) / r - (T + g - 1) / g <= round_steps) g = r;
    }
    return g;
}
// (T * grid < 2^31 is checked on the host, so 32-bit arithmetic suffices)
__device__ __forceinline__ int cta_lo(int c, int T, int geff) { return (int)(((unsigned)c * (unsigned)T) / (unsigned)geff); }
// The CTA whose range holds place g of the line.
__device__ __forceinline__ int cta_of(int g, int T, int geff) {
    int c = (int)((((unsigned)g + 1u) * (unsigned)geff - 1u) / (unsigned)T);
    c = c > geff - 1 ? geff - 1 : c;
    while (cta_lo(c, T, geff) > g) --c;
    while (c + 1 < geff && cta_lo(c + 1, T, geff) <= g) ++c;
    return c;
}

struct Seg {
    int b, kvh, mblock, st0, n, steps, S, slot;    // slot < 0: the segment is a whole unit
};
// The line that the even split cuts: every unit is seg_cost places without work, then its steps.  A CTA whose range takes in the
// start of a unit pays for one more segment (a Q tile, an empty pipeline and an epilogue: 5 us with rows <= 64, as long as 4
// steps), and so gets as many steps less; without it llava13b_b4's CTAs, the Q rows sent ahead already, ended after 44, 49 or 54 us by
// the number of their segments.
// COST: seg_cost may be other than 0 (rows <= 64; elsewhere the register that it takes costs more).
template <bool COST>
struct SegIter {
    const Sched* s;
    int B, n_mblocks, seg_cost_, g, lo, hi, cta;
    bool cl, cl_done;          // cluster schedule: exactly one segment (possibly empty), given in cl_seg
    Seg cl_seg;
    __device__ __forceinline__ bool next(Seg& o) {
        if (cl) {
            if (cl_done) return false;
            cl_done = true;
            o = cl_seg;
            return true;
        }
        const int seg_cost = COST ? seg_cost_ : 0;
        for (;;) {
            if (g >= hi) return false;
            int l = 0, r = B;                               // first b with base[b] > g, minus one
            while (l < r) { const int m = (l + r) >> 1; if (s->base[m] <= g) l = m + 1; else r = m; }
            o.b = l - 1;
            o.steps = s->steps[o.b];
            o.S = s->len[o.b];
            const int rel = g - s->base[o.b], len = o.steps + seg_cost;
            const int uib = rel / len, off = rel - uib * len, end = min(len, off + hi - g);   // of this unit, places [off, end)
            o.st0 = COST ? max(off - seg_cost, 0) : off;
            o.n = end - seg_cost - o.st0;
            o.kvh = uib / n_mblocks;
            o.mblock = uib - o.kvh * n_mblocks;
            const bool whole = (o.st0 == 0 && o.n == o.steps);
            o.slot = whole ? -1 : (g == lo ? 2 * cta : 2 * cta + 1);
            g += end - off;
            if (!COST || o.n > 0) return true;
        }
    }
};

// One (row, 16 output columns) of a unit: the partials of CTAs c0..c1 (slot 2c if the unit starts CTA c's range,
// else 2c + 1) folded into the final output.  Shared by the merge kernel and by the attention kernel's own merge.
template <int ROWS, int HD, bool WAIT = false>      // WAIT: for the kernel that writes the partials, ahead of the first load
__device__ __forceinline__ void merge_row_cols(const float4* __restrict__ part_o, const float2* __restrict__ part_ml,
                                               __nv_bfloat16* __restrict__ out, float* __restrict__ lse, int T, int geff,
                                               int ub, int c0, int c1, int b, int node, int head, int Hq, int N,
                                               int lrow, int cw, int smul = 1, int sadd = 0) {
    auto slot_of = [&](int c) { return (cta_lo(c, T, geff) >= ub ? 2 * c : 2 * c + 1) * smul + sadd; };
    // Segments are taken four at a time with every load of a group issued before the first use, so that a
    // group costs one memory round trip; groups are folded with the usual running-maximum rescale.
    float m_all = -INFINITY, l_all = 0.f;
    float4 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (WAIT && c1 < c0) pdl_wait();                  // (a lane without a row)
    for (int cb = c0; cb <= c1; cb += 4) {
        float2 ml[4];
        float4 v[4][4];
        int slot[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) slot[j] = slot_of(min(cb + j, c1));
        if (WAIT && cb == c0) pdl_wait();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = cb + j;
            ml[j] = make_float2(-INFINITY, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) v[j][k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c <= c1) {
                ml[j] = __ldcg(&part_ml[(size_t)slot[j] * ROWS + lrow]);
                const float4* src = part_o + ((size_t)slot[j] * (HD / 4) + cw * 4) * ROWS + lrow;
#pragma unroll
                for (int k = 0; k < 4; ++k) v[j][k] = __ldcg(src + (size_t)k * ROWS);
            }
        }
        float m_new = m_all;
#pragma unroll
        for (int j = 0; j < 4; ++j) m_new = fmaxf(m_new, ml[j].x);
        const float m_fin = (m_new == -INFINITY) ? 0.f : m_new;
        const float a = exp2f(m_all - m_fin);                 // 0 while nothing has been accumulated
        l_all *= a;
#pragma unroll
        for (int k = 0; k < 4; ++k) { acc[k].x *= a; acc[k].y *= a; acc[k].z *= a; acc[k].w *= a; }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float w = exp2f(ml[j].x - m_fin);           // 0 for a segment that saw nothing (or is absent)
            l_all += ml[j].y * w;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                acc[k].x += w * v[j][k].x; acc[k].y += w * v[j][k].y; acc[k].z += w * v[j][k].z; acc[k].w += w * v[j][k].w;
            }
        }
        m_all = m_new;
    }
    if (WAIT && c1 < c0) return;
    const float inv = inv_sum(l_all);
    __nv_bfloat16* orow = out + (((size_t)b * N + node) * Hq + head) * HD + cw * 16;
#pragma unroll
    for (int k = 0; k < 2; ++k)
        *reinterpret_cast<uint4*>(orow + k * 8) =
            make_uint4(pack_bf16(acc[2 * k].x * inv, acc[2 * k].y * inv), pack_bf16(acc[2 * k].z * inv, acc[2 * k].w * inv),
                       pack_bf16(acc[2 * k + 1].x * inv, acc[2 * k + 1].y * inv), pack_bf16(acc[2 * k + 1].z * inv, acc[2 * k + 1].w * inv));
    if (lse && cw == 0)
        lse[((size_t)b * Hq + head) * N + node] = l_all > 0.f ? (m_all + log2f(l_all)) * 0.6931471805599453f : -INFINITY;
}

// One (row, 4 output columns) of a unit, the merge kernel's fine piece, by Q lanes of a warp (lanes 32/Q apart): lane part
// `part` takes the segments c0 + part, c0 + part + Q, ..., U at a time with every load issued before the first use (a
// unit cut over many CTAs - few sequences, long caches - is merged from dozens of partials, and a round of loads is a memory
// round trip); the Q sums meet by shuffles.  All lanes of the warp take part; those of a row that does not exist pass
// row_ok = false.
template <int ROWS, int HD, int Q>
__device__ __forceinline__ void merge_row_c4(const float4* __restrict__ part_o, const float2* __restrict__ part_ml,
                                             __nv_bfloat16* __restrict__ out, float* __restrict__ lse, int T, int geff,
                                             int ub, int c0, int c1, int b, int node, int head, int Hq, int N,
                                             int lrow, int c4, int part, bool row_ok, int smul, int sadd) {
    constexpr int U = Q == 1 ? 16 : 10;
    auto slot_of = [&](int c) { return (cta_lo(c, T, geff) >= ub ? 2 * c : 2 * c + 1) * smul + sadd; };
    float m_all = -INFINITY, l_all = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int cb = c0; cb <= c1; cb += Q * U) {
        float2 ml[U];
        float4 v[U];
        int slot[U];
#pragma unroll
        for (int j = 0; j < U; ++j) slot[j] = slot_of(min(cb + part + j * Q, c1));
        if (cb == c0) pdl_wait();                         // the partials are complete
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int c = cb + part + j * Q;
            ml[j] = make_float2(-INFINITY, 0.f);
            v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c <= c1 && row_ok) {
                ml[j] = __ldcg(&part_ml[(size_t)slot[j] * ROWS + lrow]);
                v[j] = __ldcg(part_o + ((size_t)slot[j] * (HD / 4) + c4) * ROWS + lrow);
            }
        }
        float m_new = m_all;
#pragma unroll
        for (int j = 0; j < U; ++j) m_new = fmaxf(m_new, ml[j].x);
        const float m_fin = (m_new == -INFINITY) ? 0.f : m_new;
        const float a = exp2f(m_all - m_fin);                 // 0 while nothing has been accumulated
        l_all *= a;
        acc.x *= a; acc.y *= a; acc.z *= a; acc.w *= a;
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const float w = exp2f(ml[j].x - m_fin);           // 0 for a segment that saw nothing (or is absent)
            l_all += ml[j].y * w;
            acc.x += w * v[j].x; acc.y += w * v[j].y; acc.z += w * v[j].z; acc.w += w * v[j].w;
        }
        m_all = m_new;
    }
#pragma unroll
    for (int o = 32 / Q; o < 32; o <<= 1) {
        const float m_o = __shfl_xor_sync(0xffffffffu, m_all, o), m_new = fmaxf(m_all, m_o);
        const float m_fin = (m_new == -INFINITY) ? 0.f : m_new;
        const float a = exp2f(m_all - m_fin);
        // (both sides scale by their own weight before the exchange, so the sum is the same in all of them)
        l_all *= a; acc.x *= a; acc.y *= a; acc.z *= a; acc.w *= a;
        l_all += __shfl_xor_sync(0xffffffffu, l_all, o);
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
        acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
        m_all = m_new;
    }
    if (!row_ok || part != 0) return;
    const float inv = inv_sum(l_all);
    *reinterpret_cast<uint2*>(out + (((size_t)b * N + node) * Hq + head) * HD + c4 * 4) =
        make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
    if (lse && c4 == 0)
        lse[((size_t)b * Hq + head) * N + node] = l_all > 0.f ? (m_all + log2f(l_all)) * 0.6931471805599453f : -INFINITY;
}

// The whole unit, by the softmax threads of the CTA that delivered the unit's last partial (thread st of nthreads).
// Not inlined: its accumulators stay out of the attention kernel's register budget.
struct MergeArgs { const float4* part_o; const float2* part_ml; __nv_bfloat16* out; float* lse; int Hq, G, N, rows_total; };
template <int ROWS, int HD>
__device__ __noinline__ void merge_unit(const MergeArgs m, int T, int geff, int ub, int c0, int c1, int b, int kvh,
                                        int mblock, int st, int nthreads) {
    for (int item = st; item < ROWS * (HD / 16); item += nthreads) {
        const int cw = item / ROWS, lrow = item - cw * ROWS;
        const int row = mblock * ROWS + lrow;
        if (row >= m.rows_total) continue;
        merge_row_cols<ROWS, HD>(m.part_o, m.part_ml, m.out, m.lse, T, geff, ub, c0, c1, b, row / m.G, kvh * m.G + row % m.G,
                             m.Hq, m.N, lrow, cw);
    }
}

// pool [num_blocks][Hkv][page_rows][D] (tensor map (d, slot, block * Hkv + head)) or, token_major,
// [num_blocks][page_rows][Hkv][D] (tensor map (d, head, block * page_rows + slot));
// block_table[b][i] = pool block of logical slots [i * page_rows, (i + 1) * page_rows)
// Fourth kernel parameter of the instantiations with the fused rotary embedding (they serve contiguous caches, so it
// takes the place of PagedArgs; a larger common parameter block costs the other instantiations registers).
struct RopeArgs {
    const double2* rope_k;     // [B][N][D/2] (cos, sin) of positions * theta^(-2j/D), fp64: the k rows' rotation
    const float2* rope_q;      // the same angles in fp32: the q rows' rotation (q is only consumed, never written back)
    const __nv_bfloat16* k_new; const __nv_bfloat16* v_new;   // [B][N][Hkv][D] rows of the tree, to be placed at slots S + i
    __nv_bfloat16* k_cache; __nv_bfloat16* v_cache;            // [B][Hkv][S_max][D]
};
struct PagedArgs { const int32_t* block_table; int table_stride, page_rows, num_blocks, Hkv, N, token_major; int* status;
                   int* unit_counters; };   // even split: arrivals per unit (all zero between calls); nullptr: a merge kernel follows
static_assert(sizeof(RopeArgs) <= 48 && sizeof(PagedArgs) <= 48, "a larger parameter block makes every launch slower (see Tc5Params)");

// ---- producer of a paged segment ---------------------------------------------------------------------
// Paged cache: a step's 128 slots are 128 / page_rows pool blocks, each its own box.  Run by the whole producer
// warp: lane j owns block j of every step - its table entry and its four copies (two d-halves of K and of V) -
// so that one instruction issues the copies of all the step's blocks; lane 0 alone waits for the free stage and
// posts the expected byte count.  The block numbers travel from the table to a small ring in shared memory by
// asynchronous 4-byte copies issued six steps ahead of their use: a plain load held in a register that long would
// share a scoreboard with the waits and copies in between and stall them for its whole latency.  Blocks that start
// at or past kv_len + N are not fetched: their table entries need not exist, and the rows they would fill are
// masked like any slot past the end.  Not inlined, so that it stays out of the kernel's register budget, and
// everything by value, so that the caller's counters stay in registers.  Returns steps issued in full | K-only
// step << 28 | a wait gave up << 29 | has waited for the preceding kernel << 30 | Q rows sent << 31 (the same in every lane).
constexpr int STEP = 128;                      // tokens per pipeline step = rows of one K or V stage
constexpr int HALF_BYTES = STEP * 128;         // one d-half (64 columns) of a stage: 128 rows x 128 B
constexpr int kTabRing = 4, kTabAhead = 3;     // steps held in a ring / steps a copy is issued ahead (two rings of
                                               // 128 bytes: the K producer's and, where V has its own warp, the V producer's)
// The Q rows of a unit that come through the K ring ahead of its first step (n == 0: they do not): row r of the n is that of
// node (row0 + r) / G, the (row0 + r) % G-th head of the kv head.  Here and not in a call of its own: what lived across both calls did
// not fit the registers that a call preserves (44 bytes of spills in the kernel with 128 rows per unit).
struct QStage { const __nv_bfloat16* q; int Hq, G, row0, n; };
template <class R>   // ring geometry: stages, bytes, offsets in shared memory, barrier indices
__device__ __noinline__ uint32_t produce_paged(const PagedArgs p, const CUtensorMap* k_map, const CUtensorMap* v_map,
                                               int b, int kvh, int st0, int n, int S, uint32_t base, uint32_t bars,
                                               uint32_t ring, volatile int* abort_flag, uint64_t pol, int it,
                                               bool waited, int lane, int which /* 0: K and V, 1: K only, 2: V only */,
                                               int koff = 0 /* stages of the K ring used beyond one per step */, QStage qs = {}) {
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    uint32_t told = 0;                                                   // the upper bits of the answer
    if (qs.n > 0) {
        const int ik = it + koff, sk = ik % R::NSK;
        if (!waited) { pdl_wait(); waited = true; }
        if (!__all_sync(0xffffffffu, mbar_wait(bar(R::KEMPTY + sk), ((ik / R::NSK) & 1) ^ 1, abort_flag))) return 2u << 28 | 1u << 30;
        if (lane == 0) mbar_expect_tx(bar(R::KFULL + sk), (uint32_t)qs.n * (R::STAGE / STEP));
        __syncwarp();                                                    // the byte count is posted before any lane copies
        for (int r = lane; r < qs.n; r += 32) {
            const int row = qs.row0 + r;
            bulk_load(base + R::OFF_K + sk * R::STAGE + r * (R::STAGE / STEP),
                      qs.q + (((size_t)b * p.N + row / qs.G) * qs.Hq + kvh * qs.G + row % qs.G) * (R::STAGE / STEP / 2), R::STAGE / STEP, bar(R::KFULL + sk));
        }
        ++koff;
        told = 1u << 31;
    }
    const int nsub = STEP / p.page_rows;
    const uint32_t sub_bytes = (uint32_t)p.page_rows * 128u;
    const int32_t* trow = p.block_table + (size_t)b * p.table_stride;
    const int total = S + p.N;
    const bool mine = lane < nsub;
    auto issue = [&](int t) {                  // one group per step and lane, empty where there is nothing to fetch
        const int blk = (st0 + t) * nsub + lane;
        if (mine && t < n && blk * p.page_rows < total)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(ring + 4u * (uint32_t)((t % kTabRing) * 8 + lane)), "l"(trow + blk) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int t = 0; t < kTabAhead; ++t) issue(t);
    int t = 0;
    for (; t < n; ++t, ++it) {
        issue(t + kTabAhead);
        asm volatile("cp.async.wait_group %0;" ::"n"(kTabAhead) : "memory");     // this lane's entry of step t has landed
        const int tok = (st0 + t) * STEP;
        if (!waited && tok + STEP > S) { pdl_wait(); waited = true; }   // the tree's rows come from the preceding kernel
        const bool load = mine && tok + lane * p.page_rows < total;
        int c1 = 0, c2 = -p.page_rows;                                   // a box outside the pool: reads as zeros
        if (load) {
            int e;
            asm volatile("ld.shared.s32 %0, [%1];" : "=r"(e) : "r"(ring + 4u * (uint32_t)((t % kTabRing) * 8 + lane)) : "memory");
            if (e >= 0 && e < p.num_blocks) {
                c1 = p.token_major ? kvh : 0;
                c2 = p.token_major ? e * p.page_rows : e * p.Hkv + kvh;
            } else if (p.status) {
                atomicCAS(p.status, 0, VISPEC_E_RANGE);
            }
        }
        const uint32_t tx = (uint32_t)__popc(__ballot_sync(0xffffffffu, load)) * sub_bytes * 2u;
        const int ik = it + koff, sk = ik % R::NSK, sv = it % R::NSV;
        bool w = true;
        if (which != 2) {
            if (lane == 0) {
                w = mbar_wait(bar(R::KEMPTY + sk), ((ik / R::NSK) & 1) ^ 1, abort_flag);
                if (w) mbar_expect_tx(bar(R::KFULL + sk), tx);
            }
            w = __shfl_sync(0xffffffffu, w, 0);                          // the byte count is posted before any lane copies
            if (!w) { told |= 2u << 28; break; }
            if (load) {
                tma_load_3d(base + R::OFF_K + sk * R::STAGE + lane * sub_bytes, k_map, bar(R::KFULL + sk), 0, c1, c2, pol);
                tma_load_3d(base + R::OFF_K + sk * R::STAGE + HALF_BYTES + lane * sub_bytes, k_map, bar(R::KFULL + sk), 64, c1, c2, pol);
            }
        }
        if (which != 1) {
            if (lane == 0) {
                w = mbar_wait(bar(R::VEMPTY + sv), ((it / R::NSV) & 1) ^ 1, abort_flag);
                if (w) mbar_expect_tx(bar(R::VFULL + sv), tx);
            }
            w = __shfl_sync(0xffffffffu, w, 0);
            if (!w) { told |= (which == 2 ? 2u : 3u) << 28; break; }      // (V only: nothing of this step was issued)
            if (load) {
                tma_load_3d(base + R::OFF_V + sv * R::STAGE + lane * sub_bytes, v_map, bar(R::VFULL + sv), 0, c1, c2, pol);
                tma_load_3d(base + R::OFF_V + sv * R::STAGE + HALF_BYTES + lane * sub_bytes, v_map, bar(R::VFULL + sv), 64, c1, c2, pol);
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");                     // nothing of this segment stays in flight
    return (uint32_t)t | told | (waited ? 1u << 30 : 0u);
}

// Rejected sequences (kv_len < 0 or kv_len + N > S_max): zero output, -inf lse, status word.  By the NT softmax threads.
template <int HD, int NT = 256>
__device__ __forceinline__ void zero_rejected(const Tc5Params& p, const Sched& sched, int cta, int st) {
    const int N = p.N;
    bool any_bad = false;
    for (int b = 0; b < p.B; ++b) {
        const int S = sched.len[b];
        if (S >= 0 && S + N <= p.S_max) continue;
        any_bad = true;
        const int vecs = N * p.Hq * (HD / 8);
        uint4* o = reinterpret_cast<uint4*>(p.out + (size_t)b * N * p.Hq * HD);
        for (int i = cta * NT + st; i < vecs; i += (int)gridDim.x * NT) o[i] = make_uint4(0, 0, 0, 0);
        if (p.lse)
            for (int i = cta * NT + st; i < N * p.Hq; i += (int)gridDim.x * NT) p.lse[(size_t)b * p.Hq * N + i] = -INFINITY;
    }
    if (any_bad && cta == 0 && st == 0) atomicCAS(p.status, 0, (int)VISPEC_E_RANGE);
}

// Cluster form: rank cr of ck merges its rows of the unit's partials, parked by every rank at pbuf_a ([HD/4 col4][ROWS]
// float4) and pst_a ([ROWS] (m, l)) of its own shared memory, and writes them out.  By the NT softmax threads (st).
// Contains the meeting of the cluster and this warp's arrival at the closing one: the indices (a chain of divisions) are formed
// between the arrival at the meeting and the wait, and a warp arrives at the closing barrier as soon as its last loads from
// the peers are back, so that neither the divisions nor the output's arithmetic and stores lie on the way.
// What bounds it is the bytes that cross between the SMs: 16 per cycle and SM, whatever instruction moves them (32 KB in
// 2170 cycles by loads, bulk copies and asynchronous stores alike; by way of L2 3400).  So a rank's own partial does not
// cross, only rows that exist are dealt out to the ranks, a thread keeps to one row and fetches its (m, l) once, and each
// rank goes on from its own partial to the next rank's, so that the ranks do not all read from the same one.
template <int ROWS, int HD, int NT = 256>
__device__ __forceinline__ void cluster_merge(const Tc5Params& p, const Seg& sg, int ck, int cr, uint32_t pbuf_a, uint32_t pst_a, int st, volatile int* abort_flag) {
    cluster_arrive_release();
    constexpr int C4 = HD / 4;                                          // column quads of a row
    const int N = p.N, G = p.Hq / p.Hkv;
    const int rows = min(ROWS, G * N - sg.mblock * ROWS);               // of this unit
    const int rp = (rows + ck - 1) / ck, row0 = cr * rp, nrows = max(1, min(rp, rows - row0));
    const bool any = row0 < rows;                                       // (fewer rows than ranks: the last ranks have none)
    const int part = st / nrows, r = st - part * nrows, tpr = min(NT / nrows, C4);   // threads st < tpr * nrows, tpr to a row
    const bool mine = any && part < tpr;
    const int grow = sg.mblock * ROWS + row0 + r, node = grow / G, head = sg.kvh * G + (grow - node * G);
    __nv_bfloat16* orow = p.out + (((size_t)sg.b * N + node) * p.Hq + head) * HD;
    auto peer = [&](int j) { const int x = cr + j; return (uint32_t)(x >= ck ? x - ck : x); };
    // bit j of parts: rank peer(j) had steps.  (In short calls some have none: rank x's share [ceil(x s / ck), ceil((x + 1) s / ck)) of
    // s < ck steps is empty unless x s % ck is 0 or above ck - s.)
    unsigned parts = (1u << ck) - 1;
    if (sg.steps < ck) {
        unsigned has = 0;
        for (int x = 0, m = 0; x < ck; ++x) {
            if (m == 0 || m + sg.steps > ck) has |= 1u << x;
            m += sg.steps;
            if (m >= ck) m -= ck;
        }
        if (sg.steps == 0) has = 0;
        parts &= (has >> cr) | (has << (ck - cr));
    }
    if (!mine) parts = 0;
    cluster_wait();
    if (*abort_flag) { cluster_arrive_release(); return; }
    const uint32_t prow = pbuf_a + (uint32_t)((part * ROWS + row0 + r) * 16), prow_ml = pst_a + (uint32_t)((row0 + r) * 8);
    // IT column quads at a time per thread, all loads of all KM pieces issued before the first use
    auto merge_rows = [&](auto km_tag, auto it_tag) {
        constexpr int KM = decltype(km_tag)::value, IT = decltype(it_tag)::value;
        float w[KM], mm, ll;
        for (int e0 = 0;; e0 += IT) {
            float2 ml[KM];
            if (e0 == 0) {
#pragma unroll
                for (int j = 0; j < KM; ++j) {
                    ml[j] = make_float2(-INFINITY, 0.f);
                    if ((parts >> j) & 1) ml[j] = j == 0 ? smem_ld2(prow_ml) : dsmem_ld2(dsmem_addr(prow_ml, peer(j)));
                }
            }
            float4 pv[IT][KM];
#pragma unroll
            for (int e = 0; e < IT; ++e)
#pragma unroll
                for (int j = 0; j < KM; ++j) {
                    pv[e][j] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (((parts >> j) & 1) && part + tpr * (e0 + e) < C4)
                        pv[e][j] = j == 0 ? smem_ld4(prow + (uint32_t)(tpr * (e0 + e) * ROWS * 16))
                                          : dsmem_ld4(dsmem_addr(prow + (uint32_t)(tpr * (e0 + e) * ROWS * 16), peer(j)));
                }
            const bool last = tpr * (e0 + IT) >= C4;
            if (last) cluster_arrive_release();
            if (e0 == 0) {
                mm = -INFINITY; ll = 0.f;
#pragma unroll
                for (int j = 0; j < KM; ++j) mm = fmaxf(mm, ml[j].x);
                const float m_fin = (mm == -INFINITY) ? 0.f : mm;
#pragma unroll
                for (int j = 0; j < KM; ++j) { w[j] = exp2f(ml[j].x - m_fin); ll += ml[j].y * w[j]; }   // 0 for an empty or absent part
                const float inv = inv_sum(ll);
#pragma unroll
                for (int j = 0; j < KM; ++j) w[j] *= inv;
            }
#pragma unroll
            for (int e = 0; e < IT; ++e) {
                const int c4 = part + tpr * (e0 + e);
                if (!mine || c4 >= C4) continue;
                float4 a4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int j = 0; j < KM; ++j) {
                    a4.x += w[j] * pv[e][j].x; a4.y += w[j] * pv[e][j].y; a4.z += w[j] * pv[e][j].z; a4.w += w[j] * pv[e][j].w;
                }
                *reinterpret_cast<uint2*>(orow + c4 * 4) = make_uint2(pack_bf16(a4.x, a4.y), pack_bf16(a4.z, a4.w));
            }
            if (last) break;
        }
        if (p.lse && mine && part == 0)
            p.lse[((size_t)sg.b * p.Hq + head) * N + node] = ll > 0.f ? (mm + log2f(ll)) * 0.6931471805599453f : -INFINITY;
    };
    if (ck <= 2) merge_rows(std::integral_constant<int, 2>{}, std::integral_constant<int, 4>{});
    else if (ck <= 4) merge_rows(std::integral_constant<int, 4>{}, std::integral_constant<int, 4>{});
    else if (tpr >= C4) merge_rows(std::integral_constant<int, 8>{}, std::integral_constant<int, 1>{});
    else merge_rows(std::integral_constant<int, 8>{}, std::integral_constant<int, 2>{});
}

// Merge of the partials of every unit that more than one CTA worked on, 4 warps per block.  Q = 0, coarse: grid (unit, group
// of 32 rows x group of 64 columns), lane <-> row, a warp sums 16 output columns over the unit's segments four at a time -
// for units cut into a few pieces.  Q = 1, 2, 4, 8, fine: grid (unit, group of 32/Q rows x group of 16 columns), Q lanes share
// a row, a warp sums 4 output columns - for units cut over many CTAs (few sequences, long caches), where the rounds of
// loads are what the merge takes: qwen3b_S32768_N16_B1 (2 units over 148 CTAs, 74 partials each) 42.7 us per layer coarse,
// 28.1 with Q = 1, 19.7 with Q = 8; with many units of two partials the coarse shape is 3 % faster.
// The blocks are small: they are launched early (programmatic dependent launch) and must not keep the next layer's
// attention CTAs off the SMs.
template <int ROWS, int Q, int HD>
__global__ void __launch_bounds__(128)
attn_tc5_merge_kernel(const Tc5Params p) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_launch_dependents();
    // The schedule, recomputed per thread from kv_len (which the attention kernel does not write) without
    // shared memory: beside a resident attention CTA an SM has no shared memory to spare.
    constexpr bool LOCK = ROWS == 256;                 // (p.lock, known at compile time)
    const int upb = p.Hkv * p.n_mblocks, spb = LOCK ? p.Hkv : upb;      // units / units of the schedule per sequence
    const int unit = blockIdx.x, b = unit / upb, uib = unit - b * upb;
    int T = 0, live = 0, base_b = 0, steps = 0;
    for (int bb = 0; bb < p.B; ++bb) {
        const int S = p.kv_len[bb];
        const int st = (S >= 0 && S + p.N <= p.S_max) ? (S + p.N + p.step - 1) / p.step : 0;
        if (bb == b) { base_b = T; steps = st; }
        T += st > 0 ? (st + p.seg_cost) * spb : 0;
        live += st > 0 ? spb : 0;
    }
    // Everything that does not hang on the partials comes ahead of the dependency, down to the first group's addresses (each
    // behind a division); every block waits, also one with nothing to do: what follows on the stream waits for this kernel only.
    if (steps == 0) { pdl_wait(); return; }
    const int geff = sched_ctas(T, live, LOCK ? p.grid_attn / p.n_mblocks : p.grid_attn, p.min_steps, sched_round_steps(p));
    const int ub = base_b + (LOCK ? uib / p.n_mblocks : uib) * (steps + p.seg_cost), u0 = ub + p.seg_cost;   // where the unit starts, its first step
    const int c0 = cta_of(u0, T, geff), c1 = cta_of(u0 + steps - 1, T, geff);
    if (c0 == c1) { pdl_wait(); return; }              // one CTA had the whole unit and wrote the output itself
    const int G = p.Hq / p.Hkv, N = p.N;
    const int kvh = uib / p.n_mblocks, mblock = uib - kvh * p.n_mblocks;
    constexpr int CB = Q > 0 ? HD / 16 : HD / 64, RW = Q > 0 ? 32 / Q : 32;     // blocks and rows per group of rows
    const int lrow = (blockIdx.y / CB) * RW + lane % RW;
    const int cw = (blockIdx.y % CB) * 4 + warp;       // which 4 (fine) or 16 output columns
    const int row = mblock * ROWS + lrow;
    const bool row_ok = row < G * N;
    const int node = row_ok ? row / G : 0, head = kvh * G + (row_ok ? row % G : 0);

    const int smul = LOCK ? p.n_mblocks : 1, sadd = LOCK ? mblock : 0;
    if constexpr (Q > 0)
        merge_row_c4<ROWS, HD, Q>(p.part_o, p.part_ml, p.out, p.lse, T, geff, ub, c0, c1, b, node, head, p.Hq, N, lrow, cw, lane / RW, row_ok, smul, sadd);
    else
        merge_row_cols<ROWS, HD, true>(p.part_o, p.part_ml, p.out, p.lse, T, geff, ub, c0, row_ok ? c1 : c0 - 1, b, node, head, p.Hq, N, lrow, cw, smul, sadd);
}

// Host side: the merge of `units` units written by `ctas` CTAs; as many lanes share a row as keep the grid within what
// starts at once beside the next call's CTAs (8 units of 128 rows: 512 blocks with Q = 2; 1024 with Q = 4 took 3 us more).
constexpr int kMergeBlocks = 512;
template <int ROWS, int HD>
cudaError_t launch_merge(const Tc5Params& p, int units, int ctas, cudaStream_t st) {
    auto go = [&](auto q) {
        constexpr int Q = decltype(q)::value;
        constexpr int GY = Q > 0 ? ROWS * Q / 32 * (HD / 16) : ROWS / 32 * (HD / 64);
        return launch_pdl(attn_tc5_merge_kernel<ROWS, Q, HD>, dim3(units, GY), dim3(128), 0, st, 0, p);
    };
    const long long blocks = (long long)units * (ROWS / 32) * (HD / 16);       // at Q = 1
    if (ctas < 4 * units || blocks > 2 * kMergeBlocks) return go(std::integral_constant<int, 0>{});
    if (blocks * 8 <= kMergeBlocks) return go(std::integral_constant<int, 8>{});
    if (blocks * 4 <= kMergeBlocks) return go(std::integral_constant<int, 4>{});
    if (blocks * 2 <= kMergeBlocks) return go(std::integral_constant<int, 2>{});
    return go(std::integral_constant<int, 1>{});
}
// Per-device set-up of those kernels: the merge blocks ask for the split of shared memory and L1 that the attention CTAs have
// configured, so that an SM takes them as soon as its attention CTA has left, and the next call's CTA after them.  (Beside an attention
// CTA there is room for neither a merge block nor one of the rotation: 16 bytes of shared memory and 1024 registers.)
template <int ROWS, int HD>
cudaError_t init_merge() {
    const void* kernels[5] = {(const void*)attn_tc5_merge_kernel<ROWS, 0, HD>, (const void*)attn_tc5_merge_kernel<ROWS, 1, HD>,
                              (const void*)attn_tc5_merge_kernel<ROWS, 2, HD>, (const void*)attn_tc5_merge_kernel<ROWS, 4, HD>, (const void*)attn_tc5_merge_kernel<ROWS, 8, HD>};
    for (const void* k : kernels) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace tc5
}  // namespace vispec
