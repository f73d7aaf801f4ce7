// Tree-verification attention for sm_100a (D = 128 and 64): TMA-staged K/V tiles, tcgen05 tensor-core products
// with fp32 accumulators in TMEM, fp32 online softmax (Eq. 1 restricted to prefix + ancestors), work split
// over the SMs.
//
// Work.  A *unit* is (sequence, kv head, block of <= 128 query rows, rows ordered node-major so that all heads
// and nodes of a head group share every K/V tile); it needs ceil((S+N)/128) *steps*, one per 128 cached
// tokens.  Two ways to spread the units over the CTAs (at most one CTA per SM):
//   cluster form     one thread-block cluster of k <= 8 CTAs per unit; the CTA of rank r takes the r-th of k
//                    equal parts of the unit's steps and parks its unnormalised partial (O, m, l) in its own
//                    shared memory; after a hardware cluster barrier rank r merges rows [r*rows/k, ...) of all
//                    k partials through distributed shared memory and writes them out.  One launch.
//   even split       all steps of all units, in the order (sequence, kv head, row block, step), form one line
//                    of T steps cut into equal ranges, one per CTA (the CTA count is a multiple of the unit
//                    count when the units are fewer than the SMs, so that equally long units are cut into
//                    whole CTAs).  A CTA runs a few *segments*: the tail of one unit, whole units, the head of
//                    another.  A segment that covers its whole unit writes the final bf16 output; any other
//                    writes a partial into one of the CTA's two slots (first segment -> slot 2c, a later one
//                    -> slot 2c+1) and a second, small kernel merges the partials of each unit.
// Both kernels derive the schedule from kv_len on the device, so the host never reads lengths.
//
// Inside a CTA the 12 warps are specialised:
//   warp 0     TMA producer: K ring and V ring of 128-token stages (3 x 32 KB each, 128-byte swizzle, evict-first
//              in L2; head size 64: 6 x 16 KB); it runs ahead across segment boundaries
//   warp 1     issuer of S = Q K^T as 128x128x16 tcgen05.mma (the warp walks the steps and waits, one elected lane
//              issues); owns the TMEM allocation
//   warp 2     issuer of O += P V, likewise; the two chains wait on different barriers, so each has its own warp and
//              neither's waits delay the other's instructions.  With the fused rotary embedding it also tells the ranks of the
//              cluster that this one's tree rows are placed
//   warp 3     derives the schedule from kv_len; with at most 64 rows per unit (its lane 0 in the cluster form of a
//              contiguous cache, else the whole warp) and on pools of 16-row blocks it then produces the V ring, so that
//              warp 0's K copies never queue behind a wait for a V stage
//   warps 4-11 softmax: thread <-> TMEM lane; warps w and w+4 share the same 32 accumulator rows and each takes
//              half of a step's columns (the row maximum is exchanged through shared memory), so a row costs
//              no shuffles; they also load Q at the start of every segment (a later segment's comes through the K ring) and run
//              the segment epilogue.  Units of 128 rows in the cluster form: the two groups take alternate steps instead, and warp 1
//              issues all products (alternate_softmax, alternate_issue)
// TMEM map (512 columns x 128 lanes): S[0] 0..127, S[1] 128..255, O 256..383, P[0] 384..447, P[1] 448..511.
// P (bf16, packed two per column) is the A operand of the PV product and never touches shared memory; Q
// sits in shared memory in the same swizzled K-major layout as a K stage.  S and P are double-buffered: S
// is released as soon as the softmax threads have read it, so the S product of step u+1 and the PV
// product of step u-1 run while step u is in the softmax.
//
// Two row layouts share the code:
//   FULL  (G*N > 64):  lane r holds query row r of the block.
//   PAIR  (G*N <= 64): the <= 64 query rows are duplicated, lanes 0-63 take tokens 0-63 of each step and
//                      lanes 64-127 tokens 64-127 (P is block-diagonal); the two halves keep independent
//                      softmax states and are merged once per segment through shared memory.
// The running maximum is only moved when a tile exceeds it by more than 2^8 (O and l share the reference, so
// the result is exact either way); O is therefore re-scaled in TMEM rarely.
//
// Programmatic dependent launch: every launch carries the programmatic stream serialisation attribute.  The
// attention kernel reads kv_len and (when early prefetch is on) streams K/V tiles that lie wholly inside the
// committed prefix before it waits for the preceding kernel; q, tree_mask, the tree's own K/V rows and every
// write come after that wait.
//
// Every wait on an mbarrier is bounded; on a timeout the CTA records VISPEC_E_TIMEOUT, drains its own
// copies, frees its TMEM and returns.  The cluster form's hardware cluster barriers (two; three phases with the
// fused rotary embedding, whose first is arrived at after set-up and waited for by whole warps before their first
// signal to a peer) are reached by every thread of every CTA of the cluster (all other waits being bounded), so
// they end.
//
// Fused rotary embedding (ROPE instantiations, cluster form, contiguous caches): each rank of a unit's cluster
// rotates and places its share of the unit's N tree rows beside its (rotating) Q load and tells every rank; the
// producers hold back the tiles that contain those slots until all ranks have told.
#include <cuda_bf16.h>
#include <cstdio>
#include <cstdlib>
#include <type_traits>

#include "tc5_common.cuh"

namespace vispec {

using namespace tc5;

namespace {

constexpr int STAGE_BYTES = 2 * HALF_BYTES;    // 32 KB
constexpr int NSK = 3, NSV = 3;
constexpr int kThreads = 384;                  // 12 warps: producer, two issuers, one spare, eight softmax
constexpr int kSmx = 256;                      // softmax threads
constexpr int SMEM_K = 0;
constexpr int SMEM_V = SMEM_K + NSK * STAGE_BYTES;
constexpr int SMEM_Q = SMEM_V + NSV * STAGE_BYTES;             // Q tile, 128 rows, laid out like a K stage; between
                                                               // segments it is the PAIR exchange [32 col4][64 rows] float4
constexpr int SMEM_XM = SMEM_Q + STAGE_BYTES;                  // 512 floats: tile maxima / row statistics exchanged between threads
constexpr int SMEM_BAR = SMEM_XM + 2048;
constexpr int BAR_BYTES = 352;
constexpr int SMEM_SCHED = SMEM_BAR + BAR_BYTES;
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t COL_S = 0, COL_O = 256, COL_P = 384;

constexpr int kMaxRing = 2 * NSK;              // stages of a ring at head size 64: half the bytes each, twice as many
enum { B_KFULL = 0, B_KEMPTY = B_KFULL + kMaxRing, B_VFULL = B_KEMPTY + kMaxRing, B_VEMPTY = B_VFULL + kMaxRing,
       B_SFULL = B_VEMPTY + kMaxRing, B_SFREE = B_SFULL + 2, B_PFULL = B_SFREE + 2, B_PVDONE = B_PFULL + 2,
       B_QFULL = B_PVDONE + 2, B_PAIRX = B_QFULL + 1, B_XCH = B_PAIRX + 4, B_XFREE = B_XCH + 1,
       B_SEGSYNC = B_XFREE + 1,
       B_ROWS = B_SEGSYNC + 1,      // fused rotary embedding: every rank of the cluster has put its share of the tree rows into the cache
       B_COUNT = B_ROWS + 1 };
static_assert(B_COUNT * 8 + 20 <= BAR_BYTES, "barrier block too small");

// the rings' geometry, for the paged producer
struct Ring128 {
    static constexpr int NSK = 3, NSV = 3, STAGE = STAGE_BYTES, OFF_K = SMEM_K, OFF_V = SMEM_V;
    static constexpr int KFULL = B_KFULL, KEMPTY = B_KEMPTY, VFULL = B_VFULL, VEMPTY = B_VEMPTY;
};

constexpr int SMEM_TABRING = SMEM_SCHED + ((int)sizeof(Sched) + 15) / 16 * 16;   // 8 steps x 8 block numbers (paged cache)
constexpr int SMEM_TOTAL = SMEM_TABRING + 256;
constexpr int SMEM_ALLOC = SMEM_TOTAL;                         // the base must come out 1024-byte aligned (checked)
static_assert(SMEM_ALLOC <= 232448, "over the 227 KB a CTA may have");

// ---- fused rotary embedding ---------------------------------------------------------------------------
// Pairs (x = element j of the lower half, y = element j + D/2) rotated by their angles: fp64 with one rounding to bf16 for
// the k rows that go to the cache (two pairs), fp32 for q rows (eight pairs; consumed by the product, never stored).
__device__ __forceinline__ void rope2_f64(uint32_t& lo, uint32_t& hi, const double2* cs) {
    __nv_bfloat16* a = reinterpret_cast<__nv_bfloat16*>(&lo);
    __nv_bfloat16* b = reinterpret_cast<__nv_bfloat16*>(&hi);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const double x = (double)__bfloat162float(a[t]), y = (double)__bfloat162float(b[t]);
        a[t] = __double2bfloat16(x * cs[t].x - y * cs[t].y);
        b[t] = __double2bfloat16(y * cs[t].x + x * cs[t].y);
    }
}
__device__ __forceinline__ void rope8_f32(uint4& lo, uint4& hi, const float2* cs) {
    __nv_bfloat16* a = reinterpret_cast<__nv_bfloat16*>(&lo);
    __nv_bfloat16* b = reinterpret_cast<__nv_bfloat16*>(&hi);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const float x = __bfloat162float(a[t]), y = __bfloat162float(b[t]);
        a[t] = __float2bfloat16_rn(x * cs[t].x - y * cs[t].y);
        b[t] = __float2bfloat16_rn(y * cs[t].x + x * cs[t].y);
    }
}
// Prologue of a CTA with the fused rotary embedding (one function, so that both memory round trips overlap): the upper
// half of the softmax threads fetches this rank's share of the tree rows, tree index in [t_lo, t_hi), of (sequence b,
// kv head kvh), and every thread its part of the Q tile; then the k rows are rotated (fp64, one rounding: bit-compatible with
// the rotation kernel) and written to slots S + t of the cache with the v rows, and the Q rows are rotated (fp32: they feed
// the score product only) into the swizzled tile.  Shares of more than 16 rows take further passes after that.  Not
// inlined: its registers stay out of the step loop's budget and its code out of the step loop's way.
// What bounds it is the load path's lines per instruction and the registers of what is in flight, most of it angles (16 bytes
// per k pair, 8 per q pair, against 4 of data).  So the eight threads of a k row take pairs 2c + 16u, 2c + 1 + 16u of it (neighbours
// read neighbouring angles), and a thread's Q rows follow one another, so that they belong to one node or two and share its angles:
// everything is in flight at once also with 128 rows per unit.
template <bool PAIR, int ROWS>
__device__ __noinline__ void rope_prologue(unsigned char* sm, const __nv_bfloat16* __restrict__ q, const RopeArgs p, int N_, int Hq,
                                           int Hkv_, int S_max_, int G, int rows_total, int b, int kvh, int mblock, int S,
                                           int t_lo, int t_hi, int st) {
    constexpr int HALF = kSmx / 2;
    const int ps = st - HALF;                     // >= 0: this thread places rows
    const size_t cache_row0 = ((size_t)b * Hkv_ + kvh) * S_max_ + S;
    const int nk = (t_hi - t_lo) * 8, nv = (t_hi - t_lo) * 16;
    uint32_t klo[4], khi[4];                      // pairs 2c + 16u, 2c + 1 + 16u of row t_lo + i / 8, c = i % 8
    double2 cs[4][2];
    uint4 vx[2];
    auto k_load = [&](int i) {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(p.k_new + (((size_t)b * N_ + t_lo + (i >> 3)) * Hkv_ + kvh) * D) + (i & 7);
        const double2* tab = p.rope_k + ((size_t)b * N_ + t_lo + (i >> 3)) * (D / 2) + 2 * (i & 7);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            klo[u] = src[8 * u]; khi[u] = src[8 * u + D / 4];
            cs[u][0] = tab[16 * u]; cs[u][1] = tab[16 * u + 1];
        }
    };
    auto k_store = [&](int i) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(p.k_cache + (cache_row0 + t_lo + (i >> 3)) * D) + (i & 7);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            rope2_f64(klo[u], khi[u], cs[u]);
            dst[8 * u] = klo[u]; dst[8 * u + D / 4] = khi[u];
        }
    };
    auto v_load = [&](int i) { return reinterpret_cast<const uint4*>(p.v_new + (((size_t)b * N_ + t_lo + (i >> 4)) * Hkv_ + kvh) * D)[i & 15]; };
    auto v_store = [&](int i, const uint4& x) { reinterpret_cast<uint4*>(p.v_cache + (cache_row0 + t_lo + (i >> 4)) * D)[i & 15] = x; };
    auto rows_load = [&](int i, int j) {
        if (i < nk) k_load(i);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (j + HALF * u < nv) vx[u] = v_load(j + HALF * u);
    };
    auto rows_store = [&](int i, int j) {
        if (i < nk) k_store(i);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (j + HALF * u < nv) v_store(j + HALF * u, vx[u]);
    };

    // K rows of the Q tile from row r0 on, one or two nodes' worth: chunk pair (c, c + 8) of each.
    const int c = st & 7;
    auto q_rows = [&](auto k_tag, int r0, auto between) {
        constexpr int K = decltype(k_tag)::value;
        uint4 lo[K], hi[K];
        float4 tab[2][4];
        const int row0 = mblock * ROWS + r0, n0 = row0 / G, n1 = min(row0 + K - 1, rows_total - 1) / G;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int row = row0 + k;
            lo[k] = make_uint4(0, 0, 0, 0); hi[k] = lo[k];
            if (row < rows_total) {
                const int node = row / G;
                const uint4* src = reinterpret_cast<const uint4*>(q + (((size_t)b * N_ + node) * Hq + kvh * G + (row - node * G)) * D);
                lo[k] = src[c]; hi[k] = src[c + 8];
            }
        }
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const float4* t4 = reinterpret_cast<const float4*>(p.rope_q + ((size_t)b * N_ + (x ? n1 : n0)) * (D / 2) + 8 * c);
#pragma unroll
            for (int j = 0; j < 4; ++j) tab[x][j] = make_float4(1.f, 0.f, 1.f, 0.f);
            if (row0 < rows_total && (x == 0 || n1 != n0)) {
#pragma unroll
                for (int j = 0; j < 4; ++j) tab[x][j] = t4[j];
            }
        }
        between();
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool second = row0 + k >= (n0 + 1) * G;
            float4 t[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                t[j] = second ? tab[1][j] : tab[0][j];
            rope8_f32(lo[k], hi[k], reinterpret_cast<const float2*>(t));
            const int r = r0 + k;
            unsigned char* dst = sm + SMEM_Q + r * 128 + ((c ^ (r & 7)) << 4);
            *reinterpret_cast<uint4*>(dst) = lo[k];
            *reinterpret_cast<uint4*>(dst + HALF_BYTES) = hi[k];
            if (PAIR) {
                *reinterpret_cast<uint4*>(dst + 64 * 128) = lo[k];
                *reinterpret_cast<uint4*>(dst + HALF_BYTES + 64 * 128) = hi[k];
            }
        }
    };
    constexpr int K = ROWS * 8 / kSmx;            // Q rows of a thread: (st / 8) * K ...
    if (ps >= 0) rows_load(ps, ps);
    auto finish_rows = [&]() { if (ps >= 0) rows_store(ps, ps); };
    if (K <= 2 || G >= K - 1) {                   // K rows in a row touch at most two nodes
        q_rows(std::integral_constant<int, K>{}, (st >> 3) * K, finish_rows);
    } else {
        q_rows(std::integral_constant<int, 2>{}, (st >> 3) * K, finish_rows);
        q_rows(std::integral_constant<int, 2>{}, (st >> 3) * K + 2, []() {});
    }
    // tree rows beyond the first 16 of the share
    if (ps >= 0)
        for (int i = ps + HALF, j = ps + 2 * HALF; i < nk || j < nv; i += HALF, j += 2 * HALF) {
            rows_load(i, j);
            rows_store(i, j);
        }
}

// The softmax's exponentials are what the special-function pipe (16 lanes per SM) spends a step on; one in eight of them is
// formed on the FMA pipe instead: in the duplicated-row layout and in alternate steps two neighbouring columns of every sixteen by one
// packed evaluation, in the even split with 128 rows, where two threads share a row, one column of every eight (packed in that loop, which
// then served clusters too: 517.6 against 507.1 us per pass on qwen3b_S8192_N60_B4).  Measured on the loop with two threads per row,
// none / 1 in 16 / 1 in 8, us per pass: llava7b 559.6 / 558.4 / 550.3, qwen3b_S8192_N60_B4 532.1 / 526.1 / 507.1, qwen7b fused
// 455.3 / 454.8 / 451.8; 1 in 6 moves nothing, 1 in 4 and 1 in 2 are slower (issue slots).
constexpr int kPolyEvery = 4;

// ---- 128 rows per unit in the cluster form: two groups of softmax warps on alternate steps ----------------------
// With two threads per row (below) all eight warps move in lock-step: they wait, load and exchange maxima together, and meanwhile
// neither the special-function pipe nor the tensor pipe has work (2240 cycles per step, of which the exponentials are 1024 and the
// products 1024).  Here a row belongs to one thread of each group of four warps; group x takes the steps of parity x whole, with a
// reference maximum, a sum and an accumulator of its own (added up at the end), so nothing is exchanged, and while one group is in
// its exponentials the products of the other run.  P overwrites S, which makes room for the second accumulator; one warp issues all
// products, S(0) S(1) | PV(0) S(2) | PV(1) S(3) | ...: S(t + 2) overwrites P(t) behind PV(t), which reads it, and its completion, for which
// a commit also waits for all that was issued before, tells that PV(t) is complete.  That the overwriting product does not overtake the
// reading one rests on how the tensor core works - one CTA's products start in the order of issue -, not on a documented guarantee, which
// covers products of one shape on one accumulator (test_products_in_shared_tensor_memory_repeat_bit_for_bit looks; the two-tile kernel rests
// on the same).  A wait for PV(t) ahead of S(t + 2): 16 query and 2 kv heads, 4 x 60 nodes on 8192 tokens 443.7 -> 450.5 us per pass of 16
// layers, 8 x 128 on 4096 385.1 -> 388.8, 28 / 4 heads, 1 x 128 on 8192 408.0 -> 413.7, head size 64 no change.  1880 cycles per step (qwen3b_S8192_N60_B4 485 -> 465 us per pass; tensor pipe active 35 %
// of a launch against 31 %).  What is left is a group's chain, products of its own step and of the other group's among it, and beside
// it shared memory, whose 128 bytes per cycle feed both operands of S (512 cycles), V (256) and the copies coming in (512).  In the even
// split, whose CTAs have fewer steps here, the longer first step costs more than the loop gains (qwen3b_S32768_N16_B1 324 -> 329),
// and rows <= 64, where a thread has half the columns, gain 0.5 % and lose 2.5 % in the smallest calls: both keep two threads per row.
// TMEM: S_0 0..127, S_1 128..255 (P of the step in the first 64 columns of its S), O_0 256, O_1 384.
enum { B_PHALF0 = B_PFULL, B_PHALF1 = B_SFREE };     // halves of P, by accumulator (128 arrivals)

template <int HD>
__device__ __forceinline__ void alternate_issue(uint32_t base, uint32_t bars, uint32_t tmem, int n_, volatile int* abort_flag) {
    constexpr int NH = HD / 64, STAGE = NH * HALF_BYTES, NSK = kMaxRing / NH, NSV = kMaxRing / NH;
    constexpr uint32_t IDESC_S = instr_desc(0), IDESC_O = instr_desc(1, HD);   // B = K stage, K-major; V stage, MN-major
    constexpr uint32_t DESC_HI = desc_hi(1024);
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    const bool leader = elect_one();
    const int n = __shfl_sync(0xffffffffu, n_, 0);
    const uint32_t k0 = desc_lo(base + SMEM_K, 16), v0 = desc_lo(base + SMEM_V, HALF_BYTES), qb = desc_lo(base + SMEM_Q, 16);
    uint32_t sk = 0, pk = 0, sv = 0, pv = 0;                    // ring positions with their phases
    // A wait costs 150 cycles also where the answer is there.  So what a step needs is asked for ahead, without blocking, between
    // the last step's PV and S products, whose issue takes long enough for the answers to come; only where the answer was no it is
    // waited for.
    bool k_ok = false, v_ok = false, p_ok[2] = {false, false};
    auto have = [&](bool asked, uint32_t b, uint32_t phase) {
        return __all_sync(0xffffffffu, asked) || mbar_wait_warp(b, phase, abort_flag);
    };
    auto score = [&](uint32_t x) {                             // S_x = Q K^T
        if (!have(k_ok, bar(B_KFULL) + 8u * sk, pk)) return false;
        k_ok = false;
        tc_fence_after();
        if (leader) {
            const uint32_t kb = k0 + sk * (STAGE >> 4), d = tmem + COL_S + x * 128;
#pragma unroll
            for (int ks = 0; ks < HD / 16; ++ks) {             // 16 d-columns per instruction: 32 B of each Q and K row
                const uint32_t koff = ((ks >> 2) * HALF_BYTES + (ks & 3) * 32) >> 4;
                tc_mma_ss(d, qb + koff, DESC_HI, kb + koff, DESC_HI, IDESC_S, ks > 0 ? 1u : 0u);
            }
            tc_commit(bar(B_SFULL) + 8u * x);
            tc_commit(bar(B_KEMPTY) + 8u * sk);
        }
        if (++sk == NSK) { sk = 0; pk ^= 1; }
        return true;
    };
    if (!mbar_wait_warp(bar(B_QFULL), 0, abort_flag)) return;
    if (n > 0 && !score(0)) return;
    if (n > 1 && !score(1)) return;
    for (int t = 0; t < n; ++t) {
        const uint32_t x = t & 1;
        if (t + 2 < n) k_ok = mbar_test(bar(B_KFULL) + 8u * sk, pk);
        if (!have(v_ok, bar(B_VFULL) + 8u * sv, pv)) return;
        const uint32_t vb = v0 + sv * (STAGE >> 4), pb = tmem + COL_S + x * 128, d = tmem + COL_O + x * 128;
#pragma unroll
        for (int h = 0; h < 2; ++h) {                          // O_x += P_x V(step), each half of the tokens as soon as its P is there
            if (!have(p_ok[h], bar(h ? B_PHALF1 : B_PHALF0) + 8u * x, (t >> 1) & 1)) return;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int ks = 4 * h; ks < 4 * h + 4; ++ks)     // 16 tokens per instruction: 8 P columns, 16 V rows (2 KB)
                    tc_mma_ts(d, pb + ks * 8, vb + ks * 128, DESC_HI, IDESC_O, (t > 1 || ks > 0) ? 1u : 0u);
            }
        }
        if (leader) {
            tc_commit(bar(B_VEMPTY) + 8u * sv);
            tc_commit(bar(B_PVDONE) + 8u * x);
        }
        if (++sv == NSV) { sv = 0; pv ^= 1; }
        v_ok = p_ok[0] = p_ok[1] = false;
        if (t + 1 < n) {
            v_ok = mbar_test(bar(B_VFULL) + 8u * sv, pv);
            p_ok[0] = mbar_test(bar(B_PHALF0) + 8u * (x ^ 1), ((t + 1) >> 1) & 1);
            p_ok[1] = mbar_test(bar(B_PHALF1) + 8u * (x ^ 1), ((t + 1) >> 1) & 1);
        }
        if (t + 2 < n && !score(x)) return;
    }
}

// One softmax thread's row of the segment (lane tl, group x), down to the partial parked in shared memory.  False: a wait gave up.
template <int HD>
__device__ __forceinline__ bool alternate_softmax(unsigned char* sm, uint32_t bars, uint32_t tmem, const Seg& sg, int N, float scale_log2,
                                                  uint64_t mk0, uint64_t mk1, bool row_ok, int x, int tl, volatile int* abort_flag) {
    constexpr int NH = HD / 64, STAGE = NH * HALF_BYTES, NSV = kMaxRing / NH, ROWS = 128;
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    const uint32_t lane_addr = tmem + ((uint32_t)(tl & ~31) << 16), s_addr = lane_addr + COL_S + x * 128, o_addr = lane_addr + COL_O + x * 128;
    const int S = sg.S, total = S + N;
    float m_ref = -INFINITY, l_run = 0.f;
    bool has_o = false;
    for (int t = x; t < sg.n; t += 2) {
        const int tok0 = (sg.st0 + t) * STEP;
        // (this product was issued after this group's last PV product, so that one is complete too: O_x and P are free)
        if (!mbar_wait_warp(bar(B_SFULL + x), (t >> 1) & 1, abort_flag)) return false;
        tc_fence_after();
        const bool tail = tok0 + STEP > S;                     // reaches past the committed prefix: ancestor bits
        uint64_t a0 = 0, a1 = 0;                               // bit c: column c may be attended to (prefix column, or visible tree node)
        if (tail) {
            const int t0 = tok0 - S;                           // tree index of column 0 (may be negative)
            if (t0 >= 0) shr128(mk0, mk1, t0, a0, a1); else shl128_fill(mk0, mk1, -t0, a0, a1);
        }
        // The row is read in halves of 64 columns, the upper half twice (held whole it would take the registers of both).
        uint32_t s[64];
        auto load_half = [&](int h) {
            tmem_ld32(s_addr + h * 64, s);
            tmem_ld32(s_addr + h * 64 + 32, s + 32);
            tmem_wait_ld();
            if (tail) {
                const uint64_t a = h ? a1 : a0;
#pragma unroll
                for (int c = 0; c < 64; ++c)
                    if (!((a >> c) & 1ull)) s[c] = 0xff800000u;   // -inf
            }
        };
        float mx[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) mx[e] = -INFINITY;
#pragma unroll 1
        for (int h = 1; h >= 0; --h) {
            load_half(h);
#pragma unroll
            for (int c = 0; c < 64; c += 16)
#pragma unroll
                for (int e = 0; e < 8; ++e) mx[e] = max3_nan(mx[e], __uint_as_float(s[c + e]), __uint_as_float(s[c + 8 + e]));
        }
        // the scale is positive, so it commutes with the maximum
        const float tmax = max_nan(max3_nan(max3_nan(mx[0], mx[1], mx[2]), max3_nan(mx[3], mx[4], mx[5]), mx[6]), mx[7]) * scale_log2;
        // move the reference maximum only when the tile exceeds it by more than the gap
        float alpha = 1.f;
        bool rescale = false;
        if (tmax > m_ref + kRescaleGap) {                      // also true on the first finite tile (m_ref = -inf)
            alpha = exp2f(m_ref - tmax);                       // 0 when m_ref = -inf
            m_ref = tmax;
            l_run *= alpha;
            rescale = has_o;
        }
        if (!(tmax < INFINITY)) l_run = tmax - tmax;            // a NaN or an infinite score: the row is NaN (see inv_sum)
        if (__any_sync(0xffffffffu, rescale)) {
#pragma unroll
            for (int c = 0; c < HD / 16; ++c) {
                uint32_t o[16];
                tmem_ld16(o_addr + c * 16, o);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                tmem_st16(o_addr + c * 16, o);
            }
        }
        bool fail = false;
        if (tok0 + STEP > total) {
            // last step of the sequence: V rows past the last key may hold anything, and they meet weight-0 columns of P in the
            // product: clear them (lane r clears row r)
            const int sv = t % NSV;
            fail = !mbar_wait(bar(B_VFULL + sv), (t / NSV) & 1, abort_flag);
            if (!fail && tok0 + tl >= total) {
                unsigned char* vrow = sm + SMEM_V + sv * STAGE + tl * 128;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    *reinterpret_cast<uint4*>(vrow + c * 16) = make_uint4(0, 0, 0, 0);
                    if (NH == 2) *reinterpret_cast<uint4*>(vrow + HALF_BYTES + c * 16) = make_uint4(0, 0, 0, 0);
                }
            }
            fence_async_smem();
        }
        if (__any_sync(0xffffffffu, fail)) return false;
        // P = exp2(scale * s - m_ref) as bf16 pairs (column c of P holds tokens 2c, 2c+1), handed on by halves
        const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
        const uint64_t sc2 = pk2(scale_log2, scale_log2), mm2 = pk2(-m_use, -m_use);
        uint64_t sum2 = pk2(0.f, 0.f), sum2b = sum2;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            if (h == 1) load_half(1);                          // (P of the first half lies in columns 0..31)
            uint32_t pd[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                float x0, x1, e0, e1;
                up2(fma2(pk2(__uint_as_float(s[2 * c]), __uint_as_float(s[2 * c + 1])), sc2, mm2), x0, x1);
                if (c % (2 * kPolyEvery) == 2 * kPolyEvery - 1) exp2_fma_pair(x0, x1, e0, e1);
                else { e0 = exp2f(x0); e1 = exp2f(x1); }
                if (c & 1) sum2b = add2(sum2b, pk2(e0, e1)); else sum2 = add2(sum2, pk2(e0, e1));
                pd[c] = pack_bf16(e0, e1);
            }
            tmem_st32(s_addr + h * 32, pd);
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar(h ? B_PHALF1 : B_PHALF0) + 8u * x);
        }
        float l0, l1;
        up2(add2(sum2, sum2b), l0, l1);
        l_run += l0 + l1;
        has_o = true;
    }

    // The row's statistics, of both groups, go round while the last products run; then this thread adds up columns
    // [HD/2 x, HD/2 x + HD/2) of the lane's two accumulators and parks them over the K ring, [HD/4 col4][ROWS].
    float* xm = reinterpret_cast<float*>(sm + SMEM_XM);       // [group][lane] l, then the same of m
    xm[x * 128 + tl] = l_run;
    xm[256 + x * 128 + tl] = has_o ? m_ref : -INFINITY;
    mbar_arrive(bar(B_XCH));
    // (everybody past its last step: every product but each accumulator's last PV is complete, and a wait can tell the phase it
    // waits for from the one before)
    if (!mbar_wait_warp(bar(B_XCH), 0, abort_flag)) return false;
#pragma unroll
    for (int y = 0; y < 2; ++y) {
        const int t = sg.n - 1 - ((sg.n - 1 - y) & 1);         // the accumulator's last step
        if (t >= 0 && !mbar_wait_warp(bar(B_PVDONE + y), (t >> 1) & 1, abort_flag)) return false;
    }
    tc_fence_after();
    const float m0 = xm[256 + tl], m1 = xm[384 + tl], m_all = fmaxf(m0, m1), m_fin = (m_all == -INFINITY) ? 0.f : m_all;
    const float w0 = exp2f(m0 - m_fin), w1 = exp2f(m1 - m_fin);   // 0 where nothing was seen
    const float l_all = xm[tl] * w0 + xm[128 + tl] * w1;
    float4* prow = reinterpret_cast<float4*>(sm + SMEM_K) + (size_t)x * (HD / 8) * ROWS + tl;
#pragma unroll
    for (int cc = 0; cc < HD / 2; cc += 32) {
        uint32_t o0[32], o1[32];
        tmem_ld32(lane_addr + COL_O + x * (HD / 2) + cc, o0);
        tmem_ld32(lane_addr + COL_O + 128 + x * (HD / 2) + cc, o1);
        tmem_wait_ld();
        float v[32];
        // (an accumulator is only defined once a product has run: select, never multiply, where the weight is zero)
#pragma unroll
        for (int e = 0; e < 32; ++e)
            v[e] = (w0 > 0.f ? __uint_as_float(o0[e]) * w0 : 0.f) + (w1 > 0.f ? __uint_as_float(o1[e]) * w1 : 0.f);
        if (row_ok) {
#pragma unroll
            for (int c4 = 0; c4 < 8; ++c4)
                prow[(size_t)(cc / 4 + c4) * ROWS] = make_float4(v[4 * c4], v[4 * c4 + 1], v[4 * c4 + 2], v[4 * c4 + 3]);
        }
    }
    tc_fence_before();
    if (x == 0 && row_ok)
        reinterpret_cast<float2*>(sm + SMEM_K + (HD / 4) * ROWS * 16)[tl] = make_float2(l_all > 0.f ? m_all : -INFINITY, l_all);
    return true;
}

// PAGED instantiations carry the paged producer; the others are compiled without it (its call sites cost the
// contiguous kernels registers they do not have to spare).
template <bool PAIR, bool CL, bool PAGED, bool ROPE = false, int HD = 128>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc5_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap v_map, const Tc5Params p,
                const std::conditional_t<ROPE, RopeArgs, PagedArgs> pa) {
    static_assert(!(ROPE && PAGED), "the fused rotary embedding serves contiguous caches");
    static_assert(!ROPE || CL, "the fused rotary embedding exists in the cluster form only (the even split goes through the rotation kernel)");
    static_assert(HD == 128 || (HD == 64 && !PAGED && !ROPE), "head size 64: plain calls on contiguous caches");
    // A stage holds NH halves of 64 d-columns.  At head size 64 the rings have twice the stages, so that the bytes in flight
    // per SM stay the same; the scores cost half the product, the softmax is unchanged, O has half the columns.
    // Against the mma.sync kernel and its merge that served head size 64 before (us per layer, mask and commit aside): 38 -> 17
    // at 8 sequences x 4 heads x 67 nodes on 3325 tokens, 86 -> 51 at 6 x 16 heads (4 kv) x 128 nodes on 2300-4096.
    constexpr int D = HD, NH = HD / 64, STAGE_BYTES = NH * HALF_BYTES, NSK = kMaxRing / NH, NSV = kMaxRing / NH;
    constexpr int ROWS = PAIR ? 64 : 128;      // distinct query rows per CTA
    constexpr int NC = PAIR ? 32 : 64;         // tokens of a step one softmax thread handles (two threads per row)
    constexpr bool ALT = CL && !PAIR;          // alternate steps instead (alternate_softmax)
    // The V ring can have a producer of its own, the spare warp (its lane 0; paged: all of it).  With at most 64 rows per
    // unit it always has; with 128 only for pools of 16-row blocks, where one warp issuing a step's 32 copies is what
    // holds the call back (larger blocks lose 1 % with two producers, like the contiguous cache).
    constexpr bool SPLIT_V = PAIR || PAGED;
    bool split_v = PAIR;
    if constexpr (PAGED && !PAIR) split_v = pa.page_rows <= 16;
    extern __shared__ __align__(1024) unsigned char sm[];
    // the schedule hangs on kv_len, and a CTA that starts after its predecessor kernel has ended hangs on the
    // schedule: the load goes out first
    int kv_first = 0;
    if (p.early && threadIdx.x >= 96 && threadIdx.x < 128 && (int)threadIdx.x - 96 < p.B) kv_first = p.kv_len[threadIdx.x - 96];
    const uint32_t base = smem_u32(sm);
    if (base & 1023u) {
        // the swizzled tiles need a 1024-byte aligned base; every CTA sees the same base, so all of them leave
        if (threadIdx.x == 0) atomicCAS(p.status, 0, (int)VISPEC_E_UNSUPPORTED);
        return;
    }
    const uint32_t bars = base + SMEM_BAR;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + SMEM_BAR + B_COUNT * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + SMEM_BAR + B_COUNT * 8 + 8);
    volatile int* seg_flag = abort_flag + 1;               // this CTA delivered the last partial of the unit just finished
    Sched& sched = *reinterpret_cast<Sched*>(sm + SMEM_SCHED);
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int cta = blockIdx.x;
    const int G = p.Hq / p.Hkv, N = p.N, W = (N + 63) >> 6;
    const int rows_total = G * N;

    if (tid == 0) {
        for (int i = 0; i < NSK; ++i) { mbar_init(bar(B_KFULL + i), 1); mbar_init(bar(B_KEMPTY + i), 1); }
        for (int i = 0; i < NSV; ++i) { mbar_init(bar(B_VFULL + i), 1); mbar_init(bar(B_VEMPTY + i), 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(B_SFULL + i), 1); mbar_init(bar(B_SFREE + i), ALT ? 128 : kSmx);
            mbar_init(bar(B_PFULL + i), ALT ? 128 : kSmx); mbar_init(bar(B_PVDONE + i), 1);
        }
        for (int i = 0; i < 4; ++i) mbar_init(bar(B_PAIRX + i), 64);
        mbar_init(bar(B_QFULL), kSmx);
        mbar_init(bar(B_XCH), kSmx); mbar_init(bar(B_XFREE), kSmx);
        mbar_init(bar(B_SEGSYNC), kSmx);
        if (ROPE) mbar_init(bar(B_ROWS), cluster_size());
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (!p.early) {                                          // nothing is read before the preceding kernel has ended
        pdl_wait();
        if (warp == 3 && lane < p.B) kv_first = p.kv_len[lane];
    }
    pdl_launch_dependents();
    if (warp == 3) sched_build(sched, p, lane, kv_first);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Fused rotary embedding: the ranks signal one another's barriers, which must exist by then.  Everybody arrives at
    // the cluster barrier here (relaxed: fence.mbarrier_init has published the barriers); a warp waits, as a whole,
    // where it first needs the guarantee.
    bool cl_waited = !ROPE;
    if (ROPE) cluster_arrive();

    // Schedule.  Cluster form: cluster <-> unit, the CTA of rank r takes the r-th of k equal parts of the
    // unit's steps (an empty part still takes part in the exchange).  Otherwise: equal ranges of the line of
    // all steps.
    const int T = sched.base[p.B];
    const int geff = CL ? (int)gridDim.x : (T > 0 ? sched_ctas(T, sched.units, (int)gridDim.x, p.min_steps, sched_round_steps(p)) : 0);
    const bool active = cta < geff;
    const int lo = (!CL && active) ? cta_lo(cta, T, geff) : 0, hi = (!CL && active) ? cta_lo(cta + 1, T, geff) : 0;
    const uint32_t tmem = *tmem_slot;
    const int ck = CL ? (int)cluster_size() : 1, cr = CL ? (int)cluster_ctarank() : 0;
    Seg cl_seg = {};
    if (CL) {
        const int upb = p.Hkv * p.n_mblocks;
        const int unit = cta / ck, b = unit / upb, uib = unit - b * upb;
        cl_seg.b = b; cl_seg.kvh = uib / p.n_mblocks; cl_seg.mblock = uib - cl_seg.kvh * p.n_mblocks;
        cl_seg.steps = sched.steps[b]; cl_seg.S = sched.len[b];
        // (the first ranks get the odd steps: the last one has the tree's tiles, which cannot be fetched ahead and cost a mask;
        // qwen3b_S2048_N16_B1 9.7 -> 8.9 us per layer, qwen7b 14.5 -> 13.7)
        cl_seg.st0 = (cr * cl_seg.steps + ck - 1) / ck;
        cl_seg.n = ((cr + 1) * cl_seg.steps + ck - 1) / ck - cl_seg.st0;
        cl_seg.slot = -1;
    }
    using Iter = SegIter<PAIR && !CL>;
    auto make_iter = [&]() {
        Iter it; it.s = &sched; it.B = p.B; it.n_mblocks = p.n_mblocks; it.seg_cost_ = p.seg_cost; it.g = lo; it.lo = lo; it.hi = hi; it.cta = cta;
        it.cl = CL; it.cl_done = false; it.cl_seg = cl_seg;
        return it;
    };

    auto prod_wait = [&](uint32_t bar_addr, uint32_t parity) -> bool {     // by one lane in the cluster form, by the warp otherwise
        const bool r = mbar_wait(bar_addr, parity, abort_flag);
        return CL ? r : (bool)__all_sync(0xffffffffu, r);
    };
    if (warp == 0) {
        // ================= TMA producer =================
        // Paged: the whole warp, each lane one block of a step.  Contiguous, even split: the whole warp with one elected lane
        // issuing, as the product issuers do (qwen3b_S32768_N16_B1 29.1 -> 28.1 us per layer, llava13b_b4 65.7 -> 64.7);
        // in the cluster form one lane (2 x 60 nodes at head size 64 lose 1 % otherwise, the rest does not move).
        if ((PAGED || !CL || lane == 0) && active) {
            const bool leader = (CL && !PAGED) || elect_one();
            const uint64_t pol = l2_evict_first_policy();
            bool waited = !p.early;
            int it = 0, nk = 0, nv = 0;          // steps started; K stages used (one per step, one per later segment's Q), V stages issued
            bool ok = true;
            Iter si = make_iter();
            Seg sg;
            // Even split: the Q rows of a CTA's later segments come through the K ring, one stage ahead of the segment's first K tile,
            // so that they are there when the segment before ends (a round trip to memory behind a saturated HBM is 3.5 us; a
            // CTA's every further segment cost 7 us with it, for which its rings stood still: llava13b_b4's CTAs ended after 41, 49
            // or 56 us by the number of their segments, and with the rows sent ahead after 44, 49 or 54).  The softmax threads copy them on into the Q tile.
            auto q_stage = [&](const Seg& sg) -> bool {
                const int sk = nk % NSK, r_n = min(ROWS, rows_total - sg.mblock * ROWS);
                if (!waited) { pdl_wait(); waited = true; }
                if (!prod_wait(bar(B_KEMPTY + sk), ((nk / NSK) & 1) ^ 1)) return false;
                if (leader) mbar_expect_tx(bar(B_KFULL + sk), (uint32_t)r_n * D * 2);
                __syncwarp();
                for (int r = lane; r < r_n; r += 32) {
                    const int row = sg.mblock * ROWS + r;
                    bulk_load(base + SMEM_K + sk * STAGE_BYTES + r * (D * 2), p.q + (((size_t)sg.b * N + row / G) * p.Hq + sg.kvh * G + row % G) * D,
                              D * 2, bar(B_KFULL + sk));
                }
                ++nk;
                return true;
            };
            if constexpr (PAGED) {
                for (int seg = 0; ok && si.next(sg); ++seg) {
                    const QStage qs = {p.q, p.Hq, G, sg.mblock * ROWS, !CL && seg > 0 ? min(ROWS, rows_total - sg.mblock * ROWS) : 0};
                    const uint32_t r = produce_paged<Ring128>(pa, &k_map, &v_map, sg.b, sg.kvh, sg.st0, sg.n, sg.S, base, bars, base + SMEM_TABRING, abort_flag, pol, it, waited, lane, split_v ? 1 : 0, nk - it, qs);
                    const int done = (int)(r & 0x0fffffffu);
                    it += done; nv += split_v ? 0 : done; nk += done + (int)((r >> 28) & 1u) + (int)(r >> 31);
                    ok = !((r >> 29) & 1u);
                    waited = (r >> 30) & 1u;
                }
            }
            for (int seg = 0; !PAGED && ok && si.next(sg); ++seg) {
                if (!CL && seg > 0 && !q_stage(sg)) { ok = false; break; }
                const int bh = sg.b * p.Hkv + sg.kvh;
                const int n = CL ? sg.n : __shfl_sync(0xffffffffu, sg.n, 0);
                for (int t = 0; t < n; ++t, ++it) {
                    const int tok = (sg.st0 + t) * STEP;
                    if (!waited && tok + STEP > sg.S) { pdl_wait(); waited = true; }   // the tree's rows come from the preceding kernel
                    if (ROPE && tok + STEP > sg.S) {
                        // the tile holds tree rows: every rank's share must be in the cache, and ordered before this copy
                        if (!mbar_wait_cluster(bar(B_ROWS), 0, abort_flag)) { ok = false; break; }
                        asm volatile("fence.proxy.async.global;" ::: "memory");
                    }
                    const int sk = nk % NSK;
                    if (!prod_wait(bar(B_KEMPTY + sk), ((nk / NSK) & 1) ^ 1)) { ok = false; break; }
                    if (leader) {
                        mbar_expect_tx(bar(B_KFULL + sk), STAGE_BYTES);
                        tma_load_3d(base + SMEM_K + sk * STAGE_BYTES, &k_map, bar(B_KFULL + sk), 0, tok, bh, pol);
                        if constexpr (NH == 2) tma_load_3d(base + SMEM_K + sk * STAGE_BYTES + HALF_BYTES, &k_map, bar(B_KFULL + sk), 64, tok, bh, pol);
                    }
                    ++nk;
                    if constexpr (!SPLIT_V) {
                        const int sv = it % NSV;
                        if (!prod_wait(bar(B_VEMPTY + sv), ((it / NSV) & 1) ^ 1)) { ok = false; break; }
                        if (leader) {
                            mbar_expect_tx(bar(B_VFULL + sv), STAGE_BYTES);
                            tma_load_3d(base + SMEM_V + sv * STAGE_BYTES, &v_map, bar(B_VFULL + sv), 0, tok, bh, pol);
                            if constexpr (NH == 2) tma_load_3d(base + SMEM_V + sv * STAGE_BYTES + HALF_BYTES, &v_map, bar(B_VFULL + sv), 64, tok, bh, pol);
                        }
                        ++nv;
                    }
                }
            }
            if (*abort_flag && lane == 0) {
                // drain: wait (bounded, fresh timer) until every copy this warp issued has landed
                volatile int never = 0;
                for (int u = max(0, nk - NSK); u < nk; ++u) mbar_wait(bar(B_KFULL + u % NSK), (u / NSK) & 1, &never);
                for (int u = max(0, nv - NSV); u < nv; ++u) mbar_wait(bar(B_VFULL + u % NSV), (u / NSV) & 1, &never);
            }
        }
        __syncwarp();
    } else if (warp == 3) {
        // ================= TMA producer of the V ring (contiguous caches, rows <= 64) =================
        // A V stage is free only after the PV product of the step it held, a softmax later than the K stage of the
        // same step: one thread issuing both in order holds the K copies back behind every wait for a V stage.
        // Measured in one call, one thread against two: 17.70 -> 17.50 us per layer on llava7b, 17.11 -> 16.91 on
        // paper_tree, 71.4 -> 71.0 on llava13b_b4; with 128 rows per unit the two threads lose 1 % (16.43 -> 16.59 on
        // qwen7b, 63.3 -> 63.8 on qwen3b_S32768_N16_B8), so those keep the single producer.
        if constexpr (SPLIT_V && PAGED) {
            if (active && split_v) {
                const uint64_t pol = l2_evict_first_policy();
                bool waited = !p.early, ok = true;
                int it = 0;
                Iter si = make_iter();
                Seg sg;
                while (ok && si.next(sg)) {
                    const uint32_t r = produce_paged<Ring128>(pa, &k_map, &v_map, sg.b, sg.kvh, sg.st0, sg.n, sg.S, base, bars, base + SMEM_TABRING + 128, abort_flag, pol, it, waited, lane, 2);
                    it += (int)(r & 0x0fffffffu);
                    ok = !((r >> 29) & 1u);
                    waited = (r >> 30) & 1u;
                }
                if (*abort_flag && lane == 0) {
                    volatile int never = 0;
                    for (int u = max(0, it - NSV); u < it; ++u) mbar_wait(bar(B_VFULL + u % NSV), (u / NSV) & 1, &never);
                }
            }
        } else if (SPLIT_V && (!CL || lane == 0) && active) {
            const bool leader = CL || elect_one();
            const uint64_t pol = l2_evict_first_policy();
            bool waited = !p.early;
            int it = 0;
            bool ok = true;
            Iter si = make_iter();
            Seg sg;
            while (ok && si.next(sg)) {
                const int bh = sg.b * p.Hkv + sg.kvh;
                const int n = CL ? sg.n : __shfl_sync(0xffffffffu, sg.n, 0);
                for (int t = 0; t < n; ++t, ++it) {
                    const int tok = (sg.st0 + t) * STEP;
                    if (!waited && tok + STEP > sg.S) { pdl_wait(); waited = true; }
                    if (ROPE && tok + STEP > sg.S) {
                        if (!mbar_wait_cluster(bar(B_ROWS), 0, abort_flag)) { ok = false; break; }
                        asm volatile("fence.proxy.async.global;" ::: "memory");
                    }
                    const int sv = it % NSV;
                    if (!prod_wait(bar(B_VEMPTY + sv), ((it / NSV) & 1) ^ 1)) { ok = false; break; }
                    if (leader) {
                        mbar_expect_tx(bar(B_VFULL + sv), STAGE_BYTES);
                        tma_load_3d(base + SMEM_V + sv * STAGE_BYTES, &v_map, bar(B_VFULL + sv), 0, tok, bh, pol);
                        if constexpr (NH == 2) tma_load_3d(base + SMEM_V + sv * STAGE_BYTES + HALF_BYTES, &v_map, bar(B_VFULL + sv), 64, tok, bh, pol);
                    }
                }
            }
            if (*abort_flag && lane == 0) {
                volatile int never = 0;
                for (int u = max(0, it - NSV); u < it; ++u) mbar_wait(bar(B_VFULL + u % NSV), (u / NSV) & 1, &never);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= issuer of the S products =================
        // The whole warp walks through the steps and waits, one elected lane issues: with uniform control flow the
        // descriptors live in uniform registers, where the instructions take them from.  Against one lane doing it all:
        // llava7b 16.7 -> 16.2 us per layer, qwen7b 15.2 -> 14.5, qwen3b_S8192_N60_B4 31.3 -> 29.7, qwen3b_S32768_N16_B1 29.2 -> 28.9.
        if constexpr (ALT) {
            alternate_issue<HD>(base, bars, tmem, cl_seg.n, abort_flag);
        } else if (active) {
            constexpr uint32_t IDESC_S = instr_desc(0);            // B = K stage, K-major
            constexpr uint32_t DESC_HI = desc_hi(1024);            // 8 rows x 128 B between row groups, everywhere
            const bool leader = elect_one();
            const uint32_t k0 = desc_lo(base + SMEM_K, 16), qb = desc_lo(base + SMEM_Q, 16);
            bool ok = true;
            uint32_t sk = 0, pk = 0, it = 0, seg = 0;              // ring position with its phase, steps, segments
            Iter si = make_iter();
            Seg sg;
            while (ok && si.next(sg)) {
                const int n = __shfl_sync(0xffffffffu, sg.n, 0);
                if (!mbar_wait_warp(bar(B_QFULL), seg & 1, abort_flag)) { ok = false; break; }
                if (!CL && seg > 0) {                                  // the stage that the Q rows came in has been read
                    if (leader) mbar_arrive(bar(B_KEMPTY) + 8u * sk);
                    if (++sk == NSK) { sk = 0; pk ^= 1; }
                }
                for (int t = 0; t < n; ++t, ++it) {
                    const uint32_t bs = it & 1;
                    if (!mbar_wait_warp(bar(B_KFULL) + 8u * sk, pk, abort_flag)) { ok = false; break; }
                    // S[bs] is free once the softmax threads have read the scores of step it-2 out of it
                    if (it >= 2 && !mbar_wait_warp(bar(B_SFREE) + 8u * bs, ((it >> 1) - 1) & 1, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    if (leader) {
                        const uint32_t kb = k0 + sk * (STAGE_BYTES >> 4), d = tmem + COL_S + bs * 128;
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks) {      // 16 d-columns per instruction: 32 B of each Q and K row
                            const uint32_t koff = ((ks >> 2) * HALF_BYTES + (ks & 3) * 32) >> 4;
                            tc_mma_ss(d, qb + koff, DESC_HI, kb + koff, DESC_HI, IDESC_S, ks > 0 ? 1u : 0u);
                        }
                        tc_commit(bar(B_SFULL) + 8u * bs);
                        tc_commit(bar(B_KEMPTY) + 8u * sk);
                    }
                    if (++sk == NSK) { sk = 0; pk ^= 1; }
                }
                ++seg;
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ================= issuer of the PV products =================
        if (active) {
            constexpr uint32_t IDESC_O = instr_desc(1, D);         // B = V stage, MN-major
            constexpr uint32_t DESC_HI = desc_hi(1024);
            const bool leader = elect_one();
            const uint32_t v0 = desc_lo(base + SMEM_V, HALF_BYTES);
            bool ok = true;
            if constexpr (ROPE) {
                // Each rank of the cluster puts its share of the unit's N tree rows into the cache (its softmax threads, beside
                // their Q tile).  The ranks whose steps contain the rows (the last, at most the last two) hold those tiles back
                // until every rank has said that its share is in global memory: meeting of this CTA's softmax threads, fence,
                // then one arrival per rank on that rank's barrier.  By this warp, which waits for the first P anyway: the fence
                // (it covers what the meeting has made visible to this thread) and the signals held the softmax threads back
                // ahead of their first step.
                cluster_wait();                                           // the peers' barriers exist
                cl_waited = true;
                if (lane < ck) {
                    ok = mbar_wait(bar(B_SEGSYNC), 0, abort_flag);
                    if (ok) {
                        __threadfence();                                          // the rows are in global memory ...
                        asm volatile("fence.proxy.async.global;" ::: "memory");   // ... and ordered before bulk copies that read them
                        mbar_arrive_peer(dsmem_addr(bar(B_ROWS), (uint32_t)lane));
                    }
                }
                ok = __all_sync(0xffffffffu, ok);
            }
            if constexpr (ALT) ok = false;                                // (warp 1 issues these products too)
            uint32_t sv = 0, pv = 0, u = 0;
            Iter si = make_iter();
            Seg sg;
            while (ok && si.next(sg)) {
                const int n = __shfl_sync(0xffffffffu, sg.n, 0);
                for (int t = 0; t < n; ++t, ++u) {
                    const uint32_t bu = u & 1;
                    if (!mbar_wait_warp(bar(B_PFULL) + 8u * bu, (u >> 1) & 1, abort_flag)) { ok = false; break; }
                    if (!mbar_wait_warp(bar(B_VFULL) + 8u * sv, pv, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    if (leader) {
                        const uint32_t vb = v0 + sv * (STAGE_BYTES >> 4), pb = tmem + COL_P + bu * 64;
#pragma unroll
                        for (int ks = 0; ks < STEP / 16; ++ks)      // 16 tokens per instruction: 8 P columns, 16 V rows (2 KB)
                            tc_mma_ts(tmem + COL_O, pb + ks * 8, vb + ks * 128, DESC_HI, IDESC_O,
                                      (t > 0 || ks > 0) ? 1u : 0u);   // the first product of a segment starts a fresh O
                        tc_commit(bar(B_VEMPTY) + 8u * sv);
                        tc_commit(bar(B_PVDONE) + 8u * bu);
                    }
                    if (++sv == NSV) { sv = 0; pv ^= 1; }
                }
            }
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ================= softmax: two threads per accumulator row, each takes half of a step's columns =================
        const int sp = warp & 3;                              // TMEM lane quarter of this warp
        const int ch = (warp - 4) >> 2;                       // which half of the row's columns (and of the O columns)
        const int tl = sp * 32 + lane;                        // TMEM lane
        const int half = PAIR ? (tl >> 6) : 0;                // PAIR: which 64 tokens of each step the lane's row copy covers
        const int lrow = PAIR ? (tl & 63) : tl;               // row within the block
        const uint32_t lane_addr = tmem + ((uint32_t)(32 * sp) << 16);
        const int st = tid - 128;                             // 0..255
        float* xm = reinterpret_cast<float*>(sm + SMEM_XM);   // [2 step parities][2 column halves][128 lanes] tile maxima;
                                                              // in the epilogue: [0..255] l by (ch, lane), [256..383] m by lane
        int px = 0;                                           // phases of the pair barrier used so far
        int sx = 0;                                           // phases of the segment barrier used so far
        // Where this thread's chunks of the Q tile come from: (sequence, node, head) rows, -1 past the last.  The cluster
        // form's one segment is known before the wait, and so are these.
        constexpr int QC = D / 8, QR = kSmx / QC, ITEMS = ROWS / QR;   // 16-byte chunks per row; rows per pass; passes
        const int qc = st % QC;
        int qrow[ITEMS];
        auto q_rows = [&](const Seg& sg) {
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const int row = sg.mblock * ROWS + st / QC + QR * k;
                qrow[k] = row < rows_total ? (sg.b * N + row / G) * p.Hq + sg.kvh * G + row % G : -1;
            }
        };
        // The ancestor bits of this thread's row, fetched beside the Q rows; where they are, -1 past the last row.
        int mrow = -1;
        uint64_t mk0 = 0, mk1 = 0;
        auto mask_row = [&](const Seg& sg) {
            const int row = sg.mblock * ROWS + lrow;
            mrow = row < rows_total ? (sg.b * N + row / G) * W : -1;
        };
        auto mask_fetch = [&]() {
            mk0 = mk1 = 0;
            if (mrow >= 0) {
                mk0 = p.mask[mrow];
                if (W > 1) mk1 = p.mask[mrow + 1];
            }
        };
        if (CL) { if (!ROPE) q_rows(cl_seg); mask_row(cl_seg); }
        pdl_wait();                                           // q, tree_mask and every output come after the preceding kernel

        // rejected sequences (kv_len < 0 or kv_len + N > S_max): zero output, -inf lse, status word
        zero_rejected<D>(p, sched, cta, st);

        // Q of a segment -> shared memory, rows in the swizzled K-major layout of a K stage (PAIR: rows 64-127
        // repeat rows 0-63).  Thread t moves 16-byte chunk t%16 of rows t/16, t/16 + 16, ... (head size 64: t%8 of t/8, t/8 + 32, ...)
        auto load_q = [&](const Seg& sg, int seg, int it) -> bool {
            if (PAIR && seg > 0) {
                // the tile doubles as the exchange area of the previous segment's epilogue
                if (!mbar_wait_warp(bar(B_XFREE), (seg - 1) & 1, abort_flag)) return false;
            }
            if constexpr (ROPE) {
                mask_fetch();
                // the Q tile and, beside it, this rank's share of the unit's tree rows into the cache (a rejected
                // sequence, steps == 0, has no slots to write to: an empty share)
                const int t_lo = (cr * N) / ck;
                rope_prologue<PAIR, ROWS>(sm, p.q, pa, N, p.Hq, p.Hkv, p.S_max, G, rows_total, sg.b, sg.kvh, sg.mblock, sg.S,
                                          t_lo, sg.steps > 0 ? ((cr + 1) * N) / ck : t_lo, st);
                fence_async_smem();
                mbar_arrive(bar(B_QFULL));
                return true;
            }
            uint4 v[ITEMS];
            if (CL || seg == 0) {
                if (!CL) { q_rows(sg); mask_row(sg); }
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) {
                    v[k] = make_uint4(0, 0, 0, 0);
                    if (qrow[k] >= 0) v[k] = *(reinterpret_cast<const uint4*>(p.q + (size_t)qrow[k] * D) + qc);
                }
                mask_fetch();
            } else {
                const int ik = it + seg - 1, sk = ik % NSK;          // the producer's stage for it
                if (!mbar_wait_warp(bar(B_KFULL + sk), (ik / NSK) & 1, abort_flag)) return false;
#pragma unroll
                for (int k = 0; k < ITEMS; ++k) {
                    const int r = st / QC + QR * k;
                    v[k] = make_uint4(0, 0, 0, 0);
                    if (sg.mblock * ROWS + r < rows_total) v[k] = *reinterpret_cast<const uint4*>(sm + SMEM_K + sk * STAGE_BYTES + r * (D * 2) + qc * 16);
                }
            }
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const int r = st / QC + QR * k;
                unsigned char* dst = sm + SMEM_Q + (qc >> 3) * HALF_BYTES + r * 128 + (((qc & 7) ^ (r & 7)) << 4);
                *reinterpret_cast<uint4*>(dst) = v[k];
                if (PAIR) *reinterpret_cast<uint4*>(dst + 64 * 128) = v[k];
            }
            fence_async_smem();
            mbar_arrive(bar(B_QFULL));
            return true;
        };
        // Meeting of the two warps that share this warp's rows (bounded; warp-uniform result).
        auto pair_sync = [&]() -> bool {
            mbar_arrive(bar(B_PAIRX + sp));
            const bool r = mbar_wait_warp(bar(B_PAIRX + sp), px & 1, abort_flag);
            ++px;
            return r;
        };

        if (PAIR && active) {
            // block-diagonal P: a lane's row copy weighs only its own half's 64 tokens of a step; the columns of the
            // other half are zero in both P buffers for the whole call, and nobody else writes them
            uint32_t zero[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) zero[c] = 0u;
            tmem_st16(lane_addr + COL_P + (half ^ 1) * 32 + ch * 16, zero);
            tmem_st16(lane_addr + COL_P + 64 + (half ^ 1) * 32 + ch * 16, zero);
            tmem_wait_st();
        }
        if (active) {
            Iter si = make_iter();
            Seg sg;
            int it = 0, seg = 0;
            bool ok = true;
            float4* xch = reinterpret_cast<float4*>(sm + SMEM_Q);
            while (ok && si.next(sg)) {
                // every S product of the previous segment has been consumed by now, so Q may be replaced
                if (!load_q(sg, seg, it)) { ok = false; break; }
                // (fused rotary embedding: this rank's share of the tree rows is stored; warp 2 tells the other ranks)
                if (ROPE) mbar_arrive(bar(B_SEGSYNC));

                const int row = sg.mblock * ROWS + lrow;         // query row within the kv head's G*N rows
                const bool row_ok = row < rows_total;
                const int node = row_ok ? row / G : 0, head = sg.kvh * G + (row_ok ? row % G : 0);
                const int S = sg.S, total = S + N;
                // bits at or beyond N are not tree nodes
                if (N < 64) mk0 &= (1ull << N) - 1;
                if (N < 128) mk1 &= N > 64 ? (1ull << (N - 64)) - 1 : 0ull;
                if constexpr (ALT) {
                    ok = alternate_softmax<HD>(sm, bars, tmem, sg, N, p.scale_log2, mk0, mk1, row_ok, ch, tl, abort_flag);
                    break;
                }
                // m_ref and has_o are the same in both threads of a row; l_run covers this thread's columns only
                float m_ref = -INFINITY, l_run = 0.f;
                bool has_o = false;

                for (int t = 0; t < sg.n; ++t, ++it) {
                    const int bs = it & 1;
                    const int tok0 = (sg.st0 + t) * STEP;
                    if (!mbar_wait_warp(bar(B_SFULL + bs), (it >> 1) & 1, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    uint32_t sraw[NC];
#pragma unroll
                    for (int c = 0; c < NC / 32; ++c) tmem_ld32(lane_addr + COL_S + bs * 128 + half * 64 + ch * NC + c * 32, sraw + c * 32);
                    tmem_wait_ld();
                    tc_fence_before();
                    mbar_arrive(bar(B_SFREE + bs));             // the S product of step it+2 may overwrite the buffer

                    const int jr = tok0 + half * 64;                        // first token of the row's part of the tile
                    const int j0 = jr + ch * NC;                            // first token this thread looks at
                    const bool row_valid = jr < total, valid = j0 < total;
                    float lmax = -INFINITY;
                    if (valid) {
                        if (j0 + NC > S) {
                            // reaches past the committed prefix: ancestor bits for tree rows, nothing beyond them
                            // bit c of a0: column c may be attended to (prefix column, or visible tree node)
                            const int t0 = j0 - S;                           // tree index of column 0 (may be negative)
                            uint64_t a0, a1;
                            if (t0 >= 0) shr128(mk0, mk1, t0, a0, a1); else shl128_fill(mk0, mk1, -t0, a0, a1);
#pragma unroll
                            for (int c = 0; c < NC; ++c)
                                if (!((a0 >> c) & 1ull)) sraw[c] = 0xff800000u;   // -inf
                        }
                        float mx[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) mx[c] = __uint_as_float(sraw[c]);
#pragma unroll
                        for (int c = 8; c < NC; ++c) mx[c & 7] = max_nan(mx[c & 7], __uint_as_float(sraw[c]));
                        // the scale is positive, so it commutes with the maximum
                        lmax = max_nan(max_nan(max_nan(mx[0], mx[1]), max_nan(mx[2], mx[3])), max_nan(max_nan(mx[4], mx[5]), max_nan(mx[6], mx[7]))) * p.scale_log2;
                    }
                    // the row's maximum over the tile: the other thread of the row has the other columns
                    xm[(it & 1) * 256 + ch * 128 + tl] = lmax;
                    if (!pair_sync()) { ok = false; break; }
                    const float tmax = max_nan(lmax, xm[(it & 1) * 256 + (ch ^ 1) * 128 + tl]);
                    // move the reference maximum only when the tile exceeds it by more than the gap
                    float alpha = 1.f;
                    bool rescale = false;
                    if (row_valid && tmax > m_ref + kRescaleGap) {      // also true on the first finite tile (m_ref = -inf)
                        alpha = exp2f(m_ref - tmax);                     // 0 when m_ref = -inf
                        m_ref = tmax;
                        l_run *= alpha;
                        rescale = has_o;
                    }
                    if (!(tmax < INFINITY)) l_run = tmax - tmax;             // a NaN or an infinite score: the row is NaN (see inv_sum)
                    if (__any_sync(0xffffffffu, rescale)) {
                        // O was last written by the PV product of step it-1 (same segment: has_o is set); this thread
                        // rescales its half of the row's columns
                        if (!mbar_wait_warp(bar(B_PVDONE + (bs ^ 1)), ((it - 1) >> 1) & 1, abort_flag)) { ok = false; break; }
                        tc_fence_after();
#pragma unroll
                        for (int c = 0; c < NH; ++c) {
                            uint32_t o[32];
                            tmem_ld32(lane_addr + COL_O + ch * (D / 2) + c * 32, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                            tmem_st32(lane_addr + COL_O + ch * (D / 2) + c * 32, o);
                        }
                    }
                    // P[bs] is free once the PV product of step it-2 has completed: as a rule it has, long ago, and one test
                    // issued here, ahead of the exponentials, says so without a wait after them
                    const bool p_free = it < 2 || mbar_test(bar(B_PVDONE + bs), ((it >> 1) - 1) & 1);
                    // P = exp2(scale * s - m_ref) as bf16 pairs (column c of P holds tokens 2c, 2c+1)
                    uint32_t pd[NC / 2];
                    if (valid) {
                        const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
                        float sum0 = 0.f, sum1 = 0.f;
#pragma unroll
                        for (int c = 0; c < NC / 2; ++c) {
                            const float x0 = fmaf(__uint_as_float(sraw[2 * c]), p.scale_log2, -m_use);
                            const float x1 = fmaf(__uint_as_float(sraw[2 * c + 1]), p.scale_log2, -m_use);
                            float e0, e1;
                            if (PAIR && c % (2 * kPolyEvery) == 2 * kPolyEvery - 1) {
                                exp2_fma_pair(x0, x1, e0, e1);
                            } else {
                                e0 = exp2f(x0);
                                e1 = (!PAIR && c % kPolyEvery == kPolyEvery - 1) ? exp2_fma(x1) : exp2f(x1);
                            }
                            sum0 += e0; sum1 += e1;
                            pd[c] = pack_bf16(e0, e1);
                        }
                        l_run += sum0 + sum1;
                    } else {
#pragma unroll
                        for (int c = 0; c < NC / 2; ++c) pd[c] = 0u;
                    }
                    if (row_valid) has_o = true;
                    if (it >= 2) {
                        if (!__all_sync(0xffffffffu, p_free) &&
                            !mbar_wait_warp(bar(B_PVDONE + bs), ((it >> 1) - 1) & 1, abort_flag)) { ok = false; break; }
                        tc_fence_after();
                    }
                    if (PAIR) {
                        // block-diagonal P: the row weighs only its own half's tokens (the other 32 columns stay zero)
                        tmem_st16(lane_addr + COL_P + bs * 64 + half * 32 + ch * 16, pd);
                    } else {
                        tmem_st32(lane_addr + COL_P + bs * 64 + ch * 32, pd);
                    }
                    bool fail = false;
                    if (tok0 + STEP > total) {
                        // last step of the sequence: V rows past the last key may hold anything, and they meet
                        // weight-0 columns of P in the product: clear them (thread r of the first 128 clears row r)
                        const int sv = it % NSV;
                        fail = !mbar_wait(bar(B_VFULL + sv), (it / NSV) & 1, abort_flag);
                        if (!fail && ch == 0 && tok0 + tl >= total) {
                            unsigned char* vrow = sm + SMEM_V + sv * STAGE_BYTES + tl * 128;
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                *reinterpret_cast<uint4*>(vrow + c * 16) = make_uint4(0, 0, 0, 0);
                                if (NH == 2) *reinterpret_cast<uint4*>(vrow + HALF_BYTES + c * 16) = make_uint4(0, 0, 0, 0);
                            }
                        }
                        fence_async_smem();
                    }
                    tmem_wait_st();
                    if (__any_sync(0xffffffffu, fail)) { ok = false; break; }
                    tc_fence_before();
                    mbar_arrive(bar(B_PFULL + bs));
                }
                if (!ok) break;
                // (the next segment's mask row is on its way from here on)
                if constexpr (!CL) {
                    Iter ahead = si;
                    Seg nx;
                    if (ahead.next(nx)) { mask_row(nx); mask_fetch(); }
                }

                // ---- segment epilogue: wait for the last product, add up the row statistics, (PAIR) merge the two
                // halves, write out.  FULL: a thread owns columns [D/2 ch, D/2 ch + D/2) of its lane's accumulator row.  PAIR:
                // the two lanes with copies of a row each take half of those columns and hand the other half over. ----
                if (sg.n > 0) ok = mbar_wait_warp(bar(B_PVDONE + ((it - 1) & 1)), ((it - 1) >> 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                constexpr int KC = PAIR ? D / 4 : D / 2;             // output columns of a thread, from col0 on
                const int col0 = ch * (D / 2) + (PAIR ? half * KC : 0);
                uint32_t o[KC];
                auto o_load = [&](int col) {
#pragma unroll
                    for (int c = 0; c < KC; c += KC < 32 ? 16 : 32) {
                        if constexpr (KC < 32) tmem_ld16(lane_addr + COL_O + col + c, o + c);
                        else tmem_ld32(lane_addr + COL_O + col + c, o + c);
                    }
                    tmem_wait_ld();
                };
                // (the tile-maximum slots are idle: the other thread of the row read its last one before it arrived
                // for the last PV product)
                xm[ch * 128 + tl] = l_run;
                if (ch == 0) xm[256 + tl] = has_o ? m_ref : -INFINITY;
                float w_me = has_o ? 1.f : 0.f, w_other = 0.f, m_all = has_o ? m_ref : -INFINITY, l_all;
                if (PAIR) {
                    // hand the raw accumulator of the other lane's columns to it (the Q tile is idle: every S product of the
                    // segment has completed)
                    const int give = ch * (D / 2) + (half ^ 1) * KC;
                    o_load(give);
#pragma unroll
                    for (int c4 = 0; c4 < KC / 4; ++c4)
                        xch[(give / 4 + c4) * 64 + lrow] = make_float4(__uint_as_float(o[4 * c4]), __uint_as_float(o[4 * c4 + 1]),
                                                                       __uint_as_float(o[4 * c4 + 2]), __uint_as_float(o[4 * c4 + 3]));
                    mbar_arrive(bar(B_XCH));
                    o_load(col0);
                    tc_fence_before();
                    if (!mbar_wait_warp(bar(B_XCH), seg & 1, abort_flag)) { ok = false; break; }
                    const float m_o = xm[256 + (tl ^ 64)], l_o = xm[tl ^ 64] + xm[128 + (tl ^ 64)];
                    m_all = fmaxf(m_all, m_o);
                    const float m_fin = (m_all == -INFINITY) ? 0.f : m_all;
                    w_me = has_o ? exp2f(m_ref - m_fin) : 0.f;
                    w_other = exp2f(m_o - m_fin);                   // 0 when the other half saw nothing
                    l_all = (xm[tl] + xm[128 + tl]) * w_me + l_o * w_other;
                } else {
                    mbar_arrive(bar(B_PAIRX + sp));
                    o_load(col0);
                    tc_fence_before();
                    if (!mbar_wait_warp(bar(B_PAIRX + sp), px & 1, abort_flag)) { ok = false; break; }
                    ++px;
                    l_all = xm[tl] + xm[128 + tl];
                }
                // O is only defined once a product has run (an empty cluster part never ran one): select, never
                // multiply, where the weight is zero
                const bool final_out = !CL && sg.slot < 0;
                const float inv = final_out ? inv_sum(l_all) : 1.f;
                float v[KC];
#pragma unroll
                for (int e = 0; e < KC; ++e) v[e] = has_o ? __uint_as_float(o[e]) * w_me : 0.f;
                if (PAIR) {
                    if (w_other > 0.f) {
#pragma unroll
                        for (int c4 = 0; c4 < KC / 4; ++c4) {
                            const float4 w = xch[(col0 / 4 + c4) * 64 + lrow];
                            v[4 * c4] += w.x * w_other; v[4 * c4 + 1] += w.y * w_other;
                            v[4 * c4 + 2] += w.z * w_other; v[4 * c4 + 3] += w.w * w_other;
                        }
                    }
                }
                if (final_out) {
                    if (row_ok) {
                        __nv_bfloat16* orow = p.out + (((size_t)sg.b * N + node) * p.Hq + head) * D + col0;
#pragma unroll
                        for (int c8 = 0; c8 < KC / 8; ++c8)
                            *reinterpret_cast<uint4*>(orow + c8 * 8) =
                                make_uint4(pack_bf16(v[8 * c8] * inv, v[8 * c8 + 1] * inv), pack_bf16(v[8 * c8 + 2] * inv, v[8 * c8 + 3] * inv),
                                           pack_bf16(v[8 * c8 + 4] * inv, v[8 * c8 + 5] * inv), pack_bf16(v[8 * c8 + 6] * inv, v[8 * c8 + 7] * inv));
                    }
                } else if (row_ok) {
                    // cluster form: parked in this CTA's shared memory, [D/4 col4][ROWS] over the K ring
                    float4* prow = (CL ? reinterpret_cast<float4*>(sm + SMEM_K) : p.part_o + (size_t)sg.slot * (D / 4) * ROWS) + (size_t)(col0 / 4) * ROWS + lrow;
#pragma unroll
                    for (int c4 = 0; c4 < KC / 4; ++c4)
                        prow[(size_t)c4 * ROWS] = make_float4(v[4 * c4], v[4 * c4 + 1], v[4 * c4 + 2], v[4 * c4 + 3]);
                }
                if (ch == 0 && half == 0 && row_ok) {
                    const float2 stat = make_float2(l_all > 0.f ? m_all : -INFINITY, l_all);
                    if (CL) {
                        reinterpret_cast<float2*>(sm + SMEM_K + (D / 4) * ROWS * 16)[lrow] = stat;      // [ROWS] (m, l)
                    } else if (final_out) {
                        if (p.lse) p.lse[((size_t)sg.b * p.Hq + head) * N + node] =
                            l_all > 0.f ? (m_all + log2f(l_all)) * 0.6931471805599453f : -INFINITY;
                    } else {
                        p.part_ml[(size_t)sg.slot * ROWS + lrow] = stat;
                    }
                }
                if (PAIR) mbar_arrive(bar(B_XFREE));
                if constexpr (PAIR && !CL) if (pa.unit_counters && sg.slot >= 0) {
                    // ---- even split without a merge kernel (rows <= 64 only: with 128 rows the merge kernel is faster): the CTA that delivers a unit's last partial merges the
                    // unit.  Nobody waits for another CTA: a fence, one atomic per segment, and the last arrival
                    // reads the others' partials (written before their fences) from L2. ----
                    __threadfence();
                    mbar_arrive(bar(B_SEGSYNC));                       // every softmax thread has written and fenced
                    if (!mbar_wait_warp(bar(B_SEGSYNC), sx & 1, abort_flag)) { ok = false; break; }
                    ++sx;
                    const int uib = sg.kvh * p.n_mblocks + sg.mblock;
                    const int ub = sched.base[sg.b] + uib * (sg.steps + p.seg_cost), u0 = ub + p.seg_cost;
                    const int c0 = cta_of(u0, T, geff), c1 = cta_of(u0 + sg.steps - 1, T, geff);
                    if (st == 0) {
                        int* cnt = pa.unit_counters + (sg.b * p.Hkv * p.n_mblocks + uib);
                        const bool last = atomicAdd(cnt, 1) == c1 - c0;
                        if (last) *cnt = 0;                            // all zero again for the next call
                        *seg_flag = last ? 1 : 0;
                    }
                    mbar_arrive(bar(B_SEGSYNC));
                    if (!mbar_wait_warp(bar(B_SEGSYNC), sx & 1, abort_flag)) { ok = false; break; }
                    ++sx;
                    if (*seg_flag) {
                        __threadfence();
                        const MergeArgs ma = {p.part_o, p.part_ml, p.out, p.lse, p.Hq, G, N, rows_total};
                        merge_unit<ROWS, D>(ma, T, geff, ub, c0, c1, sg.b, sg.kvh, sg.mblock, st, kSmx);
                    }
                }

                tc_fence_before();        // the next segment's first product overwrites O
                ++seg;
            }
        }
    }

    if (CL) {
        // ---- cluster exchange: every CTA of the unit has parked its partial (O, m, l) in its own shared memory.
        // All threads of the cluster meet at the hardware cluster barrier (the warps that finished early wait
        // there without polling); then rank r merges rows [r*rp, (r+1)*rp) of all k partials through distributed
        // shared memory and writes them out. ----
        __syncwarp();
        if (!cl_waited) { cluster_wait(); cl_waited = true; }     // (fused rotary embedding: the start-up phase, warps 0-3)
        if (warp >= 4) {
            cluster_merge<ROWS, D>(p, cl_seg, ck, cr, base + SMEM_K, base + SMEM_K + (D / 4) * ROWS * 16, tid - 128, abort_flag);
        } else {
            cluster_sync_all();
            if (warp == 1) {
                // every thread of the CTA is past its last tensor-memory access: give the columns back now, beside the
                // merge, instead of on the way out
                tc_fence_after();
                asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(TMEM_COLS) : "memory");
            }
            cluster_arrive_release();
        }
    }

    // ---- tear-down.  Cluster form: nobody leaves while a peer may still read its shared memory or signal its barriers;
    // every thread has arrived above (all its other waits are bounded), so this hardware barrier ends.  Even split:
    // everyone meets, TMEM goes back. ----
    if (CL) {
        __syncwarp();
        cluster_wait();
    } else {
        tc_fence_before();
        __syncthreads();
    }
    if (!CL && warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(TMEM_COLS) : "memory");
    }
    if (tid == 0 && *abort_flag) atomicCAS(p.status, 0, (int)VISPEC_E_TIMEOUT);
}



}  // namespace


static size_t tc5_partial_bytes(int grid, int rows, int D) { return (size_t)2 * grid * rows * (D * 4 + 8); }

namespace {

// Streaming-read probe: the K/V rows one attention call reads, moved by the same TMA producer through the same
// rings on the even split of all steps over the CTAs, and nothing else (a second thread hands every stage
// straight back).  It measures what this way of streaming reaches on its own: the ceiling the attention kernel
// can approach.
__global__ void __launch_bounds__(64, 1)
stream_probe_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap v_map, const Tc5Params p) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t base = smem_u32(sm);
    if (base & 1023u) {
        if (threadIdx.x == 0) atomicCAS(p.status, 0, (int)VISPEC_E_UNSUPPORTED);
        return;
    }
    constexpr int NS = NSK + NSV;                              // stages: K and V of a step take consecutive ones
    const uint32_t bars = base + NS * STAGE_BYTES;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + NS * STAGE_BYTES + 2 * NS * 8);
    Sched& sched = *reinterpret_cast<Sched*>(sm + NS * STAGE_BYTES + 256);
    auto full = [&](int i) { return bars + 8u * (uint32_t)i; };
    auto empty = [&](int i) { return bars + 8u * (uint32_t)(NS + i); };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < NS; ++i) { mbar_init(full(i), 1); mbar_init(empty(i), 1); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) sched_build(sched, p, lane, lane < p.B ? p.kv_len[lane] : 0);
    pdl_launch_dependents();
    if (!p.early) pdl_wait();
    __syncthreads();
    const int T = sched.base[p.B];
    const int geff = T > 0 ? sched_ctas(T, sched.units, (int)gridDim.x, p.min_steps, sched_round_steps(p)) : 0;
    const int cta = blockIdx.x;
    if (cta < geff && lane == 0) {
        const int lo = cta_lo(cta, T, geff), hi = cta_lo(cta + 1, T, geff);
        SegIter<false> si; si.s = &sched; si.B = p.B; si.n_mblocks = p.n_mblocks; si.seg_cost_ = 0; si.g = lo; si.lo = lo; si.hi = hi; si.cta = cta;
        si.cl = false; si.cl_done = false;
        Seg sg;
        int n = 0;                                             // stages handled so far
        if (warp == 0) {
            const uint64_t pol = l2_evict_first_policy();
            bool waited = !p.early, ok = true;
            while (ok && si.next(sg)) {
                const int bh = sg.b * p.Hkv + sg.kvh;
                for (int t = 0; t < sg.n && ok; ++t) {
                    const int tok = (sg.st0 + t) * STEP;
                    if (!waited && tok + STEP > sg.S) { pdl_wait(); waited = true; }
                    for (int kv = 0; kv < 2; ++kv, ++n) {
                        const int s = n % NS;
                        if (!mbar_wait(empty(s), ((n / NS) & 1) ^ 1, abort_flag)) { ok = false; break; }
                        mbar_expect_tx(full(s), STAGE_BYTES);
                        tma_load_3d(base + s * STAGE_BYTES, kv ? &v_map : &k_map, full(s), 0, tok, bh, pol);
                        tma_load_3d(base + s * STAGE_BYTES + HALF_BYTES, kv ? &v_map : &k_map, full(s), 64, tok, bh, pol);
                    }
                }
            }
            if (*abort_flag) {
                volatile int never = 0;
                for (int u = max(0, n - NS); u < n; ++u) mbar_wait(full(u % NS), (u / NS) & 1, &never);
            }
        } else {
            bool ok = true;
            while (ok && si.next(sg))
                for (int t = 0; t < 2 * sg.n; ++t, ++n) {
                    if (!mbar_wait(full(n % NS), (n / NS) & 1, abort_flag)) { ok = false; break; }
                    mbar_arrive(empty(n % NS));
                }
        }
    }
    __syncthreads();
    // nothing to stream (every sequence out of range), or none of the last tiles in this CTA's range: the probe must still not
    // end before its predecessor, because what follows it on the stream waits for the probe only
    if (tid == 0) pdl_wait();
    if (tid == 0 && *abort_flag) atomicCAS(p.status, 0, (int)VISPEC_E_TIMEOUT);
}

}  // namespace

// Largest number of co-resident clusters of each size (index: PAIR, cluster size), found once per device.
static int g_max_clusters[2][9];

static int query_max_clusters(bool pair, int k) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(k * 64); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = SMEM_ALLOC;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = k; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int n = 0;
    cudaError_t e = pair ? cudaOccupancyMaxActiveClusters(&n, attn_tc5_kernel<true, true, false>, &cfg)
                         : cudaOccupancyMaxActiveClusters(&n, attn_tc5_kernel<false, true, false>, &cfg);
    if (e != cudaSuccess) { cudaGetLastError(); return 0; }
    return n;
}

// Estimates in microseconds per call, fitted to measurements over the long-response shapes (16 query and 2 kv heads, 2048 to
// 32768 tokens, 16 to 128 nodes, 1 to 8 sequences) and the 7B and 13B ones: a fixed part, then the steps of the busiest
// CTA, each at the rate its softmax warps reach (a little slower the more SMs are at work) or at its share of HBM (64 KB
// per step over 7 TB/s; the row blocks of a kv head read the same tiles, so one in n_mblocks comes from HBM; a
// step's bytes follow the head size, its softmax does not).  The host knows only the capacity S_max, not kv_len: the
// estimate is for full caches unless the caller has given the length it expects (VISPEC_OPT_KV_LEN_HINT).
// Both sides of the line between the forms, clusters / even split, us per layer: 16 query and 2 kv heads, 1 x 16 nodes on 2048 10.1 /
// 11.9, on 8192 16.3 / 14.2, on 32768 38.2 / 19.2, 4 x 60 on 8192 25.2 / 32.4; 32 heads, 1 x 60 on 3904 15.3 / 19.5, 2 x 60 on
// 4000 25.4 / 28.5; 40 heads, 1 x 30 on 8000 29.4 / 34.6, 2 x 30 on 4000 37.0 / 34.3.
// (alternate: units of 128 rows in clusters, whose softmax groups take alternate steps: 0.92 us per step where two threads per row take
// 1.18.  Where many row blocks share few heads in large clusters a step takes a quarter longer - 16 query and 2 kv heads, 128 nodes: one
// sequence of 32768 in clusters of eight 1.16, four of 8192 in clusters of two 0.90 -, beyond four ranks the merge grows, and in long
// calls the power cap weighs more on it than on the two-tile kernel, whose rows share their K/V tiles.  One-tile clusters / two-tile
// kernel, us per layer in runs of seconds: 8 x 60 nodes on 8192 44.6 / 45.6, 4 x 60 on 16384 44.6 / 47.8, on 32768 81.1 / 79.8, 8 x 128 on
// 8192 77.6 / 82.1, 2 x 128 on 40000 92.1 / 89.4; in short ones 39.5 / 43.4, 39.5 / 44.8, 72.3 / 70.9, 70.1 / 74.9; 1 x 128 on 32768
// 49.0 / 42.0; 28 / 4 heads, 2 x 92 on 40000 142 / 125; 16 / 4 heads of size 64, 6 x 60 on 3000 17.7 / 21.7, 6 x 128 30.1 / 27.0.)
static double tc5_compute_us(const AttnArgs& a, bool pair, double ctas, bool alternate) {
    const double busy = ctas / a.sm_count, us = pair ? 0.8 + 0.25 * busy : alternate ? 0.80 + 0.14 * busy : 1.05 + 0.15 * busy;
    return a.D == 64 ? 0.9 * us : us;
}
static double tc5_step_us(const AttnArgs& a, bool pair, int n_mblocks, double ctas, bool alternate) {
    return fmax(tc5_compute_us(a, pair, ctas, alternate), ctas * 0.0093 * (a.D / 128.0) / n_mblocks);
}
static int tc5_steps(const AttnArgs& a) {
    const int slots = (a.kv_len_hint > 0 && a.kv_len_hint + a.N < a.S_max) ? a.kv_len_hint + a.N : a.S_max;
    return (slots + STEP - 1) / STEP;
}
// (late: 128 rows per kv head in clusters of four and more, which leave 20 to 50 SMs without work.  From about the fourteenth step of a
// CTA on, when what its rings held at the start is used up and the clusters have drifted apart, a step takes longer by what the
// CTAs draw on HBM, and the even split, on all SMs, is the faster form.  16 query and 2 kv heads, clusters / even split, us per
// layer: 8 x 16 nodes on 12000 tokens 26.9 / 27.9, on 16384 35.2 / 34.4, on 20000 43.3 / 39.4, on 24000 51.6 / 46.5, on 32000 67.4 / 58.0; on
// half to all of 20000 30.4 / 31.5, of 28000 41.6 / 38.9; 6 x 13 on 20000 31.8 / 32.4, on 24000 38.2 / 36.7, on 28000 42.7 / 39.5; 5 x 16 on
// 24000 37.1 / 32.2.  Clusters of two have no such loss: 32 heads, 2 x 128 on 8000 53.5 / 62.7.)
static double tc5_cluster_us(const AttnArgs& a, bool pair, int n_mblocks, int k) {
    const double ctas = (double)a.B * a.Hkv * n_mblocks * k, steps = (double)((tc5_steps(a) + k - 1) / k);
    const double step = tc5_step_us(a, pair, n_mblocks, ctas, !pair);
    if (pair) return 6.9 + steps * step;
    const double over = 0.005 * ctas * (a.D / 128.0) - (step - tc5_compute_us(a, pair, ctas, !pair));
    const double late = n_mblocks == 1 && k >= 4 ? fmax(0.0, over) * fmax(0.0, steps - 14.0) : 0.0;
    return 9.4 + steps * step + late + 0.35 * (k > 4 ? k - 4 : 0) + (n_mblocks > 4 && k > 4 ? 0.24 * steps : 0.0) +
           0.22 * (ctas / a.sm_count) * fmax(0.0, steps - 32.0);
}
// (even split: the CTAs as sched_ctas counts them; partials of 128 rows cost 34 ns per CTA, written and merged, those of 64
// rows go in the fixed part; where there are more units than CTAs and several row blocks every further segment of a CTA costs a Q
// tile, a pipeline start and an epilogue.  A call with the fused rotary embedding, which exists in clusters only, would need the rotation
// kernel ahead of it: 16 / 2 heads, 5 x 16 on 16384 28.8 in clusters, 29.6 with kernel and even split, where the plain calls take
// 27.1 and 25.6)
static double tc5_even_us(const AttnArgs& a, bool pair, int n_mblocks) {
    const int units = a.B * a.Hkv * n_mblocks;
    const double T = (double)tc5_steps(a) * units;
    double n = fmin((double)a.sm_count, fmax(1.0, floor(T / 2.0)));
    if (units <= n) {
        const double r = floor(n / units) * units;
        if (n_mblocks > 1 || ceil(T / r) - ceil(T / n) <= 3.0) n = r;
    }
    return (pair ? 9.5 : 10.4 + 0.034 * n) + ceil(T / n) * tc5_step_us(a, pair, n_mblocks, n, false) + (units > n && n_mblocks > 1 ? 11.0 * units / n : 0.0) +
           (a.rope_table ? 3.0 : 0.0);
}

// Cluster size of the cluster form: one cluster per unit, as large as all clusters fit at once (0: they do not).
static int tc5_max_cluster(const AttnArgs& a, bool pair, int n_mblocks) {
    const int units = a.B * a.Hkv * n_mblocks;
    int best = 0;
    for (int k = 1; k <= 8; ++k)
        if (units * k <= a.sm_count && g_max_clusters[pair][k] >= units) best = k;
    return best;
}

// Row layout and form of a call.  At most 64 query rows per kv head: one unit of 64 rows, rows duplicated over the two lane
// halves.  More: blocks of 128 rows, lane = row - unless that leaves most of the GPU idle (few sequences and kv
// heads, rows just over 64: one cluster of at most 8 CTAs per unit is all the cluster form can use): then blocks of 64
// rows in the duplicated layout make twice the units, and a step of such a unit costs its softmax threads half the
// columns, at the price of every K/V tile crossing from L2 twice as often and half of each product computed for nothing.
// (As an even split the smaller blocks gain nothing.)  The best estimate decides, a form that options ask for first.
// Clusters with 64-row units / with 128: 16 query and 2 kv heads, 1 x 16 nodes on 2048 8.3 / 10.1, 4 x 16 on 8192 17.0 / 17.6, 1 x 128 on
// 2048 11.5 / 12.2; 28 / 4 heads, 1 x 60 on 3344 13.4 / 14.3, on 1000 9.9 / 12.9; 16 / 4 heads of size 64, 1 x 128 on 4096 12.8 / 12.4.
constexpr int kSegCost = 4;                     // see SegIter; in steps
struct Tc5Layout { bool pair; int rows, n_mblocks, ck; double est_us; };
static Tc5Layout tc5_layout(const AttnArgs& a) {
    const int rows_total = (a.Hq / a.Hkv) * a.N;
    const bool small = rows_total <= 64;
    const int nmb = small ? 1 : (rows_total + 127) / 128, k = tc5_max_cluster(a, small, nmb);
    const bool want_even = a.tc5_path == 1 || a.tc5_path == 3, want_clusters = a.tc5_path == 2;
    Tc5Layout best = {small, small ? 64 : 128, nmb, 0, tc5_even_us(a, small, nmb)};
    if (k > 0 && !want_even) {
        const double us = tc5_cluster_us(a, small, nmb, k);
        if (want_clusters || us <= best.est_us) { best.ck = k; best.est_us = us; }
    }
    if (!small && a.tc5_path == 0) {
        const int nmb64 = (rows_total + 63) / 64, k64 = tc5_max_cluster(a, true, nmb64);
        const double us = k64 > 0 ? tc5_cluster_us(a, true, nmb64, k64) : 1e30;
        if (us < best.est_us) best = {true, 64, nmb64, k64, us};
    }
    return best;
}

bool attn_tc5_supports(const AttnArgs& a) {
    if (!((a.D == 128 || a.D == 64) && a.k_map && a.v_map && a.B > 0 && a.B <= kMaxB)) return false;
    if (a.D == 64 && (a.rope_table || a.page_rows)) return false;
    const int rows_total = (a.Hq / a.Hkv) * a.N;
    const int rows = rows_total <= 64 ? 64 : 128;
    const long long n_mblocks = (rows_total + 63) / 64;          // the most either layout makes
    const long long t_max = (long long)a.B * a.Hkv * n_mblocks * ((a.S_max + STEP - 1) / STEP);
    if (t_max * a.sm_count >= (1ll << 31)) return false;
    if (!(a.scale > 0.f)) return false;       // the kernel takes the maximum before scaling
    return kCounterBytes + tc5_partial_bytes(a.sm_count, rows, a.D) <= a.ws_bytes;
}

cudaError_t init_attn_tc5() {
    cudaError_t e = cudaSuccess;
    const void* kernels[12] = {(const void*)attn_tc5_kernel<true, false, false>, (const void*)attn_tc5_kernel<false, false, false>,
                               (const void*)attn_tc5_kernel<true, true, false>, (const void*)attn_tc5_kernel<false, true, false>,
                               (const void*)attn_tc5_kernel<true, false, true>, (const void*)attn_tc5_kernel<false, false, true>,
                               (const void*)attn_tc5_kernel<true, true, true>, (const void*)attn_tc5_kernel<false, true, true>,
                               (const void*)attn_tc5_kernel<true, false, false, false, 64>, (const void*)attn_tc5_kernel<false, false, false, false, 64>,
                               (const void*)attn_tc5_kernel<true, true, false, false, 64>, (const void*)attn_tc5_kernel<false, true, false, false, 64>};
    for (const void* k : kernels) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_ALLOC);
        if (e != cudaSuccess) return e;
    }
    const void* rope_kernels[2] = {(const void*)attn_tc5_kernel<true, true, false, true>, (const void*)attn_tc5_kernel<false, true, false, true>};
    for (const void* k : rope_kernels) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_ALLOC);
        if (e != cudaSuccess) return e;
    }
    for (int k = 1; k <= 8; ++k) { g_max_clusters[0][k] = query_max_clusters(false, k); g_max_clusters[1][k] = query_max_clusters(true, k); }
    if (getenv("VISPEC_DEBUG")) for (int k = 1; k <= 8; ++k) fprintf(stderr, "vispec: cluster size %d: %d (rows > 64) / %d (rows <= 64) co-resident clusters\n", k, g_max_clusters[0][k], g_max_clusters[1][k]);
    for (cudaError_t m : {init_merge<64, 128>(), init_merge<128, 128>(), init_merge<64, 64>(), init_merge<128, 64>()})
        if (m != cudaSuccess) return m;
    return cudaSuccess;
}

// Would units of 256 rows in two tiles (attn_tc5_wide.cu) serve the call better?  Measured, one-tile / two-tile kernel, us
// per layer (16 query and 2 kv heads unless said otherwise): 8 x 128 nodes on 4096 tokens 41.2 / 43.6; 28 / 4 heads: 8 x 60 on 4096
// 41.8 / 44.0, 8 x 128 on 1000 (more units than one-tile clusters fit) 42.1 / 34.7, 4 x 128 on 8192 70.9 / 73.5; long calls: the comment at
// tc5_step_us.  The two-tile kernel reads a K/V tile for twice the rows; its first step and its epilogue are longer.
static bool tc5_prefers_wide(const AttnArgs& a, const Tc5Layout& lay, const WidePlan& wide, double extra_us = 0.0) {
    return wide.est_us < 1e29 && wide.est_us + extra_us < 0.98 * lay.est_us;
}

// (the fused rotary embedding exists in the cluster form of the one-tile kernel; a call that goes elsewhere pays 3 us for
// the rotation kernel, 2 of which the fused form would have cost too)
bool attn_tc5_uses_clusters(const AttnArgs& a) {
    const Tc5Layout lay = tc5_layout(a);
    AttnArgs plain = a;
    plain.rope_table = nullptr;
    return lay.ck > 0 && !tc5_prefers_wide(a, lay, attn_tc5_wide_plan(plain), 1.0);
}

cudaError_t launch_attn_tc5(const AttnArgs& a, cudaStream_t st, int* n_launches) {
    *n_launches = 0;
    const Tc5Layout lay = tc5_layout(a);
    const WidePlan wide = attn_tc5_wide_plan(a);
    if (tc5_prefers_wide(a, lay, wide)) return launch_attn_tc5_wide(a, wide, st, n_launches);
    const bool pair = lay.pair;
    const int rows = lay.rows, n_mblocks = lay.n_mblocks, ck = lay.ck;
    const int units = a.B * a.Hkv * n_mblocks;
    const long long t_max = (long long)units * ((a.S_max + STEP - 1) / STEP);
    // (more units than CTAs, so ranges do not begin and end with units: only there does the number of segments differ)
    // (and T * grid must stay below 2^31, as attn_tc5_supports has checked it for the steps alone)
    const int seg_cost = pair && ck == 0 && units > a.sm_count && (t_max + (long long)units * kSegCost) * a.sm_count < (1ll << 31) ? kSegCost : 0;
    const int grid = ck > 0 ? units * ck : (int)(t_max < a.sm_count ? t_max : a.sm_count);

    Tc5Params p = {};
    p.q = (const __nv_bfloat16*)a.q; p.kv_len = a.kv_len; p.mask = a.mask;
    p.out = (__nv_bfloat16*)a.out; p.lse = a.lse;
    unsigned char* ws = (unsigned char*)a.ws + kCounterBytes;
    p.part_o = (float4*)ws;
    p.part_ml = (float2*)(ws + (size_t)2 * grid * rows * a.D * 4);
    p.B = a.B; p.N = a.N; p.Hq = a.Hq; p.Hkv = a.Hkv; p.S_max = a.S_max; p.n_mblocks = n_mblocks;
    p.grid_attn = grid; p.min_steps = 2; p.early = a.early_prefetch ? 1 : 0; p.step = STEP; p.seg_cost = seg_cost;
    p.scale_log2 = a.scale * 1.4426950408889634f;
    p.status = a.status;
    cudaError_t err;
    const bool paged = a.page_rows != 0;
    // Even split, at most 64 rows per unit: short calls and those of more units than CTAs merge in the attention kernel (the last
    // arrival at a unit, by the counters at the head of the workspace; the ranges then end at different units, and most merges lie
    // within the call), the others with the merge kernel.  Measured, in the kernel / with the merge kernel, us per layer (13B
    // heads): 4 x 60 nodes on 1000 tokens 28.2 / 29.1, 8 x 16 on 3000 91.1 / 91.7; 2 x 30 on 4000 37.6 / 34.3.
    // Just above one unit per CTA little lies within the call, and what is merged late counts against the rows merged: 160 units on 1500-3000
    // tokens with the rotation kernel between the calls (a quarter of a pass of four layers), 16 nodes 44.2 / 42.2, 31 nodes 46.2 / 44.8, 40 nodes 48.6 / 48.7, 60 nodes 49.6 / 50.1
    // (on 3000-5000: 16 nodes 67.1 / 66.4, 60 nodes 72.4 / 74.7); 200 units 56.4 / 56.7 and 63.4 / 64.6, 280 units 69.4 / 70.9 and 78.2 / 80.3.
    // Pools of 16-row blocks, whose producers are the slower part, gain from twice as many units as SMs on, 16 and 60 nodes: 160 units
    // 47.4 / 43.2 and 52.5 / 51.2, 200 units 60.3 / 57.2 and 67.5 / 65.3, 240 units 65.1 / 61.4 and 79.7 / 78.6, 280 units 74.9 / 72.1 and 82.5 / 82.7, 320 units
    // 79.2 / 78.2 and 97.1 / 97.5 (without the rotation kernel 74.6 / 75.4 and 86.9 / 87.1).  Blocks of 32 to 128 rows are within 1 % of the
    // contiguous cache's line with 60 nodes (200 units 65.2-65.4 / 65.3-65.7) and up to 3 % on the other side of it with 16 (58.0-58.4 / 57.2-58.0).
    // Blocks of 128 rows, a grid with more units than counters and split form 3 always get the merge kernel.
    const int crowd = a.page_rows == 16 ? 8 : (a.Hq / a.Hkv) * a.N <= 32 ? 5 : 4;      // quarters of a unit per SM
    const bool own_merge = pair && ck == 0 && a.tc5_path != 3 && !a.no_counters && (size_t)units * sizeof(int) <= kCounterBytes &&
                           (a.tc5_path == 1 || tc5_steps(a) < 12 || 4ll * units > (long long)crowd * a.sm_count);
    const PagedArgs pa = {a.block_table, a.table_stride, a.page_rows, a.num_blocks, a.Hkv, a.N, a.token_major, a.status,
                          own_merge ? (int*)a.ws : nullptr};
    auto launch_attn = [&](auto kernel, int cluster) {
        return launch_pdl(kernel, dim3(grid), dim3(kThreads), SMEM_ALLOC, st, cluster, *a.k_map, *a.v_map, p, pa);
    };
    if (a.rope_table) {
        // fused rotary embedding (contiguous caches): the table holds B*N*D/2 fp64 (cos, sin) pairs, then the same in fp32
        const size_t n = (size_t)a.B * a.N * (D / 2);
        const RopeArgs ra = {(const double2*)a.rope_table, (const float2*)((const double2*)a.rope_table + n),
                             (const __nv_bfloat16*)a.k_new, (const __nv_bfloat16*)a.v_new, (__nv_bfloat16*)a.k, (__nv_bfloat16*)a.v};
        auto launch_rope = [&](auto kernel, int cluster) {
            return launch_pdl(kernel, dim3(grid), dim3(kThreads), SMEM_ALLOC, st, cluster, *a.k_map, *a.v_map, p, ra);
        };
        if (ck <= 0) return cudaErrorInvalidValue;        // cluster form only: the caller asks attn_tc5_uses_clusters first
        err = pair ? launch_rope(attn_tc5_kernel<true, true, false, true>, ck) : launch_rope(attn_tc5_kernel<false, true, false, true>, ck);
        if (err != cudaSuccess) return err;
        ++*n_launches;
        return cudaSuccess;
    }
    // one launch in the cluster form (the CTAs of a unit merge their partials through distributed shared memory)
    auto launch_form = [&](auto cl) {
        constexpr bool CL = decltype(cl)::value;
        if (a.D == 64) return pair ? launch_attn(attn_tc5_kernel<true, CL, false, false, 64>, ck) : launch_attn(attn_tc5_kernel<false, CL, false, false, 64>, ck);
        if (paged) return pair ? launch_attn(attn_tc5_kernel<true, CL, true>, ck) : launch_attn(attn_tc5_kernel<false, CL, true>, ck);
        return pair ? launch_attn(attn_tc5_kernel<true, CL, false>, ck) : launch_attn(attn_tc5_kernel<false, CL, false>, ck);
    };
    err = ck > 0 ? launch_form(std::true_type{}) : launch_form(std::false_type{});
    if (err != cudaSuccess) return err;
    ++*n_launches;
    if (ck > 0 || own_merge) return cudaSuccess;
    err = a.D == 64 ? (pair ? launch_merge<64, 64>(p, units, grid, st) : launch_merge<128, 64>(p, units, grid, st))
                    : (pair ? launch_merge<64, 128>(p, units, grid, st) : launch_merge<128, 128>(p, units, grid, st));
    if (err != cudaSuccess) return err;
    ++*n_launches;
    return cudaSuccess;
}

namespace {

// The attention kernels' wait routine on a barrier that never completes: thread 0 runs out of its limit and raises the
// give-up flag; thread 32 waits on a second such barrier with the ordinary (long) limit and must be released by that
// flag.  Then the block reports VISPEC_E_TIMEOUT and leaves one arrival counter non-zero, as a call that gave up
// between a partial's arrival and the unit's merge would.
__global__ void __launch_bounds__(64)
bounded_wait_selftest_kernel(long long limit, int* status, int* counters) {
    __shared__ __align__(8) unsigned long long bars[2];
    __shared__ int flag;
    volatile int* abort_flag = &flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bars[0]), 1);
        mbar_init(smem_u32(&bars[1]), 1);
        flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    bool gave_up = false;
    if (threadIdx.x == 0) gave_up = !mbar_wait(smem_u32(&bars[0]), 0, abort_flag, limit);
    if (threadIdx.x == 32) gave_up = !mbar_wait(smem_u32(&bars[1]), 0, abort_flag);
    const int n = __syncthreads_count(gave_up);
    if (threadIdx.x == 0 && n == 2 && *abort_flag) {
        atomicCAS(status, 0, (int)VISPEC_E_TIMEOUT);
        atomicAdd(counters, 1);
    }
}

}  // namespace

cudaError_t launch_bounded_wait_selftest(long long limit, int* status, int* counters, cudaStream_t st) {
    bounded_wait_selftest_kernel<<<1, 64, 0, st>>>(limit, status, counters);
    return cudaGetLastError();
}

cudaError_t init_stream_probe() {
    return cudaFuncSetAttribute(stream_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (NSK + NSV) * STAGE_BYTES + 256 + (int)sizeof(Sched));
}

cudaError_t launch_stream_probe(const AttnArgs& a, cudaStream_t st) {
    const int rows_total = (a.Hq / a.Hkv) * a.N;
    const int n_mblocks = rows_total <= 64 ? 1 : (rows_total + 127) / 128;
    Tc5Params p = {};
    p.kv_len = a.kv_len;
    p.B = a.B; p.N = a.N; p.Hq = a.Hq; p.Hkv = a.Hkv; p.S_max = a.S_max;
    p.n_mblocks = 1;                                       // every K/V row once, whatever the number of row blocks
    (void)n_mblocks;
    const long long t_max = (long long)a.B * a.Hkv * ((a.S_max + STEP - 1) / STEP);
    const int grid = (int)(t_max < a.sm_count ? t_max : a.sm_count);
    p.grid_attn = grid; p.min_steps = 2; p.early = a.early_prefetch ? 1 : 0; p.step = STEP;
    p.status = a.status;
    return launch_pdl(stream_probe_kernel, dim3(grid), dim3(64), (size_t)((NSK + NSV) * STAGE_BYTES + 256 + sizeof(Sched)), st, 0,
                      *a.k_map, *a.v_map, p);
}

}  // namespace vispec
