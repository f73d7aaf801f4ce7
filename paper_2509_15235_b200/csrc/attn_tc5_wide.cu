// The TMA + tcgen05 attention kernel for calls with many query rows per kv head (grouped heads times a large tree): a
// unit is (sequence, kv head, block of 256 query rows), two accumulator tiles of 128 rows that share every K/V stage.
//
// What bounds it: the tensor pipe (2048 cycles per 128-token step: two score products and two PV products of
// 128 x 128 x 128) and beside it the exponentials (2 x 1024 cycles on the special-function pipe; at head size 64, where the
// products are half as long, an eighth of them is moved to the FMA pipe); over a long call the power cap.  The one-tile kernel spends 2670 cycles on half of that: its eight softmax
// warps move in lock-step (two threads per row exchange the row's maximum), so the special-function pipe idles while they
// wait, load and take maxima.  Here each tile has four softmax warps of its own, one thread per row (nothing to exchange),
// and the tiles run out of phase: while one is in its exponentials, the tensor pipe works for the other: 3150 cycles per
// step of both.  Each stage serves twice the rows, so L2 delivers half the bytes per product.
// qwen3b_S32768_N128_B8: 345-363 -> 273-281 us per layer (1.0 PFLOP/s, at 1530 MHz under the power cap; 252 in a burst).
// Tried: eight softmax warps per tile, two threads per row (282-286 against 273-277); 1/2, 1/3, 1/4, 1/8 of the exponentials
// on the FMA pipe (292, 283, 277, 276 with a cubic that was dropped for its error; none is as fast as 1/8, see kPolyEvery).
//
//   warp 0     TMA producer of the K ring (2 x 32 KB; head size 64: 4 x 16 KB)
//   warp 1     issuer (one elected lane) of all products, in the order S_A S_B | PV_A S_A' PV_B S_B' | ...: S of a step overwrites
//              P of the step before, which frees half of the tensor memory, and the completion of S, committed behind everything
//              issued before it, tells that O and P are free.  (That S does not overtake the PV product which reads that P rests on
//              one CTA's products starting in the order of issue: how the tensor core works, not a documented guarantee.)  A PV
//              product starts when the first half of its P is there.
//              (An issuer per tile was slower: the tiles' products interleave, both end together, and the tiles fall into
//              step, their softmaxes competing while the tensor pipe idles.)
//   warp 2     producer of the V ring (3 x 32 KB; head size 64: 6 x 16 KB)
//   warp 3     derives the schedule from kv_len
//   warps 4-7 / 8-11   softmax of tile A / B: thread <-> TMEM lane <-> query row
// TMEM (512 columns): S_A 0..127, S_B 128..255 (P of the tile, bf16, in the first 64 columns of its S), O_A 256, O_B 384.
//
// Work split: a cluster of k <= 8 CTAs per unit where all units fit at once, or an even split in lock-step: the CTAs form
// groups of n_mblocks, the (sequence, kv head, step) line is cut evenly over the groups, and a CTA takes one row block of its
// group's range, so that the row blocks of a kv head read the same K/V tiles at the same time and HBM delivers them
// once.  (Cut unit by unit, the row blocks of a head stream the cache at different times: qwen3b_S32768_N128_B8 read it eight
// times, 2.1 GB per layer, and ran at the rate of HBM.)
// The waits, time-outs, programmatic launch and merge are those of the one-tile kernel (attn_tc5.cu).
#include <cuda_bf16.h>
#include <cmath>

#include "tc5_common.cuh"

namespace vispec {

using namespace tc5;

namespace {

constexpr int kThreads = 384;
constexpr int kRows = 256;                     // query rows per unit
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t COL_S = 0, COL_O = 256;     // + 128 per tile

enum { W_KFULL = 0, W_KEMPTY = W_KFULL + 4, W_VFULL = W_KEMPTY + 4, W_VEMPTY = W_VFULL + 6, W_SFULL = W_VEMPTY + 6,
       W_PFULL = W_SFULL + 2 /* [tile][half of the columns] */, W_QFULL = W_PFULL + 4, W_OFULL = W_QFULL + 2, W_OFREE = W_OFULL + 2, W_COUNT = W_OFREE + 2 };

template <int HD>
struct WideRing {
    static constexpr int NH = HD / 64, STAGE = NH * HALF_BYTES, NSK = 4 / NH, NSV = 6 / NH;
    static constexpr int OFF_K = 0, OFF_V = NSK * STAGE, OFF_Q = OFF_V + NSV * STAGE;     // Q: one stage-like tile per row tile
    static constexpr int KFULL = W_KFULL, KEMPTY = W_KEMPTY, VFULL = W_VFULL, VEMPTY = W_VEMPTY;
};
constexpr int SMEM_BAR = 7 * 2 * HALF_BYTES;   // five stages and two Q tiles at head size 128
constexpr int BAR_BYTES = 288;
static_assert(W_COUNT * 8 + 20 <= BAR_BYTES, "barrier block too small");
constexpr int SMEM_SCHED = SMEM_BAR + BAR_BYTES;
constexpr int SMEM_TABRING = SMEM_SCHED + ((int)sizeof(Sched) + 15) / 16 * 16;
constexpr int SMEM_ALLOC = SMEM_TABRING + 256;
static_assert(SMEM_ALLOC <= 232448, "over the 227 KB a CTA may have");

// Head size 64: one pair of exponentials in this many goes to the FMA pipe (6 x 16 heads (4 kv) x 128 nodes on 3000, 16 layers:
// 469.1 us per pass, none 475.5).  At head size 128 none does: the steps are the tensor pipe's, and the power cap's (the
// benchmark's 8 x 128 nodes on 32768: none 4453, one in eight 4506; 28/4 heads, 8 x 60 on 8192 355.5 / 358.9).
constexpr int kPolyEvery = 8;

template <bool CL, bool PAGED, int HD>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc5_wide_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap v_map, const Tc5Params p,
                     const PagedArgs pa) {
    static_assert(HD == 128 || !PAGED, "paged pools have head size 128");
    using R = WideRing<HD>;
    constexpr int NH = R::NH, NSK = R::NSK, NSV = R::NSV, STAGE = R::STAGE;
    extern __shared__ __align__(1024) unsigned char sm[];
    int kv_first = 0;
    if (p.early && threadIdx.x >= 96 && threadIdx.x < 128 && (int)threadIdx.x - 96 < p.B) kv_first = p.kv_len[threadIdx.x - 96];
    const uint32_t base = smem_u32(sm);
    if (base & 1023u) {                        // the swizzled tiles need it; every CTA sees the same base, so all of them leave
        if (threadIdx.x == 0) atomicCAS(p.status, 0, (int)VISPEC_E_UNSUPPORTED);
        return;
    }
    const uint32_t bars = base + SMEM_BAR;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + SMEM_BAR + W_COUNT * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + SMEM_BAR + W_COUNT * 8 + 8);
    Sched& sched = *reinterpret_cast<Sched*>(sm + SMEM_SCHED);
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int cta = blockIdx.x;
    const int G = p.Hq / p.Hkv, N = p.N, W = (N + 63) >> 6;
    const int rows_total = G * N;

    const int ck = CL ? (int)cluster_size() : 1, cr = CL ? (int)cluster_ctarank() : 0;
    // this CTA's row block, the same in all its segments; does its second tile have rows?
    const int my_block = (CL ? cta / ck : cta) % p.n_mblocks;
    const bool two = my_block * kRows + 128 < rows_total;

    if (tid == 0) {
        for (int i = 0; i < NSK; ++i) { mbar_init(bar(W_KFULL + i), 1); mbar_init(bar(W_KEMPTY + i), 1); }
        for (int i = 0; i < NSV; ++i) { mbar_init(bar(W_VFULL + i), 1); mbar_init(bar(W_VEMPTY + i), 1); }
        for (int i = 0; i < 4; ++i) mbar_init(bar(W_PFULL + i), 128);
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(W_SFULL + i), 1); mbar_init(bar(W_QFULL + i), 128);
            mbar_init(bar(W_OFULL + i), 1); mbar_init(bar(W_OFREE + i), 128);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (!p.early) {
        pdl_wait();
        if (warp == 3 && lane < p.B) kv_first = p.kv_len[lane];
    }
    pdl_launch_dependents();
    if (warp == 3) sched_build(sched, p, lane, kv_first);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    // Schedule: cluster <-> unit, or groups of n_mblocks CTAs on equal ranges of the (sequence, kv head, step) line.
    const int T = sched.base[p.B];
    const int group = CL ? 0 : cta / p.n_mblocks;
    const int geff = (CL || T <= 0) ? 0 : sched_ctas(T, sched.units, (int)gridDim.x / p.n_mblocks, p.min_steps, sched_round_steps(p));
    const bool active = CL || group < geff;
    const int lo = (!CL && active) ? cta_lo(group, T, geff) : 0, hi = (!CL && active) ? cta_lo(group + 1, T, geff) : 0;
    const uint32_t tmem = *tmem_slot;
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
    struct Iter {
        SegIter<false> it; int n_mblocks, mblock;
        __device__ __forceinline__ bool next(Seg& o) {
            if (!it.next(o)) return false;
            if (!it.cl) { o.mblock = mblock; if (o.slot >= 0) o.slot = o.slot * n_mblocks + mblock; }
            return true;
        }
    };
    auto make_iter = [&]() {
        Iter x; x.it.s = &sched; x.it.B = p.B; x.it.n_mblocks = 1; x.it.seg_cost_ = 0; x.it.g = lo; x.it.lo = lo; x.it.hi = hi; x.it.cta = group;
        x.it.cl = CL; x.it.cl_done = false; x.it.cl_seg = cl_seg; x.n_mblocks = p.n_mblocks; x.mblock = my_block;
        return x;
    };

    if (warp < 4) {
    if (warp == 0 || warp == 2) {
        // ================= TMA producers: warp 0 the K ring, warp 2 the V ring =================
        const bool is_v = warp == 2;
        if ((PAGED || lane == 0) && active) {
            const uint64_t pol = l2_evict_first_policy();
            bool waited = !p.early, ok = true;
            int it = 0;
            Iter si = make_iter();
            Seg sg;
            const int ns = is_v ? NSV : NSK, full = is_v ? W_VFULL : W_KFULL, empty = is_v ? W_VEMPTY : W_KEMPTY;
            const uint32_t ring = base + (is_v ? R::OFF_V : R::OFF_K);
            const CUtensorMap* map = is_v ? &v_map : &k_map;
            while (ok && si.next(sg)) {
                if constexpr (PAGED) {
                    const uint32_t r = produce_paged<R>(pa, &k_map, &v_map, sg.b, sg.kvh, sg.st0, sg.n, sg.S, base, bars,
                                                        base + SMEM_TABRING + (is_v ? 128 : 0), abort_flag, pol, it, waited, lane, is_v ? 2 : 1);
                    it += (int)(r & 0x0fffffffu) + (is_v ? 0 : (int)((r >> 28) & 1u));
                    ok = !((r >> 29) & 1u);
                    waited = (r >> 30) & 1u;
                } else {
                    const int bh = sg.b * p.Hkv + sg.kvh;
                    for (int t = 0; t < sg.n; ++t, ++it) {
                        const int tok = (sg.st0 + t) * STEP, s = it % ns;
                        if (!waited && tok + STEP > sg.S) { pdl_wait(); waited = true; }   // the tree's rows come from the preceding kernel
                        if (!mbar_wait(bar(empty + s), ((it / ns) & 1) ^ 1, abort_flag)) { ok = false; break; }
                        mbar_expect_tx(bar(full + s), STAGE);
                        tma_load_3d(ring + s * STAGE, map, bar(full + s), 0, tok, bh, pol);
                        if constexpr (NH == 2) tma_load_3d(ring + s * STAGE + HALF_BYTES, map, bar(full + s), 64, tok, bh, pol);
                    }
                }
            }
            if (*abort_flag && lane == 0) {
                // drain: wait (bounded, fresh timer) until every copy this warp issued has landed
                volatile int never = 0;
                for (int u = max(0, it - ns); u < it; ++u) mbar_wait(bar(full + u % ns), (u / ns) & 1, &never);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= issuer of all products =================
        // The whole warp walks through the steps and waits, one elected lane issues: with uniform control flow the
        // descriptors live in uniform registers, where the instructions take them from.
        if (active) {
            constexpr uint32_t IDESC_S = instr_desc(0), IDESC_O = instr_desc(1, HD);
            constexpr uint32_t DESC_HI = desc_hi(1024);
            const int nt = two ? 2 : 1;
            const bool leader = elect_one();
            bool ok = true;
            uint32_t seg = 0;
            uint32_t sk = 0, pk = 0, sv = 0, pv = 0, pp = 0;   // ring positions with their phases, phase of P
            Iter si = make_iter();
            Seg sg;
            const uint32_t k0 = desc_lo(base + R::OFF_K, 16), v0 = desc_lo(base + R::OFF_V, HALF_BYTES), q0 = desc_lo(base + R::OFF_Q, 16);
            auto score = [&](int x) {                      // S_x = Q_x K^T
                if (x == 0) {
                    if (!mbar_wait_warp(bar(W_KFULL) + 8u * sk, pk, abort_flag)) return false;
                    tc_fence_after();
                }
                const uint32_t kb = k0 + sk * (STAGE >> 4), qb = q0 + x * (STAGE >> 4);
                if (leader) {
#pragma unroll
                    for (int ks = 0; ks < HD / 16; ++ks) {
                        const uint32_t off = ((ks >> 2) * HALF_BYTES + (ks & 3) * 32) >> 4;
                        tc_mma_ss(tmem + COL_S + x * 128, qb + off, DESC_HI, kb + off, DESC_HI, IDESC_S, ks > 0 ? 1u : 0u);
                    }
                    tc_commit(bar(W_SFULL + x));
                    if (x == nt - 1) tc_commit(bar(W_KEMPTY) + 8u * sk);
                }
                if (x == nt - 1 && ++sk == NSK) { sk = 0; pk ^= 1; }
                return true;
            };
            while (ok && si.next(sg)) {
                const int n = __shfl_sync(0xffffffffu, sg.n, 0);
                for (int x = 0; x < nt && ok && n > 0; ++x) ok = mbar_wait_warp(bar(W_QFULL + x), seg & 1, abort_flag) && score(x);
                for (int t = 0; t < n && ok; ++t) {
                    const uint32_t vb = v0 + sv * (STAGE >> 4);
                    ok = mbar_wait_warp(bar(W_VFULL) + 8u * sv, pv, abort_flag);
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        if (x >= nt || !ok) break;
                        // (a segment's first PV product starts a fresh O: the last segment's must have been read)
                        if (t == 0 && seg > 0 && !(ok = mbar_wait_warp(bar(W_OFREE + x), (seg - 1) & 1, abort_flag))) break;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {          // O_x += P_x V(step), half of the tokens as soon as their P is there
                            if (!ok || !(ok = mbar_wait_warp(bar(W_PFULL + 2 * x + h), pp, abort_flag))) break;
                            tc_fence_after();
                            if (leader) {
#pragma unroll
                                for (int ks = h * (STEP / 32); ks < (h + 1) * (STEP / 32); ++ks)
                                    tc_mma_ts(tmem + COL_O + x * 128, tmem + COL_S + x * 128 + ks * 8, vb + ks * 128, DESC_HI, IDESC_O, (t > 0 || ks > 0) ? 1u : 0u);
                            }
                        }
                        if (!ok) break;
                        if (x == nt - 1 && leader) tc_commit(bar(W_VEMPTY) + 8u * sv);
                        if (t + 1 < n) ok = score(x);          // overwrites P of this step, which the product before it reads (see above)
                        else if (leader) tc_commit(bar(W_OFULL + x));
                    }
                    if (++sv == NSV) { sv = 0; pv ^= 1; }
                    pp ^= 1;
                }
                ++seg;
            }
        }
        __syncwarp();
    }
    if (CL) {
        cluster_sync_all();
        cluster_arrive_release();
    }
    } else {
        // ================= softmax: one thread per query row, tile x by warps 4 + 4x .. 7 + 4x =================
        const int x = (warp - 4) >> 2, sp = warp & 3;
        const int tl = sp * 32 + lane;                        // TMEM lane = row of the tile
        const uint32_t lane_addr = tmem + ((uint32_t)(32 * sp) << 16);
        const uint32_t s_addr = lane_addr + COL_S + x * 128, o_addr = lane_addr + COL_O + x * 128;
        pdl_wait();                                           // q, tree_mask and every output come after the preceding kernel
        zero_rejected<HD>(p, sched, cta, tid - 128);
        if (active && (x == 0 || two)) {
            Iter si = make_iter();
            Seg sg;
            int it = 0, seg = 0;
            bool ok = true;
            while (ok && si.next(sg)) {
                // Q tile -> shared memory, rows in the swizzled K-major layout of a K stage (every score product of the last
                // segment has been consumed).  Thread t moves chunk t % QC of rows t / QC, t / QC + QR, ...
                {
                    constexpr int QC = HD / 8, QR = 128 / QC, ITEMS = 128 / QR, BATCH = 8;
                    const int qc = tl % QC;
#pragma unroll
                    for (int k0 = 0; k0 < ITEMS; k0 += BATCH) {
                        uint4 v[BATCH];
#pragma unroll
                        for (int k = 0; k < BATCH; ++k) {
                            const int row = sg.mblock * kRows + x * 128 + tl / QC + QR * (k0 + k);
                            v[k] = make_uint4(0, 0, 0, 0);
                            if (row < rows_total) {
                                const int nd = row / G, hd = sg.kvh * G + row % G;
                                v[k] = *(reinterpret_cast<const uint4*>(p.q + (((size_t)sg.b * N + nd) * p.Hq + hd) * HD) + qc);
                            }
                        }
#pragma unroll
                        for (int k = 0; k < BATCH; ++k) {
                            const int r = tl / QC + QR * (k0 + k);
                            *reinterpret_cast<uint4*>(sm + R::OFF_Q + x * STAGE + (qc >> 3) * HALF_BYTES + r * 128 + (((qc & 7) ^ (r & 7)) << 4)) = v[k];
                        }
                    }
                    fence_async_smem();
                    mbar_arrive(bar(W_QFULL + x));
                }
                const int lrow = x * 128 + tl;
                const int row = sg.mblock * kRows + lrow;     // query row within the kv head's G*N rows
                const bool row_ok = row < rows_total;
                const int node = row_ok ? row / G : 0, head = sg.kvh * G + (row_ok ? row % G : 0);
                const int S = sg.S, total = S + N;
                uint64_t mk0 = 0, mk1 = 0;
                if (row_ok) {
                    const uint64_t* mrow = p.mask + ((size_t)sg.b * N + node) * W;
                    mk0 = mrow[0];
                    if (W > 1) mk1 = mrow[1];
                    if (N < 64) mk0 &= (1ull << N) - 1;       // bits at or beyond N are not tree nodes
                    if (N < 128) mk1 &= N > 64 ? (1ull << (N - 64)) - 1 : 0ull;
                }
                float m_ref = -INFINITY, l_run = 0.f;
                bool has_o = false;

                for (int t = 0; t < sg.n; ++t, ++it) {
                    const int tok0 = (sg.st0 + t) * STEP;
                    // (this product was issued after the PV product of the step before, so that one is complete too: O and
                    // the columns of P are free)
                    if (!mbar_wait_warp(bar(W_SFULL + x), it & 1, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    // The row is read from tensor memory in halves of 64 columns, the upper half twice: held whole it took 200
                    // registers and code for 128 unrolled columns, which pushed the issuer's out of the instruction cache (every
                    // barrier wait of that thread then took 150-400 cycles).
                    const bool tail = tok0 + STEP > S;                  // reaches past the committed prefix: mask bits
                    uint64_t a0 = 0, a1 = 0;                            // bit c of (a0, a1): column c may be attended to
                    if (tail) {
                        const int t0 = tok0 - S;
                        if (t0 >= 0) shr128(mk0, mk1, t0, a0, a1); else shl128_fill(mk0, mk1, -t0, a0, a1);
                    }
                    uint32_t s[64];
                    auto load_half = [&](int h) {
                        tmem_ld32(s_addr + h * 64, s);
                        tmem_ld32(s_addr + h * 64 + 32, s + 32);
                        tmem_wait_ld();
                        if (tail) {
                            const uint64_t a = h ? a1 : a0;
#pragma unroll
                            for (int c = 0; c < 64; ++c)
                                if (!((a >> c) & 1ull)) s[c] = 0xff800000u;
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
                    const float tmax = max_nan(max3_nan(max3_nan(mx[0], mx[1], mx[2]), max3_nan(mx[3], mx[4], mx[5]), mx[6]), mx[7]) * p.scale_log2;
                    // move the reference maximum only when the tile exceeds it by more than the gap
                    float alpha = 1.f;
                    bool rescale = false;
                    if (tmax > m_ref + kRescaleGap) {         // also true on the first finite tile (m_ref = -inf)
                        alpha = exp2f(m_ref - tmax);
                        m_ref = tmax;
                        l_run *= alpha;
                        rescale = has_o;
                    }
                    if (!(tmax < INFINITY)) l_run = tmax - tmax;          // a NaN or an infinite score: the row is NaN (see inv_sum)
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
                    const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
                    const uint64_t sc2 = pk2(p.scale_log2, p.scale_log2), mm2 = pk2(-m_use, -m_use);
                    uint64_t sum2 = pk2(0.f, 0.f), sum2b = sum2;
                    bool fail = false;
                    if (tok0 + STEP > total) {
                        // last step of the sequence: V rows past the last key may hold anything, and they meet zero weights: made
                        // zeros before either tile's product (both tiles' warps write them, whichever product comes first)
                        const int sv = it % NSV;
                        fail = !mbar_wait(bar(W_VFULL + sv), (it / NSV) & 1, abort_flag);
                        if (!fail && tok0 + tl >= total) {
                            unsigned char* vrow = sm + R::OFF_V + sv * STAGE + tl * 128;
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                *reinterpret_cast<uint4*>(vrow + c * 16) = make_uint4(0, 0, 0, 0);
                                if (NH == 2) *reinterpret_cast<uint4*>(vrow + HALF_BYTES + c * 16) = make_uint4(0, 0, 0, 0);
                            }
                        }
                        fence_async_smem();
                    }
                    if (__any_sync(0xffffffffu, fail)) { ok = false; break; }
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1) load_half(1);             // (P of the first half lies in columns 0..31)
                        uint32_t pd[32];
#pragma unroll
                        for (int c = 0; c < 32; ++c) {
                            float x0, x1, e0, e1;
                            up2(fma2(pk2(__uint_as_float(s[2 * c]), __uint_as_float(s[2 * c + 1])), sc2, mm2), x0, x1);
                            if (HD == 64 && c % kPolyEvery == kPolyEvery - 1) exp2_fma_pair(x0, x1, e0, e1);
                            else { e0 = exp2f(x0); e1 = exp2f(x1); }
                            if (c & 1) sum2b = add2(sum2b, pk2(e0, e1)); else sum2 = add2(sum2, pk2(e0, e1));
                            pd[c] = pack_bf16(e0, e1);
                        }
                        tmem_st32(s_addr + h * 32, pd);
                        tmem_wait_st();
                        tc_fence_before();
                        mbar_arrive(bar(W_PFULL + 2 * x + h));
                    }
                    float l0, l1;
                    up2(add2(sum2, sum2b), l0, l1);
                    l_run += l0 + l1;
                    has_o = true;
                }
                if (!ok) break;

                // ---- segment epilogue: the row's output or partial ----
                if (sg.n > 0) ok = mbar_wait_warp(bar(W_OFULL + x), seg & 1, abort_flag);
                // (a parked partial overlays the rings, which the other tile's last product may still be reading)
                if (CL && ok && sg.n > 0 && two) ok = mbar_wait_warp(bar(W_OFULL + (x ^ 1)), seg & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const bool final_out = !CL && sg.slot < 0;
                const float inv = final_out ? inv_sum(l_run) : 1.f;
                __nv_bfloat16* orow = p.out + (((size_t)sg.b * N + node) * p.Hq + head) * HD;
                float4* prow = (CL ? reinterpret_cast<float4*>(sm + R::OFF_K) : p.part_o + (size_t)(final_out ? 0 : sg.slot) * (HD / 4) * kRows) + lrow;
#pragma unroll
                for (int c = 0; c < HD / 32; ++c) {
                    uint32_t o[32];
                    tmem_ld32(o_addr + c * 32, o);
                    tmem_wait_ld();
                    float v[32];
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = has_o ? __uint_as_float(o[e]) : 0.f;   // (undefined where no product ran)
                    if (final_out) {
                        if (row_ok) {
#pragma unroll
                            for (int c8 = 0; c8 < 4; ++c8)
                                *reinterpret_cast<uint4*>(orow + c * 32 + c8 * 8) =
                                    make_uint4(pack_bf16(v[8 * c8] * inv, v[8 * c8 + 1] * inv), pack_bf16(v[8 * c8 + 2] * inv, v[8 * c8 + 3] * inv),
                                               pack_bf16(v[8 * c8 + 4] * inv, v[8 * c8 + 5] * inv), pack_bf16(v[8 * c8 + 6] * inv, v[8 * c8 + 7] * inv));
                        }
                    } else if (CL || row_ok) {
#pragma unroll
                        for (int c4 = 0; c4 < 8; ++c4)
                            prow[(size_t)(c * 8 + c4) * kRows] = make_float4(v[4 * c4], v[4 * c4 + 1], v[4 * c4 + 2], v[4 * c4 + 3]);
                    }
                }
                const float2 stat = make_float2(l_run > 0.f ? m_ref : -INFINITY, l_run);
                if (CL) {
                    reinterpret_cast<float2*>(sm + R::OFF_K + (HD / 4) * kRows * 16)[lrow] = stat;
                } else if (row_ok) {
                    if (final_out) {
                        if (p.lse) p.lse[((size_t)sg.b * p.Hq + head) * N + node] =
                            l_run > 0.f ? (m_ref + log2f(l_run)) * 0.6931471805599453f : -INFINITY;
                    } else {
                        p.part_ml[(size_t)sg.slot * kRows + lrow] = stat;
                    }
                }
                tc_fence_before();
                mbar_arrive(bar(W_OFREE + x));
                ++seg;
            }
        }
        if (CL) {
            __syncwarp();
            cluster_merge<kRows, HD>(p, cl_seg, ck, cr, base + R::OFF_K, base + R::OFF_K + (HD / 4) * kRows * 16, tid - 128, abort_flag);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (CL) cluster_wait();                    // nobody leaves while a peer may still read its shared memory
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(TMEM_COLS) : "memory");
    }
    if (tid == 0 && *abort_flag) atomicCAS(p.status, 0, (int)VISPEC_E_TIMEOUT);
}

}  // namespace

// Largest number of co-resident clusters of each size, found once per device.
static int g_max_clusters[9];

cudaError_t init_attn_tc5_wide() {
    const void* kernels[6] = {(const void*)attn_tc5_wide_kernel<false, false, 128>, (const void*)attn_tc5_wide_kernel<true, false, 128>,
                              (const void*)attn_tc5_wide_kernel<false, true, 128>, (const void*)attn_tc5_wide_kernel<true, true, 128>,
                              (const void*)attn_tc5_wide_kernel<false, false, 64>, (const void*)attn_tc5_wide_kernel<true, false, 64>};
    for (const void* k : kernels) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_ALLOC);
        if (e != cudaSuccess) return e;
    }
    for (cudaError_t m : {init_merge<256, 128>(), init_merge<256, 64>()})
        if (m != cudaSuccess) return m;
    for (int k = 1; k <= 8; ++k) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(k * 64); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = SMEM_ALLOC;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = k; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, attn_tc5_wide_kernel<true, false, 128>, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
        g_max_clusters[k] = n;
    }
    return cudaSuccess;
}

WidePlan attn_tc5_wide_plan(const AttnArgs& a) {
    WidePlan w = {0, 0, 1e30};
    const int rows_total = (a.Hq / a.Hkv) * a.N;
    const int nmb = (rows_total + kRows - 1) / kRows, units = a.B * a.Hkv * nmb;
    if (rows_total <= 128 || a.rope_table || nmb > a.sm_count) return w;
    const int slots = (a.kv_len_hint > 0 && a.kv_len_hint + a.N < a.S_max) ? a.kv_len_hint + a.N : a.S_max;
    const double steps = (double)((slots + STEP - 1) / STEP), hbm = a.D / 128.0;
    // (fixed part and time of a 128-token step of both tiles, fitted like the one-tile kernel's estimates in attn_tc5.cu)
    if (a.tc5_path != 1 && a.tc5_path != 3) {
        int best = 0;
        for (int k = 1; k <= 8; ++k)
            if (units * k <= a.sm_count && g_max_clusters[k] >= units) best = k;
        if (best) {
            const double per = (double)(((int)steps + best - 1) / best);
            w.ck = best; w.grid = units * best;
            w.est_us = (a.D == 64 ? 13.5 : 16.0) + per * fmax(a.D == 64 ? 1.65 : 1.8, (double)units * best * 0.0093 * hbm / nmb);
            if (a.tc5_path == 2) return w;
        }
    }
    const int groups_max = a.sm_count / nmb;
    const long long t_max = (long long)a.B * a.Hkv * (long long)((a.S_max + STEP - 1) / STEP);
    const int groups = (int)(t_max < groups_max ? t_max : groups_max);
    if (kCounterBytes + (size_t)2 * groups * nmb * kRows * (a.D * 4 + 8) > a.ws_bytes) return w;
    const int heads = a.B * a.Hkv;
    const double T = steps * heads;
    double n = fmin((double)groups, fmax(1.0, floor(T / 2.0)));
    double uneven = 0.0;                       // ranges that cross heads: two segments in some groups
    if (heads <= n) {                          // as sched_ctas counts the groups
        const double r = floor(n / heads) * heads;
        if (ceil(T / r) - ceil(T / n) <= 3.0) n = r;
        else uneven = 3.0;
    }
    const double est = uneven + (a.D == 64 ? 13.7 : 15.5) + ceil(T / n) * fmax(a.D == 64 ? 1.6 : 2.0, n * 0.0093 * hbm) + (heads > n ? 11.0 * heads / n : 0.0);
    if (est < w.est_us) { w.ck = 0; w.grid = groups * nmb; w.est_us = est; }
    return w;
}

cudaError_t launch_attn_tc5_wide(const AttnArgs& a, const WidePlan& w, cudaStream_t st, int* n_launches) {
    const int n_mblocks = ((a.Hq / a.Hkv) * a.N + kRows - 1) / kRows, units = a.B * a.Hkv * n_mblocks;
    Tc5Params p = {};
    p.q = (const __nv_bfloat16*)a.q; p.kv_len = a.kv_len; p.mask = a.mask;
    p.out = (__nv_bfloat16*)a.out; p.lse = a.lse;
    unsigned char* ws = (unsigned char*)a.ws + kCounterBytes;
    p.part_o = (float4*)ws;
    p.part_ml = (float2*)(ws + (size_t)2 * w.grid * kRows * a.D * 4);
    p.B = a.B; p.N = a.N; p.Hq = a.Hq; p.Hkv = a.Hkv; p.S_max = a.S_max; p.n_mblocks = n_mblocks;
    p.grid_attn = w.grid; p.min_steps = 2; p.early = a.early_prefetch ? 1 : 0; p.step = STEP; p.lock = 1;
    p.scale_log2 = a.scale * 1.4426950408889634f;
    p.status = a.status;
    const PagedArgs pa = {a.block_table, a.table_stride, a.page_rows, a.num_blocks, a.Hkv, a.N, a.token_major, a.status, nullptr};
    auto launch = [&](auto kernel) {
        return launch_pdl(kernel, dim3(w.grid), dim3(kThreads), SMEM_ALLOC, st, w.ck, *a.k_map, *a.v_map, p, pa);
    };
    cudaError_t err;
    if (w.ck > 0) err = a.D == 64 ? launch(attn_tc5_wide_kernel<true, false, 64>)
                                  : a.page_rows ? launch(attn_tc5_wide_kernel<true, true, 128>) : launch(attn_tc5_wide_kernel<true, false, 128>);
    else err = a.D == 64 ? launch(attn_tc5_wide_kernel<false, false, 64>)
                         : a.page_rows ? launch(attn_tc5_wide_kernel<false, true, 128>) : launch(attn_tc5_wide_kernel<false, false, 128>);
    if (err != cudaSuccess) return err;
    ++*n_launches;
    if (w.ck > 0) return cudaSuccess;
    err = a.D == 64 ? launch_merge<256, 64>(p, units, w.grid, st) : launch_merge<256, 128>(p, units, w.grid, st);
    if (err != cudaSuccess) return err;
    ++*n_launches;
    return cudaSuccess;
}

}  // namespace vispec
