// Sampled (temperature > 0) acceptance on a draft tree (Sec. 3.1): a drafted token x is kept with probability
// min(1, p(x)/p^(x)); after a rejection the target distribution becomes norm(max(0, p - p^)); the children of
// the current node are decided one after the other and the token after the last kept node is drawn from what
// remains.
//
// What is kept in registers instead of a residual vector: after k rejections at one node the residual is
// proportional to m_k = max(0, p - c_k p^) with c_0 = 0, c_{k+1} = c_k + S_k and S_k = sum(m_k) (S_0 taken as 1:
// the rule compares against p itself), because max(0, max(0, p - c p^)/S - p^) = max(0, p - (c + S) p^)/S.
// A decision needs two scalars of the node's rows; only a rejection needs a pass over the two rows (2 * V * 4
// bytes) to form the next S, and that pass also leaves per-warp partial sums that locate the bonus token, so the
// draw re-reads one warp's slice only.
//
// What bounds it is a chain of dependent passes, each one DRAM round trip, the slice through one SM's load path, fp64
// sums and a cluster barrier, so the work of a pass is spread wide and nothing is fetched twice: one cluster per
// sequence (16 CTAs where that many SMs are free for every sequence, else 8; 1 for small vocabularies), 1024 threads
// per CTA; the slices go to shared memory by asynchronous copies (all in flight at once) and stay there while the walk
// stays at the node, so that a further rejection there costs no memory round trip; the root's rows are fetched while
// the tree and the decision scalars still are (the root is where the first rejection, if any, needs them).
// With the commit behind it, us per call, 8 CTAs re-reading the rows in every pass -> this: V = 152064, N = 60, one
// sequence 25.3 -> 18.6, four 28.3 -> 21.6; V = 32000, one sequence 17.3 -> 14.1.
//
// Every CTA takes the same decisions from the same numbers: a CTA's sum is pushed into every peer's shared memory ahead
// of a hardware cluster barrier and summed by everyone in the same order, so S is bit-identical in the cluster.  (The first
// push follows a barrier phase that every CTA arrives at when it starts: nothing is written into a CTA that does not run yet.)  Sums
// and comparisons are fp64 (the inputs are fp32): the decisions then differ from a sequential fp64 evaluation only
// where a uniform falls within ~1e-15 of a threshold.
#include "launch.cuh"
#include "vispec_internal.h"

namespace vispec {
namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxCluster = 16;
constexpr int kCacheBytes = 200 * 1024;          // most shared memory a CTA keeps its slices of a node's two rows in

__device__ __forceinline__ void record_status_as(int* status, int code) {
    if (status) atomicCAS(status, 0, code);
}
__device__ __forceinline__ uint32_t cl_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cl_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The barrier in two halves (each taken by whole warps): what a CTA writes into a peer's shared memory comes after its wait
// for the phase in which every CTA, the peer too, has arrived.
__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_st_f64(const double* local, uint32_t rank, double v) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(local);
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}
template <int BYTES>
__device__ __forceinline__ void copy_async(const float* dst, const float* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ double weight(float p, float ph, double c) {
    return fmax(0.0, (double)p - c * (double)ph);
}

// The slice of [0, V) that warp w of CTA `rank` sums: CTAs take consecutive ranges, warps consecutive sub-ranges,
// both rounded to 4 elements so that 16-byte loads stay aligned when V is a multiple of 4.
struct Slice { int lo, hi; };
__host__ __device__ __forceinline__ int cta_elems(int V, int csize) { return (((V + csize - 1) / csize) + 3) & ~3; }
__device__ __forceinline__ Slice warp_slice(int V, int rank, int csize, int w) {
    const int per = cta_elems(V, csize);
    const int wper = (((per + kWarps - 1) / kWarps) + 3) & ~3;
    const int clo = min(V, rank * per), chi = min(V, clo + per);
    Slice s;
    s.lo = min(chi, clo + w * wper);
    s.hi = min(chi, s.lo + wper);
    return s;
}

// A CTA's slices of one node's two rows: elements [clo, clo + cap) of each are kept in shared memory (every thread
// copies in, and later reads, the same elements), what lies beyond is read from global memory.
struct Rows {
    const float* pt; const float* ph;      // the node's rows in global memory
    float* sp; float* sph;                  // kept elements
    int clo, cap;
    __device__ __forceinline__ bool kept(int e) const { return e - clo < cap; }
};

template <bool VEC>
__device__ __forceinline__ void rows_fetch(const Rows& r, Slice s, int lane) {
    constexpr int PER = VEC ? 4 : 1;
    const int hi = min(s.hi, r.clo + r.cap);
    for (int e = s.lo + lane * PER; e < hi; e += 32 * PER) {
        copy_async<PER * 4>(r.sp + (e - r.clo), r.pt + e);
        copy_async<PER * 4>(r.sph + (e - r.clo), r.ph + e);
    }
}

template <bool VEC>
__device__ __forceinline__ double slice_sum(const Rows& r, double c, Slice s, int lane) {
    double acc = 0.0, acc2 = 0.0;
    if (VEC) {
        auto four = [&](const float4& a, const float4& b) {
            acc += weight(a.x, b.x, c) + weight(a.y, b.y, c);
            acc2 += weight(a.z, b.z, c) + weight(a.w, b.w, c);
        };
        const int mid = min(s.hi, r.clo + r.cap);             // (a multiple of 4 from s.lo on)
        int e = s.lo + lane * 4;
#pragma unroll 4
        for (; e < mid; e += 128)
            four(*reinterpret_cast<const float4*>(r.sp + (e - r.clo)), *reinterpret_cast<const float4*>(r.sph + (e - r.clo)));
#pragma unroll 4
        for (; e < s.hi; e += 128)
            four(__ldg(reinterpret_cast<const float4*>(r.pt + e)), __ldg(reinterpret_cast<const float4*>(r.ph + e)));
    } else {
#pragma unroll 4
        for (int e = s.lo + lane; e < s.hi; e += 32)
            acc += r.kept(e) ? weight(r.sp[e - r.clo], r.sph[e - r.clo], c) : weight(__ldg(r.pt + e), __ldg(r.ph + e), c);
    }
    acc += acc2;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

// By a whole warp: first index i < n <= 32 with (base + v[0] + ... + v[i]) > target, else the last i with v[i] > 0, else
// -1; *before = the running sum ahead of the index returned.
__device__ __forceinline__ int locate(const double* v, int n, double base, double target, double* before, int lane) {
    const double mine = lane < n ? v[lane] : 0.0;
    double incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, lane < n && base + incl > target);
    const unsigned pos = __ballot_sync(0xffffffffu, mine > 0.0);
    const int i = hit ? __ffs(hit) - 1 : 31 - __clz(pos);      // (pos == 0: -1)
    *before = base + __shfl_sync(0xffffffffu, incl - mine, i < 0 ? 0 : i);
    return i;
}

template <bool VEC>
__global__ void __launch_bounds__(kThreads)
accept_sampled_kernel(const int32_t* __restrict__ draft_ids, const int32_t* __restrict__ parents,
                      const float* __restrict__ p, const float* __restrict__ p_hat,
                      const float* __restrict__ u_accept, const float* __restrict__ u_bonus, int N, int V, int cap,
                      int32_t* __restrict__ path, int32_t* __restrict__ accept_len, int32_t* __restrict__ bonus,
                      int* status) {
    extern __shared__ __align__(16) float kept_rows[];      // [2][cap]
    __shared__ int32_t par[VISPEC_MAX_TREE_NODES], ids[VISPEC_MAX_TREE_NODES], spath[VISPEC_MAX_TREE_NODES];
    __shared__ float ua[VISPEC_MAX_TREE_NODES];
    __shared__ float px_of[VISPEC_MAX_TREE_NODES], phx_of[VISPEC_MAX_TREE_NODES];   // p[parent][token], p^[parent][token] per node
    __shared__ uint32_t kids[VISPEC_MAX_TREE_NODES][4];      // children of a node, one bit each
    __shared__ double seg[kWarps];                           // this CTA's per-warp sums of the last pass
    __shared__ double allpart[2][kMaxCluster];               // every CTA's sum, by pass parity (written by the whole cluster)
    __shared__ double sh_c, sh_S;
    __shared__ int sh_cur, sh_action, sh_bad, sh_stop, sh_len;

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int csize = (int)cl_size(), rank = (int)cl_rank();
    const int b = blockIdx.x / csize;
    const size_t nb = (size_t)b * N;
    const Slice slice = warp_slice(V, rank, csize, w);
    Rows rows;
    rows.clo = min(V, rank * cta_elems(V, csize)); rows.cap = cap;
    rows.sp = kept_rows; rows.sph = kept_rows + cap;
    auto at_node = [&](int i) { rows.pt = p + (nb + i) * (size_t)V; rows.ph = p_hat + (nb + i) * (size_t)V; };

    if (tid == 0) { sh_bad = 0; sh_stop = 0; }
    if (tid < VISPEC_MAX_TREE_NODES * 4) (&kids[0][0])[tid] = 0u;
    __syncthreads();
    cl_arrive();                                 // this CTA runs; waited for ahead of the first push, behind the first loads
    bool peers_run = false;
    pdl_wait();
    int pr = 0, id = 0;
    if (tid < N) { pr = parents[nb + tid]; id = draft_ids[nb + tid]; ua[tid] = u_accept[nb + tid]; }
    const float ub = __ldg(u_bonus + b);
    at_node(0);
    rows_fetch<VEC>(rows, slice, lane);                      // the root's rows, on the way from here on
    int kept_node = 0;
    if (tid < N) {
        par[tid] = pr;
        ids[tid] = id;
        const bool ok = tid == 0 ? pr == -1 : (pr >= 0 && pr < tid && id >= 0 && id < V);
        if (!ok) atomicOr(&sh_bad, tid == 0 || pr < 0 || pr >= tid ? 1 : 2);
        else if (tid > 0) {
            // the two scalars the node's decision needs, for every node at once
            const size_t row = (nb + pr) * (size_t)V + id;
            px_of[tid] = __ldg(p + row);
            phx_of[tid] = __ldg(p_hat + row);
            atomicOr(&kids[pr][tid >> 5], 1u << (tid & 31));
        }
    }
    __syncthreads();
    if (sh_bad) {                                // the same verdict in every CTA of the cluster: all leave here
        copy_wait();
        if (rank == 0) {
            if (tid < N) path[nb + tid] = -1;
            if (tid == 0) {
                accept_len[b] = 0;
                bonus[b] = -1;
                record_status_as(status, (sh_bad & 1) ? VISPEC_E_BAD_TREE : VISPEC_E_RANGE);
            }
        }
        __syncwarp();
        cl_wait();
        return;
    }

    enum { PASS = 0, DRAW = 1 };
    // walk state, meaningful in thread 0 only: the children of `cur` not decided yet are the bits left in `todo`
    int cur = 0, len = 1;
    uint32_t todo[4];
    double c = 0.0, S = 1.0;
    bool have_pass = false;
    auto children = [&](int i) {
#pragma unroll
        for (int x = 0; x < 4; ++x) todo[x] = kids[i][x];
    };
    if (tid == 0) { spath[0] = 0; children(0); }

    for (int iter = 0; iter < 2 * N + 4; ++iter) {
        if (tid == 0) {
            int action = -1;
            while (action < 0) {
                int ch = -1;
#pragma unroll
                for (int x = 3; x >= 0; --x)
                    if (todo[x]) ch = x * 32 + __ffs(todo[x]) - 1;
                if (ch < 0) {                    // no child left: draw from what remains (needs the sums of a pass)
                    action = have_pass ? DRAW : PASS;
                    break;
                }
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    if (x == (ch >> 5)) todo[x] &= todo[x] - 1;
                const double px = (double)px_of[ch], phx = (double)phx_of[ch];
                const double num = fmax(0.0, px - c * phx);
                if ((double)ua[ch] * S * phx < num) {          // kept: u < min(1, r(x)/p^(x)), r = m/S
                    cur = ch;
                    spath[len++] = ch;
                    children(ch);
                    c = 0.0; S = 1.0; have_pass = false;
                } else {                                        // rejected: next residual needs its sum
                    c += S;
                    action = PASS;
                }
            }
            sh_action = action; sh_c = c; sh_cur = cur;
        }
        __syncthreads();
        if (sh_action != PASS) break;

        // ---- one pass over the two rows of node sh_cur ----
        if (sh_cur != kept_node) {
            copy_wait();                         // nothing of the node before is still on its way into the same place
            kept_node = sh_cur;
            at_node(kept_node);
            rows_fetch<VEC>(rows, slice, lane);
        }
        copy_wait();
        const double sum = slice_sum<VEC>(rows, sh_c, slice, lane);
        if (lane == 0) seg[w] = sum;
        __syncthreads();
        if (!peers_run) { cl_wait(); peers_run = true; }
        const int parity = iter & 1;
        if (w == 0) {
            double t = seg[lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane < csize) cl_st_f64(&allpart[parity][rank], (uint32_t)lane, t);
        }
        cl_sync();                               // every CTA's sum has reached every CTA
        if (w == 0) {
            double t = lane < csize ? allpart[parity][lane] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);   // the same order in every CTA
            if (t > 0.0) {
                S = t; have_pass = true;
            } else if (c == 0.0) {               // the target row itself has no weight: nothing to draw
                if (lane == 0) sh_stop = 1;      // (c is thread 0's: only its verdict is kept)
            } else {                             // empty residual: stop deciding, draw from the target row
                c = 0.0; S = 1.0; have_pass = false; todo[0] = todo[1] = todo[2] = todo[3] = 0u;
            }
            if (lane == 0) sh_S = S;
        }
        if (tid == 0 && sh_stop) sh_action = -1;
        if (tid == 0) sh_len = iter & 1;         // parity of the pass whose sums stand (overwritten below with the length)
        __syncthreads();
        if (sh_stop) break;
    }

    // ---- outputs: path and length from rank 0, the bonus token from the warp whose slice holds it ----
    const int last_parity = sh_len;
    __syncthreads();
    if (tid == 0) sh_len = len;
    __syncthreads();
    if (rank == 0) {
        if (tid == 0) accept_len[b] = sh_len;
        if (tid < N) path[nb + tid] = tid < sh_len ? spath[tid] : -1;
    }

    if (sh_stop || sh_action != DRAW) {           // no weight to draw from (or, never, the pass bound ran out)
        if (rank == 0 && tid == 0) {
            bonus[b] = -1;
            if (!sh_stop) record_status_as(status, VISPEC_E_TIMEOUT);
        }
    } else {
        const double target = (double)ub * sh_S;
        double base = 0.0;
        const int r_star = locate(allpart[last_parity], csize, 0.0, target, &base, lane);
        if (r_star == rank) {
            double base2 = base;
            const int w_star = locate(seg, kWarps, base, target, &base2, lane);
            if (w_star == w) {
                const double cc = sh_c;
                double run = base2;
                int found = -1, last_pos = -1;
                for (int e0 = slice.lo; e0 < slice.hi && found < 0; e0 += 128) {
                    double m[4];
                    const int e = e0 + lane * 4;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        m[j] = 0.0;
                        if (e + j < slice.hi)
                            m[j] = rows.kept(e + j) ? weight(rows.sp[e + j - rows.clo], rows.sph[e + j - rows.clo], cc)
                                                    : weight(__ldg(rows.pt + e + j), __ldg(rows.ph + e + j), cc);
                    }
                    const double mine = (m[0] + m[1]) + (m[2] + m[3]);
                    double incl = mine;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const double t = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += t;
                    }
                    const double chunk = __shfl_sync(0xffffffffu, incl, 31);
                    // the first lane whose running sum passes the target, then the element inside that lane
                    const unsigned hit = __ballot_sync(0xffffffffu, run + incl > target);
                    int cand = -1;
                    if (hit) {
                        const int l0 = __ffs(hit) - 1;
                        if (lane == l0) {
                            double r2 = run + (incl - mine);
                            int last_in = -1;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                if (m[j] > 0.0) last_in = e + j;
                                if (cand < 0 && r2 + m[j] > target) cand = e + j;
                                r2 += m[j];
                            }
                            if (cand < 0) cand = last_in;   // rounding between the two summation orders
                        }
                        cand = __shfl_sync(0xffffffffu, cand, l0);
                    }
                    int lp = -1;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (m[j] > 0.0) lp = e + j;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) lp = max(lp, __shfl_xor_sync(0xffffffffu, lp, o));
                    if (cand >= 0) found = cand;
                    else if (lp >= 0) last_pos = lp;
                    run += chunk;
                }
                if (found < 0) found = last_pos;            // the slice's sum said "here" but the rescan fell short
                if (lane == 0) bonus[b] = found;
            }
        }
    }
    copy_wait();
    __syncwarp();
    if (!peers_run) cl_wait();                   // (no pass was made)
    cl_sync();                                   // nobody leaves while a peer may still push its sum here
}

// Clusters of 16 CTAs (with the most shared memory they use) that the device holds at once; found with the context.
int g_wide_clusters[64];
int max_wide_clusters() {
    int dev = 0;
    return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 ? g_wide_clusters[dev] : 0;
}

}  // namespace

cudaError_t init_accept_sampled(int device) {
    const void* kernels[2] = {(const void*)accept_sampled_kernel<true>, (const void*)accept_sampled_kernel<false>};
    for (const void* k : kernels) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kCacheBytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16 * 16); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kCacheBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 16; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, accept_sampled_kernel<true>, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    if (device >= 0 && device < 64) g_wide_clusters[device] = n;
    return cudaSuccess;
}

cudaError_t launch_accept_sampled(const int32_t* draft_ids, const int32_t* parents, const float* p, const float* p_hat,
                                  const float* u_accept, const float* u_bonus, int B, int N, int V, int32_t* path,
                                  int32_t* accept_len, int32_t* bonus, int* status, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    // Cluster size.  A pass is 2 * V * 4 bytes through the cluster's load paths: 16 CTAs halve it against 8, as long as
    // every sequence's cluster finds its SMs at once; below 8192 tokens one CTA reads the rows in the time a cluster
    // barrier takes.
    int cl = 1;
    if (V >= 8192) cl = B <= max_wide_clusters() ? 16 : 8;
    const int cap = min(cta_elems(V, cl), kCacheBytes / 8 / 128 * 128);
    if (V % 4 == 0)
        return launch_pdl(accept_sampled_kernel<true>, dim3(B * cl), dim3(kThreads), (size_t)cap * 8, st, cl, draft_ids, parents,
                          p, p_hat, u_accept, u_bonus, N, V, cap, path, accept_len, bonus, status);
    return launch_pdl(accept_sampled_kernel<false>, dim3(B * cl), dim3(kThreads), (size_t)cap * 8, st, cl, draft_ids, parents, p,
                      p_hat, u_accept, u_bonus, N, V, cap, path, accept_len, bonus, status);
}

}  // namespace vispec
