// bfs_small.cu -- the small push-queue levels of a search on a graph of low
// degree (grids, road networks), run by one thread-block cluster.
//
// Such a search has thousands of levels of a few thousand vertices, and a
// level costs a chain of dependent round trips whatever its size.  In the
// general kernel the chain is: queue entry (L2), column (HBM), visited OR (L2)
// with the new vertex's row bounds (HBM), queue reservation, store drain,
// barrier -- 6.2 us a level on the relabelled 4096^2 grid.  Here it is one
// memory round trip and one message between the CTAs:
//   - adjacency in rows of W = 4 or 8 entries (-1 for none), one aligned
//     sector a vertex, built once per graph.  A candidate's row is loaded
//     beside the OR that claims it, and the claimer puts it in the queue
//     entry {vertex, parent, row}: the next level needs no load at all
//     before its own ORs;
//   - queues in shared memory.  The k-th claim of CTA c goes to CTA
//     (c + k) mod CL, into the part of its queue that belongs to c, as a
//     store through distributed shared memory: no reservation at the
//     receiver, and every CTA expands the same share of the next frontier
//     wherever the wavefront runs (a CTA that kept its own claims would keep
//     its patch of it).  The claim counts are pushed to every CTA the same
//     way, so that all of a level's reads are local;
//   - the stores signal the level themselves: they are asynchronous and
//     counted by an mbarrier of the receiver (two, in turn: a sender is at most
//     a level ahead), and each sender arrives there with the bytes it has
//     stored.  A cluster barrier waits for every store before it, those to
//     memory too, and took 0.35 us a level more;
//   - depth and parent of a vertex are stored when its entry is expanded, at
//     the start of the next level, and nothing waits for them.
// A level takes 1.7 us up to 2 M cells (OR and row 0.7 us, append 0.3, the
// message and the CTA barriers the rest) and 3.1 us on the 4096^2 grid, whose rows
// and outputs (400 MB touched at random by one cluster) miss L2 and the TLB: a
// search of that grid 41.7 -> 18.2 ms.
// The level that would not fit, or that is not a push-queue level, is handed
// to the grid-wide kernel with the state that kernel continues from.
#include "level.cuh"

#include <algorithm>

namespace bfsgb {

namespace {

constexpr int ELL_T = 1024;
// A level's wait is never given up earlier, whatever the caller's limit.  No
// input makes these waits run out; a build with 0 leaves them to the caller's
// limit alone and polls, where a try_wait sleeps in the hardware for longer than
// a level takes.
#ifndef BFS_SMALL_WAIT_NS
#define BFS_SMALL_WAIT_NS 1000000000ll
#endif
constexpr long long ELL_WAIT_NS = BFS_SMALL_WAIT_NS;
constexpr long long ELL_DRAIN_NS = 1000000000ll;  // limit of a failed launch's waits for the stores under way

template <int W>
struct EllCfg {
    static constexpr int PITCH = W + 2;             // {vertex, parent, row}, 8-byte multiples
    static constexpr int PART = W == 4 ? 256 : 160; // entries a CTA's queue holds from one sender
    static constexpr int GROUPS = ELL_T / W;        // entries a CTA expands at a time, W threads each
};

template <int W>
size_t ell_smem(int cl) {
    return (size_t)2 * cl * EllCfg<W>::PART * EllCfg<W>::PITCH * sizeof(int32_t);
}

// Largest frontier a level may have: a CTA gets at most f / cl + cl of its
// entries, claims at most W for each, and cl * PART claims fit.
template <int W>
int64_t ell_max_frontier(int cl) {
    return (int64_t)cl * (cl * EllCfg<W>::PART / W - cl);
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned map_shared(const void* p, unsigned rank) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// Stores to a CTA's shared memory that its mbarrier `bar` counts, in bytes, as they land
__device__ __forceinline__ void st_async2(unsigned a, int x, int y, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(a), "r"(x),
                 "r"(y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async(unsigned a, unsigned x, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a), "r"(x), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, unsigned x) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned long long* b, int arrivals) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(b)), "r"(arrivals)
                 : "memory");
}
// One arrival at a CTA's mbarrier, with the bytes this CTA's stores bring it.
// Relaxed: a release waits for the CTA's depth and parent stores, which no one
// reads here (2.17 us a level against 1.67).  What the receiver reads are the
// counted stores alone; the sender's own reads of the queue part that is
// written next were used, and its ORs on P returned, before this.
__device__ __forceinline__ void mbar_arrive_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
#if BFS_SMALL_WAIT_NS > 0
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
#else
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
#endif
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// false: the limit has passed, and still nothing (this CTA may have been off
// the GPU since its last try)
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, int64_t limit_ns) {
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    while (!mbar_try(bar, parity))
        if ((int64_t)(globaltimer_ns() - t0) > limit_ns) return mbar_try(bar, parity);
    return true;
}
// The barrier that counts the stores of level l into the next one's queues,
// and the parity of its phase (the two take turns).
__device__ __forceinline__ int level_bar(int l) { return (l & 1) ^ 1; }
__device__ __forceinline__ unsigned level_parity(int l) { return (unsigned)(l >> 1) & 1u; }
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void ell_row(const int32_t* __restrict__ ell, int v, int (&a)[4]) {
    const int4 x = __ldg(reinterpret_cast<const int4*>(ell) + v);
    a[0] = x.x, a[1] = x.y, a[2] = x.z, a[3] = x.w;
}
__device__ __forceinline__ void ell_row(const int32_t* __restrict__ ell, int v, int (&a)[8]) {
    const int4 x = __ldg(reinterpret_cast<const int4*>(ell) + 2ll * v), y = __ldg(reinterpret_cast<const int4*>(ell) + 2ll * v + 1);
    a[0] = x.x, a[1] = x.y, a[2] = x.z, a[3] = x.w;
    a[4] = y.x, a[5] = y.y, a[6] = y.z, a[7] = y.w;
}

// Claims of a CTA in one level, and their degree sum above them: at most
// cl * PART claims of degree W, so neither field overflows.
constexpr int CNT_BITS = 14;

// Entries CTA d receives from a sender with `cnt` claims, (d - sender) mod cl = off, cl = 1 << lg.
__device__ __forceinline__ int part_len(int cnt, int off, int lg) { return (cnt - off + (1 << lg) - 1) >> lg; }

// SPEC: the rows of all candidates are loaded beside their ORs, not only the
// claimed ones' after them.
template <int W, bool SPEC>
__global__ void __launch_bounds__(ELL_T, 1) bfs_small_kernel(Params1 p) {
    using C = EllCfg<W>;
    static_assert(16 * C::PART < (1 << CNT_BITS) && 16 * C::PART * W < (1 << (32 - CNT_BITS)), "packed counts");
    extern __shared__ __align__(16) int32_t ell_q[];  // [2][cl][PART][PITCH]
    __shared__ unsigned s_cnt[2][16];                 // packed claims of each CTA, by level parity
    __shared__ unsigned s_mine[2];                    // this CTA's, being counted
    __shared__ unsigned long long s_bar[2];           // a level's arrivals and bytes, by level parity
    __shared__ unsigned s_left[16];                   // each CTA's levels sent as it left them, bit 0: it gave up a wait
    const int cl = (int)gridDim.x, lg = __ffs(cl) - 1, rank = (int)cluster_rank();
    const int lane = (int)lane_id();
    const int grp = (int)threadIdx.x / W, j = (int)threadIdx.x % W;
    const int per = C::GROUPS / cl;            // groups that expand the entries of one sender
    const int from = grp / per, r = grp % per; // warp-uniform sender: per * W >= 32
    Ctl1* ctl = p.ctl;

    if (threadIdx.x < 32) {
        const int s = p.src_value;
        if (lane < 16) {
            s_cnt[0][lane] = 0;
            s_cnt[1][lane] = 0;
        }
        __syncwarp();
        if (lane == 0) {
            s_mine[0] = s_mine[1] = 0;
            mbar_init(&s_bar[0], cl);
            mbar_init(&s_bar[1], cl);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            int row[W], deg = 0;
            ell_row(p.ell, s, row);
#pragma unroll
            for (int k = 0; k < W; ++k) deg += row[k] >= 0;
            s_cnt[0][0] = (unsigned)deg << CNT_BITS | 1u;  // F_0 as if CTA 0 had claimed it
            if (rank == 0) {
                int32_t* e = ell_q;
                e[0] = s;
                e[1] = s;
#pragma unroll
                for (int k = 0; k < W; ++k) e[2 + k] = row[k];
                // P holds the vertices without an edge; the source, and the bits past n
                atomicOr(p.P + (s >> 5), 1u << (s & 31));
                if (p.n & 31) atomicOr(p.P + p.W - 1, ~((1u << (p.n & 31)) - 1u));
            }
        }
    }
    cluster_sync();

    // the counters fit in 32 bits: a CSR has less than 2^31 entries
    int level = 0, m_u = (int)p.m, f_prev = 0, f = 0, e_f = 0;
    bool done = false, gave_up = false;
    for (;; ++level) {
        const int par = level & 1;
        const unsigned mine = lane < cl ? s_cnt[par][lane] : 0u;
        f = (int)__reduce_add_sync(0xffffffffu, mine & ((1u << CNT_BITS) - 1u));
        e_f = (int)__reduce_add_sync(0xffffffffu, mine >> CNT_BITS);
        if (f == 0) {
            if (rank == 0 && threadIdx.x == 0 && p.log && level < p.log_cap) {
                bfs_level_record rec;
                rec.level = level;
                rec.dir = -1;
                rec.f = rec.e_f = 0;
                rec.m_u = m_u;
                rec.t_ns = (int64_t)globaltimer_ns();
                p.log[level] = rec;
            }
            done = true;
            break;
        }
        if (level >= p.max_levels) {
            if (rank == 0 && threadIdx.x == 0) atomicCAS(&ctl->bar.err, 0, (int)DEV_LEVELS);
            done = true;
            break;
        }
        // push_kind and heuristic_dir after a push level, in 32-bit integers
        // (the 64-bit conversions took a tenth of the level)
        const int mu = m_u - e_f;
        const bool pull = p.policy != BFS_POLICY_PUSH && (float)e_f * p.alpha > (float)mu && f > f_prev;
        if (pull || (float)f * p.gamma > (float)p.n || f > (int)p.small_ef_max) break;
        m_u = mu;
        if (rank == 0 && threadIdx.x == 0 && p.log && level < p.log_cap) {
            bfs_level_record rec;
            rec.level = level;
            rec.dir = BFS_DIR_PUSH_QUEUE;
            rec.f = f;
            rec.e_f = e_f;
            rec.m_u = m_u;
            rec.t_ns = (int64_t)globaltimer_ns();
            p.log[level] = rec;
        }
        const int len = part_len((int)(__shfl_sync(0xffffffffu, mine, from) & ((1u << CNT_BITS) - 1u)),
                                 (rank - from) & (cl - 1), lg);
        const int32_t* q = ell_q + ((size_t)par * cl + from) * C::PART * C::PITCH;
        int32_t* qn = ell_q + ((size_t)(par ^ 1) * cl + rank) * C::PART * C::PITCH;  // this CTA's part, at any receiver
        unsigned long long* const bar = &s_bar[level_bar(level)];
        for (int i0 = 0; i0 < len; i0 += per) {  // warp-uniform
            int u = -1, w = -1;
            if (i0 + r < len) {
                const int32_t* e = q + (i0 + r) * C::PITCH;
                const int up = e[1];
                u = e[0];
                w = e[2 + j];
                if (w == up) w = -1;  // the parent is visited
                if (j == 0) {
                    p.depth[u] = level;
                    if (p.parent) p.parent[u] = up;
                }
            }
            int row[W];
#pragma unroll
            for (int k = 0; k < W; ++k) row[k] = -1;
            bool won = false;
            if (w >= 0) {
                if (SPEC) ell_row(p.ell, w, row);  // in flight beside the OR; wasted where it loses
                const unsigned bit = 1u << (w & 31);
                won = !(atomicOr(p.P + (w >> 5), bit) & bit);
                if (!SPEC && won) ell_row(p.ell, w, row);
            }
            const unsigned cm = __ballot_sync(0xffffffffu, won);
            if (!cm) continue;
            int deg = 0;
#pragma unroll
            for (int k = 0; k < W; ++k) deg += row[k] >= 0;
            const unsigned es = __reduce_add_sync(0xffffffffu, won ? (unsigned)deg : 0u);
            unsigned base = 0;
            if (lane == 0) base = atomicAdd(&s_mine[par], es << CNT_BITS | (unsigned)__popc(cm));
            base = __shfl_sync(0xffffffffu, base, 0) & ((1u << CNT_BITS) - 1u);
            if (won) {
                const int k = (int)base + __popc(cm & lanemask_lt());
                const unsigned to = (unsigned)((rank + k) & (cl - 1));
                const unsigned a = map_shared(qn + (k >> lg) * C::PITCH, to), b = map_shared(bar, to);
                st_async2(a, w, u, b);
#pragma unroll
                for (int t = 0; t < W; t += 2) st_async2(a + 8 + 4 * t, row[t], row[t + 1], b);
            }
        }
        __syncthreads();  // every claim of the CTA is counted
        if (threadIdx.x < (unsigned)cl) {
            const unsigned to = threadIdx.x, m = s_mine[par], b = map_shared(bar, to);
            const int sent = part_len((int)(m & ((1u << CNT_BITS) - 1u)), ((int)to - rank) & (cl - 1), lg);
            st_async(map_shared(&s_cnt[par ^ 1][rank], to), m, b);
            mbar_arrive_tx(b, (unsigned)(sent * C::PITCH * (int)sizeof(int32_t)) + 4u);
        }
        if (threadIdx.x == 32) s_mine[par ^ 1] = 0;  // pushed a level ago, counts the next one
        f_prev = f;
        bool ok = true;
        if (threadIdx.x < 32) {
            ok = mbar_wait((unsigned)__cvta_generic_to_shared(bar), level_parity(level), p.timeout_ns);
            __syncwarp();
        }
        if (!__syncthreads_and(ok)) {  // CTA-uniform, but each CTA finds out for itself
            if (threadIdx.x == 0) atomicCAS(&ctl->bar.err, 0, (int)DEV_TIMEOUT_SMALL);
            gave_up = true;
            break;
        }
    }
    // No CTA leaves before all have stopped sending, and every CTA learns how
    // the others left.
    const int sent = level + (gave_up ? 1 : 0);  // levels whose stores this CTA has sent; it has waited for `level` of them
    if (threadIdx.x < (unsigned)cl) st_cluster(map_shared(&s_left[rank], threadIdx.x), (unsigned)sent << 1 | (gave_up ? 1u : 0u));
    cluster_sync();
    const unsigned left = lane < cl ? s_left[lane] : 0u;
    if (__any_sync(0xffffffffu, left & 1u)) {  // cluster-uniform: the search has failed for all
        // The cluster barrier does not order counted stores: some may still be on
        // their way to a CTA that did not wait for them.  A CTA sends a level only
        // when every CTA has sent the one before, so `sent` differs by one at most:
        // who is behind arrives for that level too, without stores, and everyone
        // waits for its own barrier up to it.
        const int last = (int)__reduce_max_sync(0xffffffffu, left >> 1);
        if (sent < last && threadIdx.x < (unsigned)cl) mbar_arrive_tx(map_shared(&s_bar[level_bar(last - 1)], threadIdx.x), 0u);
        if (threadIdx.x < 32) {
            for (int l = level; l < last; ++l)
                mbar_wait((unsigned)__cvta_generic_to_shared(&s_bar[level_bar(l)]), level_parity(l), ELL_DRAIN_NS);
        }
        cluster_sync();
        // nothing of the frontier is handed over: the CTAs have left at different levels
        f = 0;
        e_f = 0;
        done = true;
    }
    // The frontier F_level that was not expanded: depths and parents, and the
    // queue entries of the grid-wide kernel.  Nothing is left of a finished one.
    if (f > 0) {
        const int par = level & 1;
        const unsigned mine = lane < cl ? s_cnt[par][lane] & ((1u << CNT_BITS) - 1u) : 0u;
        int before = 0;  // entries of the CTAs before this one
        for (int d = 0; d < rank; ++d) {
            const int x = lane < cl ? part_len((int)mine, (d - lane) & (cl - 1), lg) : 0;
            before += (int)__reduce_add_sync(0xffffffffu, (unsigned)x);
        }
        int4* Q = par ? p.Q1 : p.Q0;
        for (int c = 0; c < cl; ++c) {
            const int len = part_len((int)__shfl_sync(0xffffffffu, mine, c), (rank - c) & (cl - 1), lg);
            const int32_t* q = ell_q + ((size_t)par * cl + c) * C::PART * C::PITCH;
            for (int i = (int)threadIdx.x; i < len; i += ELL_T) {
                const int u = q[i * C::PITCH];
                p.depth[u] = level;
                if (p.parent) p.parent[u] = q[i * C::PITCH + 1];
                Q[before + i] = make_int4(u, __ldg(p.row_ptr + u), __ldg(p.row_ptr + u + 1), 0);
            }
            before += len;
        }
    }
    if (rank == 0 && threadIdx.x == 0) {
        Counters* c = &ctl->slot[level % 3];  // the others are zero
        c->q_len = (unsigned long long)f;
        c->e_f = (unsigned long long)e_f;
        ctl->next_level = level;
        ctl->prev_dir = BFS_DIR_PUSH_QUEUE;
        ctl->bm_valid = -1;
        ctl->q_valid = level;
        // the grid-wide kernel takes a level's e_f off itself, but for level 0's
        ctl->m_u = level > 0 ? m_u : m_u - e_f;
        ctl->f_prev = f_prev;
        ctl->done = done ? 1 : 0;
        const int e = ld_volatile_i32(&ctl->bar.err);
        if (e) atomicCAS(p.sticky, 0, e);
    }
}

// ell[v][k] = k-th neighbour of v, or -1
__global__ void ell_build_kernel(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int32_t n, int w,
                                 int32_t* __restrict__ ell) {
    const int64_t total = (int64_t)n * w;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = i / w;
        const int b = __ldg(row_ptr + v) + (int)(i % w);
        ell[i] = b < __ldg(row_ptr + v + 1) ? __ldg(col + b) : -1;
    }
}

template <int W>
cudaLaunchConfig_t ell_config(int cl, cudaLaunchAttribute* attr, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl);
    cfg.blockDim = dim3(ELL_T);
    cfg.dynamicSmemBytes = ell_smem<W>(cl);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// CTAs of the cluster: 16 where the GPU can co-schedule them, else 8 (0: neither)
template <int W, bool SPEC>
int ell_cluster() {
    static int cached[64] = {};
    const int d = device_id();
    if (d < 0 || d >= 64) return 0;
    if (cached[d]) return cached[d] > 0 ? cached[d] : 0;
    int found = -1;
    auto k = bfs_small_kernel<W, SPEC>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ell_smem<W>(16)) == cudaSuccess) {
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        for (int cl : {16, 8}) {
            cudaLaunchAttribute attr[1];
            cudaLaunchConfig_t cfg = ell_config<W>(cl, attr, nullptr);
            int nc = 0;
            if (cudaOccupancyMaxActiveClusters(&nc, k, &cfg) == cudaSuccess && nc >= 1) {
                found = cl;
                break;
            }
        }
    }
    cudaGetLastError();  // an unsupported size leaves a non-sticky error
    cached[d] = found;
    return found > 0 ? found : 0;
}

}  // namespace

// Limit of a level's waits for a caller's limit
int64_t small_wait_ns(int64_t timeout_ns) { return std::max<int64_t>(timeout_ns, ELL_WAIT_NS); }

int ell_width(int32_t deg_max) { return deg_max <= 4 ? 4 : deg_max <= 8 ? 8 : 0; }

// Rows of ell_width entries in w->ell, made once per workspace.  False: no
// memory for them, they could not be launched, or the stream is being captured
// (no allocation there); the search then takes the general kernel.
bool ell_prepare(const bfs_graph* g, Workspace1* w, cudaStream_t st) {
    if (w->ell) return true;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    const int width = ell_width(g->deg_max);
    if (cudaMalloc(&w->ell, (size_t)g->n * width * sizeof(int32_t)) != cudaSuccess) {
        cudaGetLastError();
        w->ell = nullptr;
        return false;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min<int64_t>(div_up((int64_t)g->n * width, 256), (int64_t)num_sms() * 32));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    if (cudaLaunchKernelEx(&cfg, ell_build_kernel, (const int32_t*)g->row_ptr, (const int32_t*)g->col, g->n, width,
                           w->ell) == cudaSuccess)
        return true;
    cudaGetLastError();
    cudaFree(w->ell);
    w->ell = nullptr;  // never rows that were not written: their entries are used as vertices
    return false;
}

// Rows are loaded with the candidates while they fit in L2 (126 MB): on a
// 1000^2 grid 1.69 us a level against 1.74, on the 4096^2 grid (268 MB of rows, two
// thirds of the loads for vertices visited before) 3.46 against 3.10, near
// equal at 2900^2 (134 MB: 2.21, 2.28).
static bool ell_speculate(const bfs_graph* g, int width) {
    return (int64_t)g->n * width * (int64_t)sizeof(int32_t) <= ((int64_t)128 << 20);
}

int ell_cluster_size(const bfs_graph* g, int width) {
    const bool spec = ell_speculate(g, width);
    if (width == 4) return spec ? ell_cluster<4, true>() : ell_cluster<4, false>();
    if (width == 8) return spec ? ell_cluster<8, true>() : ell_cluster<8, false>();
    return 0;
}

// The small levels of the search p describes; p.P holds the isolated
// vertices, the outputs -1 and the control block zeros.
cudaError_t ell_launch(const bfs_graph* g, Params1 p, int width, int cl, cudaStream_t st) {
    const bool spec = ell_speculate(g, width);
    p.timeout_ns = small_wait_ns(p.timeout_ns);
    cudaLaunchAttribute attr[1];
    if (width == 4) {
        p.small_ef_max = ell_max_frontier<4>(cl);
        cudaLaunchConfig_t cfg = ell_config<4>(cl, attr, st);
        return cudaLaunchKernelEx(&cfg, spec ? bfs_small_kernel<4, true> : bfs_small_kernel<4, false>, p);
    }
    p.small_ef_max = ell_max_frontier<8>(cl);
    cudaLaunchConfig_t cfg = ell_config<8>(cl, attr, st);
    return cudaLaunchKernelEx(&cfg, spec ? bfs_small_kernel<8, true> : bfs_small_kernel<8, false>, p);
}

}  // namespace bfsgb
