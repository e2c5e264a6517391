// cc.cu -- connected components: the smallest vertex id of each component.
//
// The fixed point of min-label propagation (the BFS cascade over the same
// graph tensor G with the min operator of the paper's operator table,
// Section 2, in place of ANY) gives every vertex the smallest id of its
// component.  Propagating labels an edge per iteration takes as many
// iterations as the graph is long and reads every edge in the dense ones
// (3.3 ms on RMAT-22, 135 ms and about 3,000 iterations on the relabelled
// 4096^2 grid).  The same labels come from a union-find forest over the label
// array itself, whose work does not depend on the diameter:
//   - label[v] is v's parent in a forest; a root is its own parent.  A hook
//     makes the larger of two roots point to the smaller (one CAS), so every
//     root is the smallest id of its tree and a parent is never larger than
//     its child (Shiloach and Vishkin 1982; lock-free as in ECL-CC, Jaiganesh
//     and Burtscher 2018);
//   - most edges are never read.  Rows ascend, so the first entry of each row
//     (hubs have low ids in RMAT and BA) and then the last one are hooked; a
//     sample of the labels then names the largest tree, and only vertices
//     outside it go through the rest of their rows (the subgraph sampling of
//     Afforest, Sutton, Ben-Nun and Barak 2018).  That is exact: an edge
//     between two vertices of the largest tree joins nothing, and any other
//     edge lies in the row of an end outside it, because G is symmetric.
//
// One cooperative kernel; phases are separated by the grid barrier of
// common.cuh.  What bounds it is the gathers: per vertex a row-offset pair, two
// column sectors and a few label hops, which stay in L2 (67 MB for 2^24
// vertices); 64 warps an SM (32 registers a thread) hide them.  Measured
// around the call: RMAT-22 3,283 -> 134 us, the 4096^2 grid 135-180 ms
// (2,800 to 3,400 iterations) -> 1.2 ms, ER-22 2.2 -> 0.35 ms.
#include "common.cuh"

#include <algorithm>

namespace bfsgb {

bfs_status device_error(int err, int64_t timeout_ns);  // bfs_single.cu

namespace {

constexpr int CC_T = 512;
constexpr int CC_HOPS = 32;      // parents a vertex climbs in one shortcut pass
constexpr int CC_SAMPLES = 1024; // labels looked at to find the largest tree
constexpr int CC_SLOTS = 2048;   // hash slots they are counted in
constexpr int CC_WARP_ROW = 16;  // longer rows are hooked by a whole warp
constexpr int CC_HUB = 256;      // a hub's row reaches 1 / CC_HUB of the vertices
constexpr int CC_LOOKS = 2;      // looks at the last neighbours before they are hooked, without hubs
constexpr int CC_BIG_ROW = 4096; // rows of at least this many entries by the whole grid

struct CtlCC {
    GridBarrier bar;
    unsigned open[3];   // shortcut pass k: set in open[k % 3] by a vertex that has not reached its root
    int32_t n_big;      // rows of at least CC_BIG_ROW entries outside the largest tree
    int32_t iters;      // passes over the vertices
};

struct ParamsCC {
    int32_t n;
    int64_t m;
    const int32_t* __restrict__ row_ptr;
    const int32_t* __restrict__ col;
    int32_t* label;
    CtlCC* ctl;
    int32_t* big;       // their vertices, m / CC_BIG_ROW + 1
    int32_t big_cap;
    int32_t many_trees; // no hubs: first neighbours leave many trees
    int64_t timeout_ns;
};

// Labels are read through L1 (ld.ca): the roots of large trees are read by
// every warp, and in L2 those reads queue on a few sectors (the 4096^2 grid's
// hooks of last neighbours took 2.3 ms, RMAT-22 in all 250 us instead of 110).
// A stale label is an older parent of the same vertex, and a hook is decided
// by its CAS; barriers make the labels of earlier phases visible.
//
// Root of v's tree.  Every vertex on the way is pointed past its parent: a
// plain store is safe, because only a root is ever hooked (by CAS) and a
// vertex that has a parent keeps one; whichever of two racing stores lands
// last, it names an ancestor.  Ends: each hop goes to a smaller id.
__device__ __forceinline__ int cc_find(int32_t* L, int v) {
    int prev = v;
    int p = __ldca(L + v);
    while (p != prev) {
        const int g = __ldca(L + p);
        if (g == p) break;
        __stcg(L + prev, g);
        prev = p;
        p = g;
    }
    return p;
}

// Join the trees of root a (or what became of it) and of vertex u; returns
// the joint tree's root.  A failed CAS found that the larger root has been
// hooked meanwhile and continues from its new parent, a smaller id: it ends.
__device__ __forceinline__ int cc_hook(int32_t* L, int a, int u) {
    int b = cc_find(L, u);
    while (a != b) {
        const int hi = max(a, b), lo = min(a, b);
        const int old = atomicCAS(L + hi, hi, lo);
        if (old == hi) return lo;
        a = lo;
        b = cc_find(L, old);
    }
    return a;
}

// Shortcut passes: label[v] <- v's root.  A vertex climbs at most CC_HOPS
// parents in a pass and only its own label is written, so a chain of any
// length (a path in its natural order starts as one) is cut by that factor
// at least in each pass, and after the last pass every label is a root.
// Grid-uniform; false when a barrier was given up.
__device__ bool cc_shortcut(const ParamsCC& p, unsigned& bar_target, int& pass, int& iters) {
    const long long gtid = (long long)blockIdx.x * CC_T + threadIdx.x;
    const long long gthreads = (long long)gridDim.x * CC_T;
    for (;;) {
        unsigned* open = &p.ctl->open[pass % 3];
        bool left = false;
        for (long long v = gtid; v < p.n; v += gthreads) {
            const int own = __ldca(p.label + v);
            int r = own, g = own;
            bool root = false;
#pragma unroll 1
            for (int k = 0; k < CC_HOPS; ++k) {
                g = __ldca(p.label + r);
                if (g == r) {
                    root = true;
                    break;
                }
                r = g;
            }
            if (r != own) __stcg(p.label + v, r);
            left |= !root;
        }
        if (__syncthreads_or(left) && threadIdx.x == 0) atomicOr(open, 1u);
        if (gtid == 0) p.ctl->open[(pass + 1) % 3] = 0;  // last read two barriers ago
        ++iters;
        ++pass;
        unsigned more = 0;
        __shared__ unsigned s_more;
        if (!grid_sync(&p.ctl->bar, gridDim.x, bar_target, p.timeout_ns, NoArrivalWork(),
                       [&]() { s_more = *(volatile unsigned*)open; }))
            return false;
        more = s_more;
        __syncthreads();
        if (!more) return true;
    }
}

__global__ void __launch_bounds__(CC_T, 4) cc_kernel(ParamsCC p) {
    __shared__ int s_key[CC_SLOTS];
    __shared__ int s_cnt[CC_SLOTS];
    __shared__ int s_best;
    CtlCC* ctl = p.ctl;
    int32_t* L = p.label;
    const unsigned lane = lane_id();
    const long long gtid = (long long)blockIdx.x * CC_T + threadIdx.x;
    const long long gthreads = (long long)gridDim.x * CC_T;
    unsigned bar_target = 0;
    int pass = 0, iters = 0;

    // every vertex points to its first neighbour if that is smaller
    for (long long v = gtid; v < p.n; v += gthreads) {
        const int b = __ldg(p.row_ptr + v), e = __ldg(p.row_ptr + v + 1);
        int l = (int)v;
        if (b < e) l = min(l, __ldg(p.col + b));
        __stcg(L + v, l);
    }
    if (p.m == 0) return;  // grid-uniform: every vertex is its own component
    ++iters;
    if (!grid_sync(&ctl->bar, gridDim.x, bar_target, p.timeout_ns)) return;
    if (!cc_shortcut(p, bar_target, pass, iters)) return;
    // The last neighbour of every row (a row's only entry is done if smaller).
    // Without hubs there are still many trees, and a million hooks at once keep
    // losing their CAS to one another.  A look at the edge then only lowers the
    // larger root's label to the smallest root seen beside it (one atomicMin, no
    // search; the labels are roots, and only roots' are written).  What such a
    // root was joined to before may be lost again, but every edge is hooked
    // properly afterwards, when most have one root.
    for (int look = p.many_trees ? CC_LOOKS : 0; look >= 0; --look) {
        for (long long v = gtid; v < p.n; v += gthreads) {
            const int b = __ldg(p.row_ptr + v), e = __ldg(p.row_ptr + v + 1);
            if (b == e) continue;
            const int u = __ldg(p.col + e - 1);
            if (e - b < 2 && u < (int)v) continue;
            const int x = __ldca(L + v), y = __ldca(L + u);
            if (x == y) continue;
            if (look > 0) {
                const int hi = max(x, y), lo = min(x, y);
                if (lo < __ldca(L + hi)) atomicMin(L + hi, lo);
            } else {
                cc_hook(L, cc_find(L, x), y);
            }
        }
        ++iters;
        if (look > 0) {
            if (!grid_sync(&ctl->bar, gridDim.x, bar_target, p.timeout_ns)) return;
            if (!cc_shortcut(p, bar_target, pass, iters)) return;
        }
    }
    if (!grid_sync(&ctl->bar, gridDim.x, bar_target, p.timeout_ns)) return;
    if (!cc_shortcut(p, bar_target, pass, iters)) return;

    // the label most sampled vertices carry; every CTA takes the same sample
    // (labels do not change before the next barrier) and so the same label
    for (int i = threadIdx.x; i < CC_SLOTS; i += CC_T) {
        s_key[i] = -1;
        s_cnt[i] = 0;
    }
    if (threadIdx.x == 0) s_best = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < CC_SAMPLES; i += CC_T) {
        const unsigned long long h = (unsigned long long)(unsigned)i * 2654435761ull + 12345ull;
        const int l = __ldca(L + (long long)(h % (unsigned long long)p.n));
        unsigned s = ((unsigned)l * 2654435761u) >> 21;  // 11 bits: CC_SLOTS
        for (int tries = 0; tries < CC_SLOTS; ++tries, s = (s + 1) & (CC_SLOTS - 1)) {
            const int old = atomicCAS(&s_key[s], -1, l);
            if (old == -1 || old == l) {
                atomicAdd(&s_cnt[s], 1);
                break;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < CC_SLOTS; i += CC_T) atomicMax(&s_best, s_cnt[i]);
    __syncthreads();
    const int best = s_best;
    __syncthreads();
    if (threadIdx.x == 0) s_best = INT32_MAX;
    __syncthreads();
    for (int i = threadIdx.x; i < CC_SLOTS; i += CC_T)
        if (s_key[i] >= 0 && s_cnt[i] == best) atomicMin(&s_best, s_key[i]);
    __syncthreads();
    const int giant = s_best;
    if (!grid_sync(&ctl->bar, gridDim.x, bar_target, p.timeout_ns)) return;

    // the rows, but for their last entries, of every vertex outside that tree
    // (the first entry has been hooked only if it was smaller): short rows by
    // their lane, longer ones by the warp, the longest listed for the grid
    for (long long v0 = gtid - lane; v0 < p.n; v0 += gthreads) {  // warp-uniform
        const long long v = v0 + lane;
        int b = 0, e = 0;
        if (v < p.n && __ldca(L + v) != giant) {
            b = __ldg(p.row_ptr + v);
            e = __ldg(p.row_ptr + v + 1) - 1;
        }
        const int len = e - b;
        if (len >= CC_BIG_ROW - 1) {
            const int at = atomicAdd(&ctl->n_big, 1);
            if (at < p.big_cap) p.big[at] = (int)v;
            else atomicCAS(&ctl->bar.err, 0, (int)DEV_OVERFLOW);  // cannot happen: rows sum to m
        } else if (len > 0 && len <= CC_WARP_ROW) {
            int a = cc_find(L, (int)v);
            for (int j = b; j < e; ++j) {
                const int u = __ldg(p.col + j);
                if (__ldca(L + u) != a) a = cc_hook(L, a, u);
            }
        }
        unsigned wm = __ballot_sync(0xffffffffu, len > CC_WARP_ROW && len < CC_BIG_ROW - 1);
        while (wm) {
            const int l = __ffs(wm) - 1;
            wm &= wm - 1;
            const int bl = __shfl_sync(0xffffffffu, b, l), el = __shfl_sync(0xffffffffu, e, l);
            int a = cc_find(L, (int)(v0 + l));
            for (int j = bl + (int)lane; j < el; j += 32) {
                const int u = __ldg(p.col + j);
                if (__ldca(L + u) != a) a = cc_hook(L, a, u);
            }
            __syncwarp();
        }
    }
    ++iters;
    if (!grid_sync(&ctl->bar, gridDim.x, bar_target, p.timeout_ns)) return;
    const int nb = min(*(volatile int*)&ctl->n_big, p.big_cap);
    for (int i = 0; i < nb; ++i) {
        const int v = __ldca(p.big + i);
        const int b = __ldg(p.row_ptr + v), e = __ldg(p.row_ptr + v + 1) - 1;
        if (b + gtid < e) {
            int a = cc_find(L, v);
            for (long long j = b + gtid; j < e; j += gthreads) {
                const int u = __ldg(p.col + j);
                if (__ldca(L + u) != a) a = cc_hook(L, a, u);
            }
        }
    }
    if (nb > 0 && !grid_sync(&ctl->bar, gridDim.x, bar_target, p.timeout_ns)) return;  // grid-uniform
    if (!cc_shortcut(p, bar_target, pass, iters)) return;
    if (gtid == 0) ctl->iters = iters;
}

}  // namespace

}  // namespace bfsgb

using namespace bfsgb;

extern "C" bfs_status bfs_components(const bfs_graph* gc, int32_t* label, int32_t* iterations, void* cuda_stream) {
    bfs_graph* g = const_cast<bfs_graph*>(gc);
    if (!g || !label) return fail(BFS_EINVAL, "null argument");
    if (!g->symmetric) return fail(BFS_EINVAL, "bfs_components needs a symmetric graph (BFS_SYMMETRIZE)");
    if (device_id() != g->device) return fail(BFS_EINVAL, "graph lives on device %d, current device is %d", g->device, device_id());
    std::lock_guard<std::mutex> guard(g->lock);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int32_t n = g->n;
    const bool host = !is_device_ptr(label);

    // control block and list of long rows, kept with the graph: the call
    // waits for its kernel under the graph's lock, so no two calls share it
    // in time (an allocation from the stream-ordered pool here cost a call
    // about as long as the kernel, since the pool gives memory back at every
    // synchronisation)
    const int32_t big_cap = g->deg_max >= CC_BIG_ROW ? (int32_t)(g->m / CC_BIG_ROW) + 1 : 0;
    if (!g->cc_scratch &&
        cudaMalloc(&g->cc_scratch, sizeof(CtlCC) + sizeof(int32_t) * (size_t)std::max(big_cap, 1)) != cudaSuccess) {
        cudaGetLastError();
        g->cc_scratch = nullptr;
        return fail(BFS_ENOMEM, "components scratch");
    }
    int32_t* d_label = label;
    if (host && cudaMallocAsync(&d_label, (size_t)n * sizeof(int32_t), st) != cudaSuccess) {
        cudaGetLastError();
        return fail(BFS_ENOMEM, "components workspace for n=%d", n);
    }
    ParamsCC p{};
    p.n = n;
    p.m = g->m;
    p.row_ptr = g->row_ptr;
    p.col = g->col;
    p.label = d_label;
    p.ctl = (CtlCC*)g->cc_scratch;
    p.big = (int32_t*)(p.ctl + 1);
    p.big_cap = big_cap;
    // A matter of time alone; us around the call with 0 / 1 / 2 / 3 looks:
    // RMAT-22 134 / 171 / 211 / 252 (a hub), with a = 0.45 and edge factor 8 300 /
    // 199 / 246 / 283 (none); ER-22 607 / 803 / 348 / 407, 2^17 vertices of degree
    // 8 195 / 328 / 76 / 83; grids 4096^2 1085 / 1083 / 1156 / 1217, 1000^2 583 /
    // 318 / 233 / 424.
    p.many_trees = (int64_t)g->deg_max * CC_HUB < n;
    p.timeout_ns = 2000000000ll;
    int per_sm = 0;
    CtlCC h{};
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cc_kernel, CC_T, 0);
    if (e == cudaSuccess) e = cudaMemsetAsync(p.ctl, 0, sizeof(CtlCC), st);
    if (e == cudaSuccess) {
        // no more CTAs than vertices to give a thread each: a small graph's
        // barriers then count fewer arrivals
        const int64_t want = std::max<int64_t>(1, div_up(n, CC_T));
        const int blocks = (int)std::min<int64_t>(want, (int64_t)std::max(per_sm, 1) * num_sms());
        void* args[] = {(void*)&p};
        e = cudaLaunchCooperativeKernel((const void*)cc_kernel, dim3(blocks), dim3(CC_T), args, 0, st);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, p.ctl, sizeof(CtlCC), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && host) e = cudaMemcpyAsync(label, d_label, (size_t)n * 4, cudaMemcpyDeviceToHost, st);
    if (host) cudaFreeAsync(d_label, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "components");
    if (h.bar.err) return device_error(h.bar.err, p.timeout_ns);
    if (iterations) *iterations = h.iters;
    return BFS_OK;
}
