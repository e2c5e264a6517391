// msbfs.cu -- batched multi-source BFS: up to 64 sources per unit, each
// vertex carrying 64-bit frontier / seen masks (one bit per source lane).
//
// Per lane j this is exactly Cascade 1 for source j; the 64 lanes share every
// read of G.  With seen_i the lanes that reached v before level i and front_i
// the lanes whose frontier holds v:
//   push: for u with front_i[u] != 0, for v in N(u):
//           bits = front_i[u] & ~seen[v]; next[v] |= bits; new = bits & ~(seen[v] |= bits)
//   pull: for v with missing = ~seen[v] != 0, OR front_i[u] over in-neighbours
//           u in ascending order, stopping once every missing lane is found
//   then front_{i+1} = next and seen |= next: the three-array identity
//   F_{i+1} = P_{i+1} AND NOT P_i of the paper's variant 26.
// The ANY reduction picks, per lane, the first u (push: the one whose OR set
// the bit; pull: the lowest-index in-neighbour), which is written as parent.
// A push claims in `seen` itself: a lane is then found once whatever buffer
// F_{i+1} is in, and a level ends with one grid barrier.  (Claiming in next[]
// and folding it into seen afterwards took a second barrier and a pass over
// the new frontier a level.)
//
// One cooperative kernel runs all levels of all units of a launch: units are
// independent searches (possibly over different graphs: bfs_run_mixed), and
// levels are separated by a grid barrier with a %globaltimer limit.
#include "common.cuh"
#include "policy_dev.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <vector>

namespace bfsgb {

struct MsUnit {
    const int32_t* row_ptr;
    const int32_t* col;
    const int32_t* csc_ptr;
    const int32_t* csc_col;
    const uint32_t* isolated;
    int64_t m;
    int32_t n;
    int32_t k;
    int32_t symmetric;
    int32_t deg_max;
    int32_t src[64];
    int32_t* depth[64];
    int32_t* parent[64];
};

struct CountersMS {
    unsigned long long a_len;  // active vertices appended (front != 0)
    unsigned long long u_len;  // chunk units appended
    unsigned long long e_f;    // degree sum of the appended vertices
    unsigned long long conv;   // cursor of a masks -> active-list conversion
    unsigned long long lanes;  // OR of the frontier masks: lanes that can still find vertices
    unsigned long long done_e; // degree sum of the vertices that the level left seen by every live lane
    unsigned long long pull_next;  // pull level: cursor of the warps over the words of the vertex range
    unsigned long long long_len;   // deferred long rows of the (pull) level this slot is current in
};

struct CtlMS {
    GridBarrier bar;
    CountersMS slot[3];
    int32_t levels;
};

struct WorkspaceMS {
    int32_t ncap = 0;
    int64_t ucap = 0;
    int32_t chunk = 0;
    uint64_t* seen = nullptr;
    uint64_t* front[2] = {nullptr, nullptr};
    int4* act[2] = {nullptr, nullptr};
    int2* U[2] = {nullptr, nullptr};
    CtlMS* ctl = nullptr;
    int* d_sticky = nullptr;
    MsUnit* d_units = nullptr;
    int32_t units_cap = 0;
    CtlMS* h_ctl = nullptr;
    int32_t* longv = nullptr;            // pull: deferred long rows of the level
    unsigned long long* acc_long = nullptr;  // their lanes found so far
    uint64_t* hist = nullptr;            // frontier masks of levels 0 .. MS_HIST-1, [MS_HIST][ncap]
    int* hist_dirty = nullptr;           // device flag, see ParamsMS
    uint32_t* full = nullptr;            // see ParamsMS
};

void free_wsms(WorkspaceMS* w) {
    if (!w) return;
    cudaFree(w->seen);
    for (int i = 0; i < 2; ++i) {
        cudaFree(w->front[i]);
        cudaFree(w->act[i]);
        cudaFree(w->U[i]);
    }
    cudaFree(w->ctl);
    cudaFree(w->d_sticky);
    cudaFree(w->d_units);
    cudaFree(w->longv);
    cudaFree(w->acc_long);
    cudaFree(w->hist);
    cudaFree(w->hist_dirty);
    cudaFree(w->full);
    cudaFreeHost(w->h_ctl);
    delete w;
}

int msbfs_sticky_error(bfs_graph* g) {
    if (!g || !g->wsms) return 0;
    int err = 0;
    if (cudaMemcpy(&err, g->wsms->d_sticky, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return DEV_OK;
    if (err) cudaMemset(g->wsms->d_sticky, 0, 4);
    return err;
}

bfs_status device_error(int err, int64_t timeout_ns);
const float* policy_device_weights(const bfs_policy* p);

struct ParamsMS {
    const MsUnit* units;
    int32_t n_units;
    uint64_t* seen;
    uint64_t* F0;
    uint64_t* F1;
    int4* A0;  // active lists: vertex, row begin, row end, 0
    int4* A1;
    int2* U0;
    int2* U1;
    int64_t ucap;
    CtlMS* ctl;
    int* sticky;
    int32_t policy;
    float alpha, beta;
    const int8_t* schedule;
    int32_t schedule_len;
    const float* mlp;
    int32_t chunk, medium, pull_serial;
    int64_t timeout_ns;
    int32_t max_levels;
    bfs_level_record* log;  // per-level records of the first unit
    int32_t log_cap;
    int32_t* longv;
    unsigned long long* acc_long;
    uint64_t* hist;  // frontier masks of the first MS_HIST levels (zero between units)
    int64_t ncap;    // vertices per history level
    int* hist_dirty; // set while a launch runs; still set at the next launch if it ended early
    uint32_t* full;  // bit v: v has no in-edge, or every lane has seen it (bits past n are set): no pull scans it
};

// Unit fields kept in registers / shared memory while a unit runs.
struct UnitView {
    const int32_t* __restrict__ row_ptr;
    const int32_t* __restrict__ col;
    const int32_t* __restrict__ csc_ptr;
    const int32_t* __restrict__ csc_col;
    const uint32_t* __restrict__ isolated;
    int64_t m;
    int32_t n;
    int32_t k;
    int32_t symmetric;
    int32_t deg_max;
    uint64_t lanes;
};

constexpr int MS_T = 512;
// Depths of the first MS_HIST levels are not written as lanes find vertices:
// the frontier masks of those levels are kept, and one pass after the last
// level writes every depth row whole (the level of the first mask holding
// the lane, -1 for an unreached vertex).  Written as found, a lane's depth
// entries are scattered 4-byte stores into partly written sectors, which the
// memory system fills from DRAM, and every row would first be set to -1.
constexpr int MS_HIST = 16;
// Per-warp staging of active-list appends (RMAT-24 x 64, ms, at 64 / 128 / 256 entries: 8.19 / 8.10 / 8.08)
constexpr int MS_QBUF = 128;
// Pull rows longer than this are scanned by CTAs after the warps' pass.  A
// warp stops within a few hundred entries of a hub's row on a dense level, a CTA
// takes at least 512 and two barriers; but a warp's long scans are the level's
// tail where every warp has only a word or two.  So the line is low for graphs
// of at most MS_FEW_WORDS words a warp and high above.  64-lane batches with
// parents, us, at 512 / 1024 / 2048 / 4096 / 16384: RMAT-16 216 / 246 / 332 / 330 /
// 444, RMAT-18 456 / 464 / 545 / 555 / 1137, RMAT-19 437 / 380 / 378 / 358 / 356,
// RMAT-22 2319 / 1958 / 1894 / 1716 / 1679, renumbered without parents 2165 /
// 1804 / 1740 / 1655 / 1986, RMAT-24 14850 / 11420 / 11440 / 10100 / 9760; 8192: 1725,
// 1659 and 9820 for the last three.
constexpr int MS_LONG_ROW_SMALL = 512, MS_LONG_ROW = 8192, MS_FEW_WORDS = 2;
static_assert(MS_LONG_ROW < 65536, "pull parent positions are staged as 16-bit row offsets");
// Row entries a warp scans together in the 32 rows of a word before it leaves
// what is left of them to CTAs.  Lanes that none of a word of hubs can find yet
// (renumbered graphs have such words) would otherwise keep one warp for
// milliseconds: RMAT-19 renumbered, 5 lanes, one seed 1258 us without a limit,
// 412 / 443 / 499 at 16384 / 24576 / 32768; RMAT-22 renumbered x 64 2227 us against
// 1641 / 1674 / 1714; RMAT-24 x 64 8.08 ms against 8.28 / 8.14 / 8.11.  (1024 entries a
// row: 514 us, 1719 us, 8.30 ms.)
constexpr int MS_WARP_ENTRIES = 24576;
constexpr int MS_LONG_ITEMS = 1;  // entries a thread tests per long-row chunk (RMAT-24: 10.08 ms, four 10.14)

#ifndef BFS_MS_PULL_R
#define BFS_MS_PULL_R 4
#endif
constexpr int MS_PULL_R = BFS_MS_PULL_R;  // in-neighbours loaded per serial pull step
constexpr int MS_COOP_U = 4;  // 32-entry groups a warp loads per step when it finishes a long row

// Words a warp takes at a time in a pull level: one while many vertices
// still miss live lanes (costly words: finest balance).  Once few do, up to
// 32, so that the takes don't queue on the cursor's atomics and most words are
// passed over by their bits in `full`, but at least MS_PULL_TAKES takes a
// warp: the words that are left may cost hundreds of microseconds each (with
// 32 words a take on 2^14 vertices, 16 warps had them all: 97 -> 320 us).
constexpr int MS_PULL_CHUNK = 32, MS_PULL_TAKES = 4;

// A level's constants.  These and the unit's live in shared memory: at 64
// registers a thread (two CTAs an SM) they were spilled, and those spills were 170
// million memory requests of an RMAT-22 batch.  (140 bytes of other state are
// still spilled, 148 without parents.)
struct MsLevelConst {
    int32_t level;
    int pull_chunk;              // pull: words a warp takes at a time
    int long_row;                // pull: rows longer than this are left to ms_long_rows
    uint64_t* f_next;
    int4* a_next;
    int2* u_next;
    CountersMS* next;
    uint64_t live;               // lanes with a non-empty frontier F_i
    unsigned long long* cursor;  // pull: next word to take (zero when the level starts)
    unsigned long long* long_len;  // pull: deferred long rows (zero when the level starts)
    bool sparse;                 // pull: few vertices miss live lanes
    bool whole;                  // pull: the unit's first; it writes every parent entry not written before
    bool write_depth;            // depths of F_{i+1} are written now (levels past the history)
    bool clear_cur;              // push: F_i's masks are zeroed as they are read (levels past the history)
};

struct MsSmem {
    UnitView g;
    MsLevelConst lv;
    int32_t* depth[64];
    int32_t* parent[64];
    int off[MS_T + 1];
    int beg[MS_T];
    int lim[MS_T];
    int src[MS_T];
    unsigned long long fmask[MS_T];
    int scan_tmp[33];
    float feat[BFS_MLP_IN];
    float mlp_out;
    unsigned long long red[4][MS_T / 32];  // a level's e_f, |F|, done_e and lanes, one share a warp
    unsigned long long base;
    int qlen[MS_T / 32];
    unsigned long long cnt[6];             // counters of the level about to start, read as the barrier opens
};

// What a thread gathers in a level.  Degree sums fit in 32 bits: a vertex is
// counted once, and a CSR has less than 2^31 entries.
struct MsLevel {
    const MsLevelConst& c;
    unsigned ef;             // degree sum of F_{i+1} vertices (this thread's share)
    unsigned cnt;            // |{v : F_{i+1}[v] != 0}| (pull levels, this thread's share)
    unsigned done_e;         // degree sum of vertices now seen by every live lane (this thread's share)
    uint64_t lanes;          // OR of the F_{i+1} masks this thread wrote
    int qn;                  // staged appends (warp-uniform)
};

// Dynamic shared memory of the MS-BFS kernel: per warp, the row offset of
// the parent found for each (vertex of the warp's word, lane l) in a pull
// level, [vertex][l], so that parents are written lane-major like depths.
// Rows are 66 entries apart: reading one l of 32 vertices, and writing 32 l of
// one vertex, both hit 32 banks.
constexpr int MS_PIDX_LD = 66;
constexpr size_t MS_PIDX_BYTES = (size_t)(MS_T / 32) * 32 * MS_PIDX_LD * sizeof(unsigned short);
extern __shared__ __align__(16) unsigned short ms_pidx_smem[];
// A push level stages a warp's active-list appends in the same bytes (MS_QBUF
// vertices, row begins and row ends), all there is without parents.  What
// the CTAs do not take is L1, which dense pulls gather masks through: with the
// staging in bytes of its own (196 KB of shared memory an SM, not 164) RMAT-24
// took 8.86 ms with parents against 8.10.
constexpr size_t MS_QBUF_BYTES = (size_t)(MS_T / 32) * 3 * MS_QBUF * sizeof(int32_t);
static_assert(MS_QBUF_BYTES <= MS_PIDX_BYTES, "staging fits the parent offsets' bytes");
__device__ __forceinline__ int32_t* ms_qbuf() { return (int32_t*)ms_pidx_smem + (threadIdx.x >> 5) * 3 * MS_QBUF; }

__device__ __forceinline__ void write_lanes(MsSmem& sm, uint64_t bits, int v, int par, int d, bool write_depth) {
    while (bits) {
        int j = __ffsll((long long)bits) - 1;
        if (write_depth) sm.depth[j][v] = d;
        if (sm.parent[j]) sm.parent[j][v] = par;
        bits &= bits - 1;
    }
}

__device__ __forceinline__ void ms_units(const ParamsMS& p, int2* u_out, CountersMS* c, int v, int deg) {
    append_units(u_out, &c->u_len, p.ucap, &p.ctl->bar.err, v, deg, p.chunk);
}

__device__ __forceinline__ void ms_flush(MsLevel& L, MsSmem& sm) {
    const int32_t* qbuf = ms_qbuf();
    if (L.qn == 0) return;
    unsigned lane = lane_id();
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&L.c.next->a_len, (unsigned long long)L.qn);
    base = __shfl_sync(0xffffffffu, base, 0);
    __syncwarp();
    for (int i = (int)lane; i < L.qn; i += 32) L.c.a_next[base + i] = make_int4(qbuf[i], qbuf[MS_QBUF + i], qbuf[2 * MS_QBUF + i], 0);
    __syncwarp();
    L.qn = 0;
}

// v entered F_{i+1} (first OR into its mask this level): stage it and its row
// bounds for the active list, add its degree, split big rows into chunk units.  Warp-uniform.
__device__ __forceinline__ void ms_emit(const ParamsMS& p, MsLevel& L, MsSmem& sm, bool first, int v, int rb,
                                        int re) {
    unsigned cm = __ballot_sync(0xffffffffu, first);
    if (!cm) return;
    int c = __popc(cm);
    if (L.qn + c > MS_QBUF) ms_flush(L, sm);
    if (first) {
        const int deg = re - rb;
        int32_t* slot = ms_qbuf() + L.qn + __popc(cm & lanemask_lt());
        slot[0] = v;
        slot[MS_QBUF] = rb;
        slot[2 * MS_QBUF] = re;
        L.ef += (unsigned)deg;
        if (deg >= p.chunk) ms_units(p, L.c.u_next, L.c.next, v, deg);
    }
    L.qn += c;
}

// Push candidate u -> v with frontier lanes fu: the lanes of fu that v has not
// seen are ORed into seen[v], whose old value names exactly one claimer per
// (v, lane), which writes the lane's parent (and depth), and into F_{i+1}[v].
// The read of seen[v] is no older than the level (the barrier before it), so a
// lane in it that another thread claims first is claimed in this level and
// belongs in F_{i+1}[v] all the same: both ORs, and the row bounds of v, are in
// flight together.  Returns true for the first entry into F_{i+1}[v] (some
// lane of it may be another thread's), with v's row bounds in rb, re.
template <bool PAR>
__device__ __forceinline__ bool ms_claim(const ParamsMS& p, const UnitView& g, MsLevel& L, MsSmem& sm, bool has, int v,
                                         int u, uint64_t fu, int& rb, int& re) {
    uint64_t bits = 0;
    // an ordinary load: hubs are read by thousands of threads, which the L1 then
    // serves; lanes only grow, so a stale word costs an OR at most
    if (has) bits = fu & ~((const unsigned long long*)p.seen)[v];
    if (!bits) return false;
    const uint64_t old = atomicOr((unsigned long long*)p.seen + v, (unsigned long long)bits);
    const uint64_t in = atomicOr((unsigned long long*)L.c.f_next + v, (unsigned long long)bits);
    rb = __ldg(g.row_ptr + v);
    re = __ldg(g.row_ptr + v + 1);
    const uint64_t nb = bits & ~old, now = old | bits;
    if (nb) {
        L.lanes |= nb;
        if (PAR || L.c.write_depth) write_lanes(sm, nb, v, u, L.c.level + 1, L.c.write_depth);
        if ((now & L.c.live) == L.c.live && (old & L.c.live) != L.c.live) L.done_e += (unsigned)(re - rb);
        if (now == g.lanes) atomicOr(p.full + (v >> 5), 1u << (v & 31));
    }
    return in == 0;
}

template <bool PAR>
__device__ __forceinline__ void ms_candidate(const ParamsMS& p, const UnitView& g, MsLevel& L, MsSmem& sm, bool has,
                                             int v, int u, uint64_t fu) {
    int rb = 0, re = 0;
    const bool first = ms_claim<PAR>(p, g, L, sm, has, v, u, fu, rb, re);
    ms_emit(p, L, sm, first, v, rb, re);
}

// End of a push level: the warps' staged appends, with one atomic for the CTA
// (one a warp queued thousands of them on the counter's sector).  Block-uniform.
template <int T>
__device__ void ms_flush_all(MsLevel& L, MsSmem& sm) {
    const int warp = (int)(threadIdx.x >> 5), lane = (int)lane_id();
    if (lane == 0) sm.qlen[warp] = L.qn;
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < T / 32; ++w) {
        const int x = sm.qlen[w];
        before += w < warp ? x : 0;
        total += x;
    }
    if (total == 0) return;
    if (threadIdx.x == 0) sm.base = atomicAdd(&L.c.next->a_len, (unsigned long long)total);
    __syncthreads();
    const int32_t* qbuf = ms_qbuf();
    for (int i = lane; i < L.qn; i += 32)
        L.c.a_next[sm.base + before + i] = make_int4(qbuf[i], qbuf[MS_QBUF + i], qbuf[2 * MS_QBUF + i], 0);
    L.qn = 0;
}

// A tile of the active list, one entry a thread (vertex < 0: none).  An entry
// carries its row's bounds, and a candidate loads its source's mask beside its
// column, so between the entry and the first ORs there are two round trips
// (the 2048 x 1531 grid with 32 lanes 44.4 -> 41.6 ms).
template <int T, bool PAR>
__device__ void ms_push_tile(const ParamsMS& p, const UnitView& g, MsLevel& L, MsSmem& sm, int4 e, uint64_t* f_cur) {
    static_assert(T <= MS_T, "tile arrays are sized for MS_T threads");
    unsigned lane = lane_id();
    const unsigned long long* F = (const unsigned long long*)f_cur;
    const int u = e.x, beg = e.y;
    int end = e.z;
    const bool unit = end - beg >= p.chunk;
    if (unit) end = beg;  // chunk units cover it
    // medium rows: 32-edge segments taken in turn by every warp of the CTA
    if (g.deg_max >= p.medium) {
        const bool med = (end - beg) >= p.medium;
        int nseg_total;
        const int soff = block_exclusive_scan(med ? (end - beg + 31) >> 5 : 0, sm.scan_tmp, &nseg_total);
        if (nseg_total > 0) {
            sm.off[threadIdx.x] = soff;
            sm.beg[threadIdx.x] = beg;
            sm.lim[threadIdx.x] = end;
            sm.src[threadIdx.x] = u;
            __syncthreads();
            for (int s = (int)(threadIdx.x >> 5); s < nseg_total; s += T / 32) {
                int lo = 0, hi = T - 1;
                while (lo < hi) {
                    int mid = (lo + hi + 1) >> 1;
                    if (sm.off[mid] <= s) lo = mid; else hi = mid - 1;
                }
                const int j = sm.beg[lo] + ((s - sm.off[lo]) << 5) + (int)lane;
                const bool has = j < sm.lim[lo];
                const int v = has ? __ldg(g.col + j) : 0;
                ms_candidate<PAR>(p, g, L, sm, has, v, sm.src[lo], F[sm.src[lo]]);
            }
        }
        if (med) end = beg;
    }
    int total;
    int off = block_exclusive_scan(end - beg, sm.scan_tmp, &total);
    sm.off[threadIdx.x] = off;
    sm.beg[threadIdx.x] = beg;
    sm.src[threadIdx.x] = u;
    if (threadIdx.x == T - 1) sm.off[T] = total;
    __syncthreads();
    for (int k0 = 0; k0 < total; k0 += T) {
        int k = k0 + threadIdx.x;
        bool has = k < total;
        int v = 0, su = 0;
        uint64_t sf = 0;
        if (has) {
            int lo = 0, hi = T - 1;
            while (lo < hi) {
                int mid = (lo + hi + 1) >> 1;
                if (sm.off[mid] <= k) lo = mid; else hi = mid - 1;
            }
            su = sm.src[lo];
            v = __ldg(g.col + sm.beg[lo] + (k - sm.off[lo]));
            sf = F[su];
        }
        ms_candidate<PAR>(p, g, L, sm, has, v, su, sf);
    }
    __syncthreads();
    // the mask has been read, by this tile alone
    if (L.c.clear_cur && u >= 0 && !unit) f_cur[u] = 0;
}

// Push level: items = chunk units of big rows, then CTA tiles of the active
// list, dealt round-robin over the CTAs.
template <int T, bool PAR>
__device__ void ms_push_level(const ParamsMS& p, const UnitView& g, MsLevel& L, MsSmem& sm, const int4* a_cur,
                              const int2* u_cur, uint64_t* f_cur, long long a, long long nunits) {
    long long per_tile = (a + gridDim.x - 1) / gridDim.x;
    per_tile = per_tile < 1 ? 1 : (per_tile > T ? T : per_tile);
    long long nitems = nunits + (a + per_tile - 1) / per_tile;
    for (long long it = blockIdx.x; it < nitems; it += gridDim.x) {
        if (it < nunits) {
            int2 un = u_cur[it];
            int u = un.x;
            uint64_t fu = ((const unsigned long long*)f_cur)[u];
            int b = __ldg(g.row_ptr + u), e = __ldg(g.row_ptr + u + 1);
            int lo = b + un.y * p.chunk, hi = min(e, lo + p.chunk);
            for (int base = lo; base < hi; base += T) {
                int j = base + threadIdx.x;
                bool has = j < hi;
                int v = has ? __ldg(g.col + j) : 0;
                ms_candidate<PAR>(p, g, L, sm, has, v, u, fu);
            }
        } else {
            long long q = (it - nunits) * per_tile + threadIdx.x;
            const int4 e = (threadIdx.x < per_tile && q < a) ? a_cur[q] : make_int4(-1, 0, 0, 0);
            ms_push_tile<T, PAR>(p, g, L, sm, e, f_cur);
        }
    }
    ms_flush_all<T>(L, sm);
}

__device__ __forceinline__ uint64_t warp_or64(uint64_t x) {
    unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)x);
    unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(x >> 32));
    return ((uint64_t)hi << 32) | lo;
}

// Pull level, one warp per 32 consecutive vertices (lane = vertex): a vertex
// missing some live lanes (lanes whose frontier F_i is not empty: only those
// can reach it at this level) ORs the frontier masks of its in-neighbours in
// ascending order and stops once every such lane is found; the first
// neighbour that supplies a lane is that lane's parent.  Rows longer than
// `pull_serial` entries are finished by the whole warp.  Depths are written
// lane-major in a warp-uniform loop over the union of the new lanes, so the
// 32 vertices' entries of one lane's depth row go out together.

// Leaves the rows of the lanes in `rows`, from entry `from` on, to ms_long_rows.
// Warp-uniform.
__device__ __forceinline__ void ms_defer(const ParamsMS& p, const MsLevel& L, unsigned rows, int v,
                                         int from) {
    const unsigned lane = lane_id();
    const int leader = __ffs(rows) - 1;
    unsigned long long base = 0;
    if ((int)lane == leader) base = atomicAdd(L.c.long_len, (unsigned long long)__popc(rows));
    base = __shfl_sync(0xffffffffu, base, leader);
    if ((rows >> lane) & 1u) {
        const unsigned long long r = base + __popc(rows & lanemask_lt());
        p.longv[r] = v;
        p.acc_long[r] = (unsigned long long)from;  // until the CTA stores what it found
    }
}

template <bool PAR>
__device__ void ms_pull_level(const ParamsMS& p, const UnitView& g, MsLevel& L, MsSmem& sm, const uint64_t* f_cur) {
    const unsigned lane = lane_id();
    unsigned short* pidx = ms_pidx_smem + (threadIdx.x >> 5) * (32 * MS_PIDX_LD);
    const int W = (g.n + 31) >> 5;
    const unsigned long long* F = (const unsigned long long*)f_cur;
    // this thread's counters in the push tiles' arrays, not in registers
    const int me = (int)threadIdx.x;
    sm.beg[me] = sm.lim[me] = sm.src[me] = 0;  // degree sum, vertices, degree sum of the finished
    sm.fmask[me] = 0;                          // lanes
    // warps take pull_chunk words at a time from a level-wide cursor: the
    // cost of a word varies by orders of magnitude (hubs, early exits), and a
    // fixed deal left most warps waiting at the level barrier.  The next take
    // is requested when a chunk starts, so its round trip overlaps the work.
    unsigned take = 0;  // W < 2^26, and each warp passes it by one take at most
    if (lane == 0) take = (unsigned)atomicAdd(L.c.cursor, (unsigned long long)L.c.pull_chunk);
    for (;;) {  // warp-uniform
        const int w0 = (int)__shfl_sync(0xffffffffu, take, 0);
        if (w0 >= W) break;
        if (lane == 0) take = (unsigned)atomicAdd(L.c.cursor, (unsigned long long)L.c.pull_chunk);
        // the vertices that need no look: the chunk's words of `full`, one a
        // lane (chunk <= 32), where few are open; on a dense level, whose
        // words nearly all have work, the constant bitmap
        const bool mine = (int)lane < min(L.c.pull_chunk, W - w0);
        const bool whole = PAR && L.c.whole;  // every word
        const unsigned fl = !mine ? 0xffffffffu : whole ? 0u : L.c.sparse ? __ldcg(p.full + w0 + lane) : __ldg(g.isolated + w0 + lane);
        for (unsigned todo = __ballot_sync(0xffffffffu, fl != 0xffffffffu); todo; todo &= todo - 1) {  // warp-uniform
        const int v = (w0 + __ffs(todo) - 1) * 32 + (int)lane;
        uint64_t miss = 0;
        if (!((__shfl_sync(0xffffffffu, fl, __ffs(todo) - 1) >> lane) & 1u) && v < g.n)
            miss = L.c.live & ~((const unsigned long long*)p.seen)[v];
        if (!whole && !__ballot_sync(0xffffffffu, miss != 0)) continue;
        int beg = 0, end = 0;
        if (miss) {
            beg = __ldg(g.csc_ptr + v);
            end = __ldg(g.csc_ptr + v + 1);
        }
        // rows longer than long_row are scanned by the whole grid after
        // this pass (ms_long_rows); defer them
        const bool longrow = miss != 0 && end - beg > L.c.long_row;
        const unsigned lm = __ballot_sync(0xffffffffu, longrow);
        if (lm) {
            ms_defer(p, L, lm, v, beg);
            if (longrow) {
                miss = 0;
                end = beg;
            }
        }
        uint64_t acc = 0;
        int j = beg;
        const int lim = min(end, beg + p.pull_serial);
        // MS_PULL_R entries per step (independent loads), taken in row order;
        // once every missing lane is found the rest of a step adds nothing
        while (j < lim && acc != miss) {
            int uu[MS_PULL_R];
            uint64_t fm[MS_PULL_R];
#pragma unroll
            for (int r = 0; r < MS_PULL_R; ++r) uu[r] = j + r < lim ? __ldg(g.csc_col + j + r) : -1;
#pragma unroll
            for (int r = 0; r < MS_PULL_R; ++r) fm[r] = uu[r] >= 0 ? F[uu[r]] & miss : 0ull;
            if (PAR) {
                unsigned short* mine = pidx + lane * MS_PIDX_LD;
#pragma unroll
                for (int r = 0; r < MS_PULL_R; ++r) {
                    const uint64_t got = fm[r] & ~acc;
                    acc |= got;
                    // (the halves apart: 32-bit bit scans)
                    for (unsigned b = (unsigned)got; b; b &= b - 1) mine[__ffs(b) - 1] = (unsigned short)(j + r - beg);
                    for (unsigned b = (unsigned)(got >> 32); b; b &= b - 1)
                        mine[__ffs(b) + 31] = (unsigned short)(j + r - beg);
                }
            } else {
#pragma unroll
                for (int r = 0; r < MS_PULL_R; ++r) acc |= fm[r];
            }
            j = min(j + MS_PULL_R, lim);  // the warp goes on from here
        }
        unsigned rm = __ballot_sync(0xffffffffu, miss != 0 && acc != miss && j < end);
        unsigned rest = 0;           // rows the warp gives up
        int left = MS_WARP_ENTRIES;  // entries it scans in the word's rows
        while (rm) {
            const int l = __ffs(rm) - 1;
            const int jl = __shfl_sync(0xffffffffu, j, l);
            const int el = __shfl_sync(0xffffffffu, end, l);
            const int bl = __shfl_sync(0xffffffffu, beg, l);
            const uint64_t ml = __shfl_sync(0xffffffffu, (unsigned long long)miss, l);
            uint64_t al = __shfl_sync(0xffffffffu, (unsigned long long)acc, l);
            // MS_COOP_U * 32 entries a step: all column loads, then all mask loads
            int b2 = jl;
            for (; b2 < el && left > 0 && al != ml; b2 += 32 * MS_COOP_U, left -= 32 * MS_COOP_U) {
                int uu[MS_COOP_U];
                uint64_t fu[MS_COOP_U];
#pragma unroll
                for (int q = 0; q < MS_COOP_U; ++q) {
                    const int idx = b2 + q * 32 + (int)lane;
                    uu[q] = idx < el ? __ldg(g.csc_col + idx) : -1;
                }
#pragma unroll
                for (int q = 0; q < MS_COOP_U; ++q) fu[q] = uu[q] >= 0 ? (F[uu[q]] & ml & ~al) : 0ull;
                uint64_t got = 0;
                if (PAR) {
                    // the entries that supply something new, in entry order;
                    // thread b records lanes b and b + 32 of each.  A row has
                    // at most 64 of them and mostly a few: 20 instructions
                    // each, where an OR scan over the 32 entries of every
                    // group took 75 and a ballot per lane 16
#pragma unroll
                    for (int q = 0; q < MS_COOP_U; ++q) {
                        uint64_t x = fu[q] & ~got;
                        for (unsigned m = __ballot_sync(0xffffffffu, x != 0); m; m = __ballot_sync(0xffffffffu, x != 0)) {
                            const int s = __ffs(m) - 1;
                            const uint64_t xs = __shfl_sync(0xffffffffu, (unsigned long long)x, s);
                            const unsigned short at = (unsigned short)(b2 + q * 32 + s - bl);
                            if (((unsigned)xs >> lane) & 1u) pidx[l * MS_PIDX_LD + lane] = at;
                            if (((unsigned)(xs >> 32) >> lane) & 1u) pidx[l * MS_PIDX_LD + 32 + lane] = at;
                            got |= xs;
                            x &= ~xs;
                        }
                    }
                } else {
                    uint64_t mine = 0;
#pragma unroll
                    for (int q = 0; q < MS_COOP_U; ++q) mine |= fu[q];
                    got = warp_or64(mine);
                }
                al |= got;
            }
            if ((int)lane == l) {
                acc = al;
                j = b2;
            }
            if (al != ml && b2 < el) rest |= 1u << l;
            rm &= rm - 1;
        }
        if (rest) ms_defer(p, L, rest, v, j);
        // depths and parents of the word, lane-major: for each lane found
        // anywhere in the word, its row entries of the 32 vertices go out
        // together.  Four lanes at a time: their parent gathers are in flight
        // together (one at a time each is a round trip of the word's chain:
        // RMAT-24 14.17 ms against 13.47), and the lane numbers are constants
        // but for the group's.
        // The unit's first pull level writes all of a word's entries but those
        // of lanes that push levels have found: -1 for a lane not found yet.
        // Rows are then written in whole lines by the level that finds most
        // entries, and not set to -1 before the search.
        const uint64_t todo_lanes = whole ? (v < g.n ? ~((const unsigned long long*)p.seen)[v] : 0ull) : acc;
        const uint64_t all = whole ? g.lanes : PAR || L.c.write_depth ? warp_or64(acc) : 0ull;
        __syncwarp();
        for (int j0 = 0; all >> j0; j0 += 4) {  // warp-uniform
            if (!((all >> j0) & 15ull)) {
                if (j0 == 60) break;
                continue;
            }
            const unsigned f = (unsigned)(acc >> j0) & 15u, wr = (unsigned)((todo_lanes & g.lanes) >> j0) & 15u;
            int par[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                par[i] = PAR && ((f >> i) & 1u) ? __ldg(g.csc_col + beg + pidx[lane * MS_PIDX_LD + j0 + i]) : -1;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (!((wr >> i) & 1u)) continue;
                if (L.c.write_depth && ((f >> i) & 1u)) sm.depth[j0 + i][v] = L.c.level + 1;
                int32_t* pp = PAR ? sm.parent[j0 + i] : nullptr;
                if (pp) pp[v] = par[i];
            }
            if (j0 == 60) break;
        }
        __syncwarp();
        if (acc) {
            ((unsigned long long*)L.c.f_next)[v] = acc;
            const uint64_t now = ((const unsigned long long*)p.seen)[v] | acc;
            ((unsigned long long*)p.seen)[v] = now;
            if (now == g.lanes) atomicOr(p.full + (v >> 5), 1u << lane);
            sm.fmask[me] |= acc;
            sm.lim[me] += 1;
            const unsigned dv = (unsigned)(g.symmetric ? (end - beg) : (__ldg(g.row_ptr + v + 1) - __ldg(g.row_ptr + v)));
            sm.beg[me] += (int)dv;  // a degree sum below 2^31
            if (acc == miss) sm.src[me] += (int)dv;  // no live lane misses v any more
        }
        }
    }
    L.ef = (unsigned)sm.beg[me];
    L.cnt = (unsigned)sm.lim[me];
    L.done_e = (unsigned)sm.src[me];
    L.lanes = sm.fmask[me];
}

// Long rows of a pull level: each is scanned by a whole CTA (rows dealt
// round-robin), MS_LONG_ITEMS*T entries per step, stopping once every live
// missing lane is found.  The CTA ORs the supplied lanes in shared memory and
// keeps the first supplier of each lane as its parent; it owns the row, so
// the accumulator and the parents are written with plain stores.
template <int T, bool PAR>
__device__ void ms_long_rows(const ParamsMS& p, const UnitView& g, MsSmem& sm, const uint64_t* f_cur, uint64_t live,
                             long long nl) {
    __shared__ unsigned long long s_or;
    __shared__ int s_prov[64];
    const unsigned long long* F = (const unsigned long long*)f_cur;
    const int per = MS_LONG_ITEMS * T;
    for (long long r = blockIdx.x; r < nl; r += gridDim.x) {
        const int v = p.longv[r];
        const int beg = (int)p.acc_long[r], end = __ldg(g.csc_ptr + v + 1);
        const uint64_t miss = live & ~((const unsigned long long*)p.seen)[v];
        if (threadIdx.x == 0) s_or = 0;
        __syncthreads();
        for (int lo = beg; lo < end && miss; lo += per) {  // CTA-uniform
            const int hi = min(end, lo + per);
#pragma unroll
            for (int k = 0; k < MS_LONG_ITEMS; ++k) {
                const int e = lo + k * T + (int)threadIdx.x;
                if (e < hi) {
                    const int u = __ldg(g.csc_col + e);
                    const uint64_t got = F[u] & miss;
                    if (got) {
                        const uint64_t old = atomicOr(&s_or, (unsigned long long)got);
                        uint64_t nb = PAR ? got & ~old : 0ull;
                        while (nb) {
                            const int b = __ffsll((long long)nb) - 1;
                            s_prov[b] = u;
                            nb &= nb - 1;
                        }
                    }
                }
            }
            __syncthreads();
            // every thread looks before any adds to s_or again: a thread that
            // saw the next step's lanes would leave a step before the others
            const bool all = s_or == miss;
            __syncthreads();
            if (all) break;
        }
        const uint64_t acc = s_or;
        if (threadIdx.x == 0) p.acc_long[r] = acc;
        if (PAR && threadIdx.x < 64 && ((acc >> threadIdx.x) & 1ull) && sm.parent[threadIdx.x])
            sm.parent[threadIdx.x][v] = s_prov[threadIdx.x];
        __syncthreads();
    }
}

// The deferred long rows found their lanes: depth, F_{i+1}, seen and the
// level counters (after ms_long_rows, before the next level).
__device__ void ms_long_finalize(const ParamsMS& p, const UnitView& g, MsSmem& sm, uint64_t* f_next, long long nl,
                                 int dnext, CountersMS* nxt, uint64_t live, bool write_depth) {
    const long long gtid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long gthreads = (long long)gridDim.x * blockDim.x;
    unsigned long long cnt = 0, ef = 0, done = 0;
    uint64_t ln = 0;
    for (long long r = gtid; r < nl; r += gthreads) {
        const uint64_t acc = __ldcg(p.acc_long + r);
        if (!acc) continue;
        const int v = p.longv[r];
        const uint64_t had = ((const unsigned long long*)f_next)[v];  // what the warp found, and counted
        ((unsigned long long*)f_next)[v] = had | acc;
        const uint64_t old = ((const unsigned long long*)p.seen)[v];
        ((unsigned long long*)p.seen)[v] = old | acc;
        uint64_t b = write_depth ? acc : 0ull;
        while (b) {
            const int j = __ffsll((long long)b) - 1;
            sm.depth[j][v] = dnext;
            b &= b - 1;
        }
        const unsigned long long dv = (unsigned long long)(__ldg(g.row_ptr + v + 1) - __ldg(g.row_ptr + v));
        if (!had) {
            cnt += 1;
            ef += dv;
        }
        if (((old | acc) & live) == live) done += dv;
        if ((old | acc) == g.lanes) atomicOr(p.full + (v >> 5), 1u << (v & 31));
        ln |= acc;
    }
    cnt = warp_sum(cnt);
    ef = warp_sum(ef);
    done = warp_sum(done);
    ln = warp_or64(ln);
    if ((threadIdx.x & 31) == 0) {
        if (cnt) atomicAdd(&nxt->a_len, cnt);
        if (ef) atomicAdd(&nxt->e_f, ef);
        if (done) atomicAdd(&nxt->done_e, done);
        if (ln) atomicOr((unsigned long long*)&nxt->lanes, (unsigned long long)ln);
    }
}

// Active list of F_i from its masks (after a pull level), with chunk units.
// A warp takes 8 x 32 masks at a time, all loaded before the first is looked
// at, and appends with one atomic where it finds any: the frontier is sparse
// here (after a pull level the next push has at most a few per cent of the
// vertices), so reading the masks is the cost.  (A block scan per 512 masks took
// 100 us for the 2^24 vertices of RMAT-24.)
__device__ void ms_masks_to_list(const ParamsMS& p, const UnitView& g, const uint64_t* f_cur, int4* a_cur,
                                 int2* u_cur, CountersMS* cur) {
    constexpr int R = 8;
    const unsigned lane = lane_id();
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    for (long long v0 = gwarp * (32 * R); v0 < g.n; v0 += nwarps * (32 * R)) {  // warp-uniform
        unsigned long long m[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long v = v0 + r * 32 + lane;
            m[r] = v < g.n ? __ldcg((const unsigned long long*)f_cur + v) : 0ull;
        }
        unsigned b[R];
        int total = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            b[r] = __ballot_sync(0xffffffffu, m[r] != 0);
            total += __popc(b[r]);
        }
        if (total == 0) continue;
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(&cur->conv, (unsigned long long)total);
        at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (m[r]) {
                const int v = (int)(v0 + r * 32 + lane);
                const int rb = __ldg(g.row_ptr + v), re = __ldg(g.row_ptr + v + 1);
                a_cur[at + __popc(b[r] & lanemask_lt())] = make_int4(v, rb, re, 0);
                if (re - rb >= p.chunk) ms_units(p, u_cur, cur, v, re - rb);
            }
            at += __popc(b[r]);
        }
    }
}

// The MS-BFS heuristic: Beamer's test on the lanes' summed counters.
__device__ __forceinline__ int ms_heuristic(const ParamsMS& p, const UnitView& g, long long a, long long e_f,
                                            long long m_u, long long a_prev, int prev_dir) {
    if (prev_dir == BFS_DIR_PULL) {
        bool stay = (a >= a_prev) || ((float)a * p.beta > (float)g.n);
        return stay ? BFS_DIR_PULL : BFS_DIR_PUSH_QUEUE;
    }
    if ((float)e_f * p.alpha > (float)m_u && a > a_prev) return BFS_DIR_PULL;
    return BFS_DIR_PUSH_QUEUE;
}

__device__ int ms_decide(const ParamsMS& p, const UnitView& g, MsSmem& sm, int level, long long a, long long e_f,
                         long long m_u, long long a_prev, int prev_dir, int deg_max) {
    int d;
    switch (p.policy) {
        case BFS_POLICY_PUSH: return BFS_DIR_PUSH_QUEUE;
        case BFS_POLICY_PULL: return BFS_DIR_PULL;
        case BFS_POLICY_SCHEDULE:
            d = p.schedule[level % p.schedule_len];
            return d == BFS_DIR_PULL ? BFS_DIR_PULL : BFS_DIR_PUSH_QUEUE;
        case BFS_POLICY_MLP: {
            const int h = ms_heuristic(p, g, a, e_f, m_u, a_prev, prev_dir);
            if (p.mlp && policy_in_band(e_f, m_u, p.alpha)) {
                if (threadIdx.x < 32) {
                    if (threadIdx.x == 0)
                        policy_features(sm.feat, a, e_f, m_u, a_prev, level, prev_dir, g.n, g.m, deg_max);
                    __syncwarp();
                    int c = policy_choice_warp(p.mlp, sm.feat, h, MLP_MARGIN);
                    if (threadIdx.x == 0) sm.mlp_out = (float)c;
                }
                __syncthreads();
                d = (int)sm.mlp_out;
                __syncthreads();
                return d == BFS_DIR_PULL ? BFS_DIR_PULL : BFS_DIR_PUSH_QUEUE;
            }
            return h;  // no weights, or a clear-cut level: the heuristic decides
        }
        default:
            return ms_heuristic(p, g, a, e_f, m_u, a_prev, prev_dir);
    }
}

// The frontier mask of level i: kept in the history for the first MS_HIST
// levels, two alternating buffers after that.
__device__ __forceinline__ uint64_t* ms_front(const ParamsMS& p, int i) {
    return i < MS_HIST ? p.hist + (int64_t)i * p.ncap : ((i & 1) ? p.F1 : p.F0);
}

// After the last level L of a unit: every depth row written whole.  A warp
// takes 32 consecutive vertices (lane = vertex).  The level of each search
// lane is gathered in bit planes: plane b holds the lanes found at a history
// level whose number has bit b, so a level costs a few ORs whatever it found;
// four lanes' plane bits are then spread over the bytes of a word (a multiply
// and a mask), all ones for an unreached lane.  A lane found only after the
// history (written as found) is left alone.  Each lane's 32 entries go out as
// one coalesced row segment.  `parents`: no level has written the parents of
// the lanes that found nothing.  The history masks used are cleared for the
// next unit.  (A byte table in shared memory, filled lane by lane, took twice the
// instructions.)
template <bool PAR>
__device__ void ms_depth_pass(const ParamsMS& p, const UnitView& g, MsSmem& sm, int levels, bool parents) {
    const unsigned lane = lane_id();
    const int lh = min(levels, MS_HIST);
    const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    const int ntiles = (g.n + 31) >> 5;
    for (int t = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); t < ntiles; t += nwarps) {
        const long long v = (long long)t * 32 + lane;
        const bool valid = v < g.n;
        uint64_t found = 0, pl[4] = {0, 0, 0, 0};
        for (int i0 = 0; i0 < lh; i0 += 4) {
            uint64_t b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) b[i] = valid && i0 + i < lh ? p.hist[(int64_t)(i0 + i) * p.ncap + v] : 0ull;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint64_t nb = b[i] & ~found;
                found |= b[i];
                if (i & 1) pl[0] |= nb;
                if (i & 2) pl[1] |= nb;
                if (i0 & 4) pl[2] |= nb;
                if (i0 & 8) pl[3] |= nb;
                if (b[i]) p.hist[(int64_t)(i0 + i) * p.ncap + v] = 0ull;
            }
        }
        // lanes found after the history have their depth already
        const uint64_t skip = levels > MS_HIST && valid ? ((const unsigned long long*)p.seen)[v] & ~found : 0ull;
        for (int j0 = 0; j0 < g.k; j0 += 4) {
            const auto spread = [&](uint64_t x) { return (((unsigned)(x >> j0) & 15u) * 0x00204081u) & 0x01010101u; };
            const unsigned w = spread(pl[0]) | spread(pl[1]) << 1 | spread(pl[2]) << 2 | spread(pl[3]) << 3 |
                               spread(~found) * 0xffu;
            const unsigned sk = valid ? (unsigned)(skip >> j0) : 15u;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (j0 + i < g.k && !((sk >> i) & 1u)) sm.depth[j0 + i][v] = (int)(signed char)(w >> (8 * i));
        }
        if (PAR && parents) {  // no pull level: -1 where a lane found nothing
            const uint64_t none = valid ? g.lanes & ~((const unsigned long long*)p.seen)[v] : 0ull;
            for (uint64_t any = warp_or64(none); any; any &= any - 1) {  // warp-uniform
                const int j = __ffsll((long long)any) - 1;
                if (((none >> j) & 1ull) && sm.parent[j]) sm.parent[j][v] = -1;
            }
        }
    }
}

template <int T, bool PAR>
__device__ void msbfs_body(const ParamsMS& p) {
    __shared__ MsSmem sm;
    CtlMS* ctl = p.ctl;
    const unsigned nblocks = gridDim.x;
    const long long gtid = (long long)blockIdx.x * T + threadIdx.x;
    const long long gthreads = (long long)gridDim.x * T;
    const unsigned warp = threadIdx.x >> 5;
    unsigned bar_target = 0;
    int total_levels = 0;
    // a launch that ended early (error, time limit) left history masks set:
    // clear the whole history before use
    if (ld_volatile_i32(p.hist_dirty)) {
        for (long long i = gtid; i < (long long)MS_HIST * p.ncap; i += gthreads) p.hist[i] = 0;
    }
    if (!grid_sync(&ctl->bar, nblocks, bar_target, p.timeout_ns)) return;
    if (gtid == 0) *p.hist_dirty = 1;
    for (int ui = 0; ui < p.n_units; ++ui) {
        const MsUnit* U = p.units + ui;
        UnitView& g = sm.g;
        if (threadIdx.x == 0) {  // the last unit's readers have passed its closing barrier
            g.row_ptr = U->row_ptr;
            g.col = U->col;
            g.csc_ptr = U->csc_ptr;
            g.csc_col = U->csc_col;
            g.isolated = U->isolated;
            g.m = U->m;
            g.n = U->n;
            g.k = U->k;
            g.symmetric = U->symmetric;
            g.deg_max = U->deg_max;
            g.lanes = (U->k >= 64) ? ~0ull : ((1ull << U->k) - 1);
        }
        int deg_max = U->deg_max;
        if (threadIdx.x < 64) {
            sm.depth[threadIdx.x] = threadIdx.x < U->k ? U->depth[threadIdx.x] : nullptr;
            sm.parent[threadIdx.x] = threadIdx.x < U->k ? U->parent[threadIdx.x] : nullptr;
        }
        __syncthreads();
        // init: masks, outputs (-1), counters
        for (long long v = gtid; v < g.n; v += gthreads) {
            p.seen[v] = 0;
            p.F0[v] = 0;
            p.F1[v] = 0;
        }
        for (long long w = gtid; w < (g.n + 31) >> 5; w += gthreads) {
            unsigned bits = __ldg(g.isolated + w);
            if (w * 32 + 32 > g.n) bits |= ~((1u << (g.n & 31)) - 1u);
            p.full[w] = bits;
        }
        // depths are written whole by ms_depth_pass, the parents of lanes that
        // find nothing by the first pull level, or there too
        if (gtid == 0) {
            for (int s = 0; s < 3; ++s) {
                ctl->slot[s].a_len = 0;
                ctl->slot[s].u_len = 0;
                ctl->slot[s].e_f = 0;
                ctl->slot[s].conv = 0;
                ctl->slot[s].lanes = 0;
                ctl->slot[s].done_e = 0;
                ctl->slot[s].pull_next = 0;
                ctl->slot[s].long_len = 0;
            }
            ctl->slot[0].lanes = g.lanes;
        }
        if (!grid_sync(&ctl->bar, nblocks, bar_target, p.timeout_ns)) return;
        if (blockIdx.x == 0 && threadIdx.x < (unsigned)g.k) {
            int j = threadIdx.x;
            int s = U->src[j];
            const unsigned long long was = atomicOr((unsigned long long*)p.seen + s, 1ull << j);
            if ((was | 1ull << j) == g.lanes) atomicOr(p.full + (s >> 5), 1u << (s & 31));
            unsigned long long old = atomicOr((unsigned long long*)ms_front(p, 0) + s, 1ull << j);
            if (sm.parent[j]) sm.parent[j][s] = s;
            if (old == 0) {
                const int rb = g.row_ptr[s], re = g.row_ptr[s + 1], deg = re - rb;
                unsigned long long idx = atomicAdd(&ctl->slot[0].a_len, 1ull);
                p.A0[idx] = make_int4(s, rb, re, 0);
                atomicAdd(&ctl->slot[0].e_f, (unsigned long long)deg);
                if (deg >= p.chunk) ms_units(p, p.U0, &ctl->slot[0], s, deg);
            }
        }
        if (!grid_sync(&ctl->bar, nblocks, bar_target, p.timeout_ns)) return;
        long long m_u = g.m, a_prev = 0;
        int prev_dir = BFS_DIR_PUSH_QUEUE;
        int unit_levels = 0;
        int list_valid = 0;  // level whose active list (and chunk units) exists
        bool cnt_ok = false;     // sm.cnt holds the level's counters
        bool par_set = false;    // every parent entry has been written once
        for (int level = 0;; ++level) {
            CountersMS* cur = &ctl->slot[level % 3];
            CountersMS* nxt = &ctl->slot[(level + 1) % 3];
            unsigned long long cv[5];
            if (cnt_ok) {
#pragma unroll
                for (int i = 0; i < 5; ++i) cv[i] = sm.cnt[i];
            } else {
                const unsigned long long* const csrc[5] = {&cur->a_len, &cur->e_f, &cur->lanes, &cur->u_len,
                                                           &cur->done_e};
                cta_load_u64<5>(csrc, cv);
            }
            long long a = (long long)cv[0];
            long long e_f = (long long)cv[1];
            const uint64_t live = (uint64_t)cv[2];
            if (a == 0) break;
            if (level >= p.max_levels) {
                if (gtid == 0) atomicCAS(&ctl->bar.err, 0, (int)DEV_LEVELS);
                return;
            }
            // m_u: degree sum of the vertices some live lane has not seen,
            // the rows a pull level would scan (the batched reading of
            // Beamer's unexplored edges; summing every lane's frontier edges
            // instead drove it to zero within a few levels of a long search)
            m_u = max(m_u - (long long)cv[4], 1ll);
            int dir = ms_decide(p, g, sm, level, a, e_f, m_u, a_prev, prev_dir, deg_max);
            if (ui == 0 && gtid == 0 && p.log && level < p.log_cap) {
                bfs_level_record r;
                r.level = level;
                r.dir = dir;
                r.f = a;
                r.e_f = e_f;
                r.m_u = m_u;
                r.t_ns = (int64_t)globaltimer_ns();
                p.log[level] = r;
            }
            int4* a_cur = (level & 1) ? p.A1 : p.A0;
            int2* u_cur = (level & 1) ? p.U1 : p.U0;
            uint64_t* f_cur = ms_front(p, level);
            long long nunits = (long long)cv[3];
            if (dir != BFS_DIR_PULL && list_valid != level) {
                // active list of a pull-made frontier (it appends the chunk units)
                ms_masks_to_list(p, g, f_cur, a_cur, u_cur, cur);
                if (!grid_sync(&ctl->bar, nblocks, bar_target, p.timeout_ns)) return;
                list_valid = level;
                const unsigned long long* const usrc[1] = {&cur->u_len};
                unsigned long long uv[1];
                cta_load_u64<1>(usrc, uv);
                nunits = (long long)uv[0];
            }
            if (gtid == 0) {
                CountersMS* z = &ctl->slot[(level + 2) % 3];
                z->a_len = 0;
                z->u_len = 0;
                z->e_f = 0;
                z->conv = 0;
                z->lanes = 0;
                z->done_e = 0;
                z->pull_next = 0;
                z->long_len = 0;
            }
            if (threadIdx.x == 0) {  // its last readers have passed the level's barrier
                MsLevelConst& c = sm.lv;
                c.level = level;
                c.f_next = ms_front(p, level + 1);
                c.write_depth = level + 1 >= MS_HIST;
                c.clear_cur = level >= MS_HIST;
                c.a_next = (level & 1) ? p.A0 : p.A1;
                c.u_next = (level & 1) ? p.U0 : p.U1;
                c.next = nxt;
                c.live = live;
                c.cursor = &cur->pull_next;
                c.long_len = &cur->long_len;
                // m_u: degree sum of the vertices some live lane has not seen
                c.sparse = 8 * m_u < g.m;
                c.whole = PAR && !par_set && dir == BFS_DIR_PULL;
                c.pull_chunk = 1;
                const int words = (g.n + 31) >> 5, warps = (int)nblocks * (T / 32);
                c.long_row = words <= MS_FEW_WORDS * warps ? MS_LONG_ROW_SMALL : MS_LONG_ROW;
                if (c.sparse) {
                    const int fair = words / (warps * MS_PULL_TAKES);
                    c.pull_chunk = min(max(fair, 1), MS_PULL_CHUNK);
                }
            }
            __syncthreads();
            MsLevel L{sm.lv, 0u, 0u, 0u, 0ull, 0};
            const bool pull = dir == BFS_DIR_PULL;
            par_set |= pull;
            if (pull) ms_pull_level<PAR>(p, g, L, sm, f_cur);
            else ms_push_level<T, PAR>(p, g, L, sm, a_cur, u_cur, f_cur, a, nunits);
            // the level's counters: a share a warp, one atomic each for the CTA
            const uint64_t ln = warp_or64(L.lanes);
            const unsigned ef = __reduce_add_sync(0xffffffffu, L.ef), cn = __reduce_add_sync(0xffffffffu, L.cnt),
                           dn = __reduce_add_sync(0xffffffffu, L.done_e);
            if ((threadIdx.x & 31) == 0) {
                sm.red[0][warp] = ef;
                sm.red[1][warp] = cn;
                sm.red[2][warp] = dn;
                sm.red[3][warp] = ln;
            }
            if (!pull) list_valid = level + 1;
            // masks of F_i that were not zeroed as they were read, in a buffer F_{i+2} needs
            const bool sweep = level >= MS_HIST && (pull || nunits > 0);
            auto add = [&]() {
                unsigned long long t[4] = {0, 0, 0, 0};
                for (int i = 0; i < T / 32; ++i) {
                    t[0] += sm.red[0][i];
                    t[1] += sm.red[1][i];
                    t[2] += sm.red[2][i];
                    t[3] |= sm.red[3][i];
                }
                if (t[0]) atomicAdd(&nxt->e_f, t[0]);
                if (t[1]) atomicAdd(&nxt->a_len, t[1]);
                if (t[2]) atomicAdd(&nxt->done_e, t[2]);
                if (t[3]) atomicOr(&nxt->lanes, t[3]);
            };
            // read once the level is complete everywhere.  A CTA may be in the
            // next level already: that changes neither these (its list
            // conversion adds units, which are read again) nor this level's
            // long_len, unless it is zero anyway or every CTA waits below
            auto load = [&]() {
                sm.cnt[0] = ld_cg_u64(&nxt->a_len);
                sm.cnt[1] = ld_cg_u64(&nxt->e_f);
                sm.cnt[2] = ld_cg_u64(&nxt->lanes);
                sm.cnt[3] = ld_cg_u64(&nxt->u_len);
                sm.cnt[4] = ld_cg_u64(&nxt->done_e);
                sm.cnt[5] = ld_cg_u64(&cur->long_len);
            };
            if (!grid_sync(&ctl->bar, nblocks, bar_target, p.timeout_ns, add, load)) return;
            const long long nl = pull ? (long long)sm.cnt[5] : 0;
            if (nl > 0) {  // grid-uniform
                ms_long_rows<T, PAR>(p, g, sm, f_cur, live, nl);
                if (!grid_sync(&ctl->bar, nblocks, bar_target, p.timeout_ns)) return;
                ms_long_finalize(p, g, sm, sm.lv.f_next, nl, level + 1, nxt, live, sm.lv.write_depth);
            }
            if (sweep) {
                if (pull) {
                    for (long long v = gtid; v < g.n; v += gthreads) f_cur[v] = 0;
                } else {
                    for (long long q = gtid; q < nunits; q += gthreads) f_cur[u_cur[q].x] = 0;
                }
            }
            if (nl > 0 || sweep) {
                if (!grid_sync(&ctl->bar, nblocks, bar_target, p.timeout_ns, NoArrivalWork(), load)) return;
            }
            cnt_ok = true;
            a_prev = a;
            prev_dir = dir;
            ++total_levels;
            ++unit_levels;
        }
        // the unit's depth rows; a barrier before the next unit reuses seen
        ms_depth_pass<PAR>(p, g, sm, unit_levels, PAR && !par_set);
        if (!grid_sync(&ctl->bar, nblocks, bar_target, p.timeout_ns)) return;
    }
    if (gtid == 0) {
        ctl->levels = total_levels;
        *p.hist_dirty = 0;  // every history level used was cleared by its depth pass
    }
}

// PAR: some search of the launch wants its parents.
template <int T, bool PAR>
__global__ void __launch_bounds__(T, 2) msbfs_kernel(ParamsMS p) {
    msbfs_body<T, PAR>(p);
    if (threadIdx.x == 0) {
        int e = ld_volatile_i32(&p.ctl->bar.err);
        if (e) atomicCAS(p.sticky, 0, e);
    }
}


__global__ void ms_count_units_kernel(const int32_t* row_ptr, int32_t n, int32_t chunk, unsigned long long* out) {
    unsigned long long s = 0;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
        int d = row_ptr[v + 1] - row_ptr[v];
        if (d >= chunk) s += (unsigned long long)((d + chunk - 1) / chunk);
    }
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

static int64_t count_units(bfs_graph* g, int32_t chunk, cudaStream_t st) {
    if (g->deg_max < chunk) return 0;
    std::lock_guard<std::mutex> guard(g->units_lock);
    if (g->units_chunk == chunk) return g->units_count;
    unsigned long long* d = nullptr;
    unsigned long long h = 0;
    if (cudaMallocAsync(&d, 8, st) != cudaSuccess) return -1;
    cudaError_t e = cudaMemsetAsync(d, 0, 8, st);
    if (e == cudaSuccess) {
        ms_count_units_kernel<<<num_sms() * 8, 256, 0, st>>>(g->row_ptr, g->n, chunk, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, 8, cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(d, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return -1;  // and nothing is kept: a count of 0 would refuse every later batch
    }
    g->units_chunk = chunk;
    g->units_count = (int64_t)h;
    return (int64_t)h;
}

// The zeroing is ordered on the stream of the launch that uses the workspace
// first (on the default stream it would not be ordered before a launch on a
// non-blocking one).
static bfs_status alloc_wsms(int32_t ncap, int64_t ucap, int32_t chunk, int32_t units_cap, cudaStream_t st,
                             WorkspaceMS** out) {
    WorkspaceMS* w = new (std::nothrow) WorkspaceMS();
    if (!w) return fail(BFS_ENOMEM, "host allocation");
    w->ncap = ncap;
    w->ucap = ucap;
    w->chunk = chunk;
    w->units_cap = units_cap;
    bool ok = cudaMalloc(&w->seen, (size_t)ncap * 8) == cudaSuccess;
    for (int i = 0; i < 2 && ok; ++i)
        ok = cudaMalloc(&w->front[i], (size_t)ncap * 8) == cudaSuccess &&
             cudaMalloc(&w->act[i], (size_t)ncap * sizeof(int4)) == cudaSuccess &&
             cudaMalloc(&w->U[i], (size_t)ucap * sizeof(int2)) == cudaSuccess;
    ok = ok && cudaMalloc(&w->ctl, sizeof(CtlMS)) == cudaSuccess;
    ok = ok && cudaMalloc(&w->d_sticky, 4) == cudaSuccess && cudaMemsetAsync(w->d_sticky, 0, 4, st) == cudaSuccess;
    ok = ok && cudaMalloc(&w->d_units, sizeof(MsUnit) * (size_t)units_cap) == cudaSuccess;
    ok = ok && cudaMalloc(&w->longv, (size_t)ncap * 4) == cudaSuccess;
    ok = ok && cudaMalloc(&w->acc_long, (size_t)ncap * 8) == cudaSuccess;
    ok = ok && cudaMalloc(&w->hist, (size_t)MS_HIST * ncap * 8) == cudaSuccess &&
         cudaMemsetAsync(w->hist, 0, (size_t)MS_HIST * ncap * 8, st) == cudaSuccess;
    ok = ok && cudaMalloc(&w->full, (size_t)div_up(ncap, 32) * 4) == cudaSuccess;
    ok = ok && cudaMalloc(&w->hist_dirty, 4) == cudaSuccess && cudaMemsetAsync(w->hist_dirty, 0, 4, st) == cudaSuccess;
    ok = ok && cudaMallocHost(&w->h_ctl, sizeof(CtlMS)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        free_wsms(w);
        return fail(BFS_ENOMEM, "MS-BFS workspace for n=%d", ncap);
    }
    *out = w;
    return BFS_OK;
}

static int coop_blocks_ms(const void* kernel, size_t smem, int blocks_per_sm) {
    int per_sm = 0;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, MS_T, smem);
    if (per_sm < 1) per_sm = 1;
    if (blocks_per_sm > 0) per_sm = std::min(per_sm, blocks_per_sm);
    return per_sm * num_sms();
}

static MsUnit make_unit(const bfs_graph* g) {
    MsUnit u;
    memset(&u, 0, sizeof(u));
    u.row_ptr = g->row_ptr;
    u.col = g->col;
    u.csc_ptr = g->csc_ptr;
    u.csc_col = g->csc_col;
    u.isolated = g->isolated;
    u.m = g->m;
    u.n = g->n;
    u.symmetric = g->symmetric;
    u.deg_max = g->deg_max;
    return u;
}

static bfs_status launch_ms(WorkspaceMS* w, const std::vector<MsUnit>& units, const bfs_options& o, const float* mlp,
                            const int8_t* d_sched, cudaStream_t st, bfs_level_record* d_log = nullptr) {
    if ((int32_t)units.size() > w->units_cap) return fail(BFS_EINVAL, "too many units");
    BFS_CUDA(cudaMemcpyAsync(w->d_units, units.data(), sizeof(MsUnit) * units.size(), cudaMemcpyHostToDevice, st));
    BFS_CUDA(cudaMemsetAsync(w->ctl, 0, sizeof(CtlMS), st));
    ParamsMS p{};
    p.units = w->d_units;
    p.n_units = (int32_t)units.size();
    p.seen = w->seen;
    p.F0 = w->front[0];
    p.F1 = w->front[1];
    p.A0 = w->act[0];
    p.A1 = w->act[1];
    p.U0 = w->U[0];
    p.U1 = w->U[1];
    p.ucap = w->ucap;
    p.ctl = w->ctl;
    p.sticky = w->d_sticky;
    p.policy = o.policy;
    p.alpha = o.batch_alpha;
    p.beta = o.batch_beta;
    p.schedule = d_sched;
    p.schedule_len = o.schedule_len;
    p.mlp = mlp;
    p.chunk = o.chunk;
    p.medium = o.medium;
    p.pull_serial = std::max(o.pull_serial, 1) * 2;  // all missing lanes are rarely found early: longer serial scans
    p.timeout_ns = o.barrier_timeout_ns;
    p.max_levels = o.max_levels > 0 ? o.max_levels : INT32_MAX / 2;
    p.log = d_log;
    p.log_cap = d_log ? o.level_log_cap : 0;
    p.longv = w->longv;
    p.acc_long = w->acc_long;
    p.hist = w->hist;
    p.ncap = w->ncap;
    p.hist_dirty = w->hist_dirty;
    p.full = w->full;
    bool par = false;
    for (const MsUnit& u : units)
        for (int j = 0; j < u.k; ++j) par |= u.parent[j] != nullptr;
    const void* kernel = par ? (const void*)msbfs_kernel<MS_T, true> : (const void*)msbfs_kernel<MS_T, false>;
    // Little work a level: one CTA an SM, for the shorter barrier.  Entries
    // bound a dense level's work; on bounded-degree graphs a level is a
    // frontier's worth, vertices times lanes over a long diameter.  us, two
    // CTAs / one: RMAT-12 79 / 68, RMAT-15 247 / 234, RMAT-16 262 / 272, RMAT-17 230 /
    // 275; grids with 4 lanes, 400^2 6054 / 5429, 1000^2 14393 / 12824, with 48,
    // 700^2 12549 / 12645, 1000^2 22289 / 22959.
    bool light = true;
    for (const MsUnit& u : units)
        light &= u.m <= (1 << 20) || (u.deg_max <= 16 && (int64_t)u.n * u.k <= (1 << 24));
    const size_t smem = par ? MS_PIDX_BYTES : MS_QBUF_BYTES;
    int blocks = coop_blocks_ms(kernel, smem, light && o.blocks_per_sm == 0 ? 1 : o.blocks_per_sm);
    void* args[] = {(void*)&p};
    BFS_CUDA(cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(MS_T), args, smem, st));
    return BFS_OK;
}

// k sources over one graph, in units of 64 lanes; depth/parent: [k][n].
bfs_status run_msbfs(bfs_graph* g, const int32_t* sources, int32_t k, int32_t* depth, int32_t* parent,
                     const bfs_options& o, const float* mlp_dev, cudaStream_t st) {
    int32_t nunits = (int32_t)div_up(k, 64);
    WorkspaceMS* w = g->wsms;
    if (!w || w->chunk != o.chunk || w->units_cap < nunits) {
        if (w) {
            BFS_CUDA(cudaStreamSynchronize(st));
            free_wsms(w);
            g->wsms = nullptr;
        }
        int64_t uc = count_units(g, o.chunk, st);
        if (uc < 0) return fail(BFS_ECUDA, "unit count");
        bfs_status s = alloc_wsms(g->n, uc + 64, o.chunk, std::max(nunits, 4), st, &w);
        if (s != BFS_OK) return s;
        g->wsms = w;
    }
    const int64_t n = g->n;
    bool dev_out = is_device_ptr(depth) && (!parent || is_device_ptr(parent));
    int32_t *dd = depth, *dp = parent;
    if (!dev_out) {
        if (cudaMallocAsync(&dd, (size_t)k * n * 4, st) != cudaSuccess ||
            (parent && cudaMallocAsync(&dp, (size_t)k * n * 4, st) != cudaSuccess)) {
            cudaGetLastError();
            return fail(BFS_ENOMEM, "staging outputs for %d sources", k);
        }
    }
    int8_t* d_sched = nullptr;
    if (o.policy == BFS_POLICY_SCHEDULE) {
        if (!o.schedule || o.schedule_len <= 0) return fail(BFS_EINVAL, "schedule policy needs a schedule");
        BFS_CUDA(cudaMallocAsync(&d_sched, o.schedule_len, st));
        BFS_CUDA(cudaMemcpyAsync(d_sched, o.schedule, o.schedule_len, cudaMemcpyHostToDevice, st));
    }
    std::vector<MsUnit> units;
    for (int32_t u0 = 0; u0 < k; u0 += 64) {
        MsUnit u = make_unit(g);
        u.k = std::min(64, k - u0);
        for (int j = 0; j < u.k; ++j) {
            u.src[j] = sources[u0 + j];
            u.depth[j] = dd + (int64_t)(u0 + j) * n;
            u.parent[j] = dp ? dp + (int64_t)(u0 + j) * n : nullptr;
        }
        units.push_back(u);
    }
    bfs_level_record* d_log = nullptr;
    if (o.level_log && o.level_log_cap > 0)
        BFS_CUDA(cudaMallocAsync(&d_log, sizeof(bfs_level_record) * o.level_log_cap, st));
    bfs_status s = launch_ms(w, units, o, mlp_dev, d_sched, st, d_log);
    if (d_sched) cudaFreeAsync(d_sched, st);
    if (d_log) {
        if (s == BFS_OK) {
            BFS_CUDA(cudaMemcpyAsync(w->h_ctl, w->ctl, sizeof(CtlMS), cudaMemcpyDeviceToHost, st));
            BFS_CUDA(cudaStreamSynchronize(st));
            int nl = std::min(w->h_ctl->levels, o.level_log_cap);
            if (nl > 0) BFS_CUDA(cudaMemcpy(o.level_log, d_log, sizeof(bfs_level_record) * nl, cudaMemcpyDeviceToHost));
        }
        cudaFreeAsync(d_log, st);
    }
    if (s == BFS_OK && o.levels_out) {
        BFS_CUDA(cudaMemcpyAsync(w->h_ctl, w->ctl, sizeof(CtlMS), cudaMemcpyDeviceToHost, st));
        BFS_CUDA(cudaStreamSynchronize(st));
        *o.levels_out = w->h_ctl->levels;
    }
    if (!dev_out) {
        cudaError_t e = cudaSuccess;
        if (s == BFS_OK) e = cudaMemcpyAsync(depth, dd, (size_t)k * n * 4, cudaMemcpyDeviceToHost, st);
        if (s == BFS_OK && e == cudaSuccess && parent) e = cudaMemcpyAsync(parent, dp, (size_t)k * n * 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        cudaFreeAsync(dd, st);
        if (dp) cudaFreeAsync(dp, st);
        if (s == BFS_OK && e != cudaSuccess) s = cuda_fail(e, "copy outputs to host");
        if (s == BFS_OK) {
            int err = msbfs_sticky_error(g);
            if (err) s = device_error(err, o.barrier_timeout_ns);
        }
    }
    return s;
}

// Queries over several graphs in one launch: grouped per graph, 64 lanes a unit.
bfs_status run_mixed(const bfs_graph* const* graphs, int32_t n_graphs, const int32_t* graph_of_query,
                     const int32_t* sources, int32_t nq, int32_t* const* depth, int32_t* const* parent,
                     const bfs_options& o, cudaStream_t st) {
    (void)n_graphs;  // bfs_run_mixed has checked every graph_of_query[q] against it
    std::map<int, std::vector<int>> by_graph;
    for (int q = 0; q < nq; ++q) by_graph[graph_of_query[q]].push_back(q);
    std::vector<MsUnit> units;
    bfs_graph* big = nullptr;
    int64_t ucap = 1;
    for (auto& kv : by_graph) {
        bfs_graph* g = const_cast<bfs_graph*>(graphs[kv.first]);
        if (!big || g->n > big->n) big = g;
        int64_t uc = count_units(g, o.chunk, st);
        if (uc < 0) return fail(BFS_ECUDA, "unit count");
        ucap = std::max(ucap, uc + 64);
        const std::vector<int>& qs = kv.second;
        for (size_t i = 0; i < qs.size(); i += 64) {
            MsUnit u = make_unit(g);
            u.k = (int32_t)std::min<size_t>(64, qs.size() - i);
            for (int j = 0; j < u.k; ++j) {
                int q = qs[i + j];
                u.src[j] = sources[q];
                u.depth[j] = depth[q];
                u.parent[j] = parent ? parent[q] : nullptr;
            }
            units.push_back(u);
        }
    }
    // The workspace stays with the largest graph, until that is freed: making,
    // zeroing and freeing 0.9 GB was 1.3 ms of a call of 256 queries over
    // scales 16 to 22 (7.6 -> 6.3 ms).  A call is complete when it returns, so
    // the workspace is idle whenever its lock is free; a call that finds it
    // taken makes its own.
    std::unique_lock<std::mutex> kept(big->mix_lock, std::try_to_lock);
    WorkspaceMS* w = kept.owns_lock() ? big->wsmix : nullptr;
    bfs_status s = BFS_OK;
    if (w && (w->ucap < ucap || w->chunk != o.chunk || w->units_cap < (int32_t)units.size())) {
        free_wsms(w);
        w = big->wsmix = nullptr;
    }
    if (!w) {
        s = alloc_wsms(big->n, ucap, o.chunk, (int32_t)units.size(), st, &w);
        if (s != BFS_OK) return s;
        if (kept.owns_lock()) big->wsmix = w;
    }
    int8_t* d_sched = nullptr;
    if (o.policy == BFS_POLICY_SCHEDULE && o.schedule && o.schedule_len > 0) {
        if (cudaMalloc(&d_sched, o.schedule_len) == cudaSuccess)
            cudaMemcpy(d_sched, o.schedule, o.schedule_len, cudaMemcpyHostToDevice);
    }
    bfs_options oo = o;
    if (oo.policy == BFS_POLICY_SCHEDULE && !d_sched) oo.policy = BFS_POLICY_HEURISTIC;
    const float* mlp = nullptr;
    if (oo.policy == BFS_POLICY_MLP && oo.mlp) mlp = policy_device_weights(oo.mlp);
    s = launch_ms(w, units, oo, mlp, d_sched, st);
    if (s == BFS_OK) {
        cudaError_t e = cudaMemcpyAsync(w->h_ctl, w->ctl, sizeof(CtlMS), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) s = cuda_fail(e, "mixed batch");
        else if (w->h_ctl->bar.err) s = device_error(w->h_ctl->bar.err, o.barrier_timeout_ns);
        if (s == BFS_OK && o.levels_out) *o.levels_out = w->h_ctl->levels;
    } else {
        cudaStreamSynchronize(st);
    }
    cudaFree(d_sched);
    if (!kept.owns_lock()) free_wsms(w);
    return s;
}

}  // namespace bfsgb
