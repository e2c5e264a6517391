// builder.cu -- graph construction on the device: the S x D tensor G of
// Cascade 1 (Eq. G) in CSR form (Section 4.C), plus its rank swizzle to
// d-major order (CSC, Section 4.B, B.4) for pull levels.
//
//   edge list --> 64-bit (s,d) keys --(LSD radix sort)--> unique keys E,
//   sorted by (s,d) --(the same sort by d alone, stable)--> L, sorted by (d,s)
//
// A directed graph's CSR is E and its CSC is L.  A symmetric graph without
// repeats and self-loops (the default flags) sorts every edge once, as
// (min, max): row v is then v's part of L (neighbours below v) followed by v's
// part of E (neighbours above), both ascending, and an entry's place needs
// only the two parts' row starts:
//   E[i] = (a, b):  col[firstL[a + 1] + i] = b
//   L[j] = (a, b):  col[firstE[b] + j] = a,    row_ptr[v] = firstE[v] + firstL[v].
// That is m keys through the full-width passes and the unique ones through
// half of them, instead of 2m through all.
//
// Bound by memory passes: every radix pass reads the keys twice and writes
// them once.  RMAT-22 (67 M edges, 128 M CSR entries), around the call: 21.1 ms
// with 2m keys in 8-bit digits, keys scattered one by one, separate flag,
// scan and compaction passes and 4.4 GB from the stream-ordered pool; 6.4 ms
// now, 4.8 ms of it kernels.
#include "common.cuh"

#include <algorithm>
#include <vector>

namespace bfsgb {

namespace {

// --------------------------------------------------------------- scan u32
constexpr int SCAN_THREADS = 1024;

__device__ __forceinline__ uint32_t block_excl_scan_u32(uint32_t x, uint32_t* tmp, uint32_t* total) {
    unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += y;
    }
    if (lane == 31) tmp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nw ? tmp[lane] : 0, wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if ((int)lane >= o) wi += y;
        }
        if (lane < nw) tmp[lane] = wi - w;
        if (lane == 31) tmp[32] = wi;
    }
    __syncthreads();
    uint32_t r = tmp[warp] + incl - x;
    *total = tmp[32];
    __syncthreads();
    return r;
}

// single CTA: exclusive scan of `count` sums in place, carrying across chunks
__global__ void scan_sums_kernel(uint32_t* sums, int64_t count, uint32_t* grand_total) {
    __shared__ uint32_t tmp[33];
    uint32_t carry = 0;
    for (int64_t base = 0; base < count; base += SCAN_THREADS) {
        int64_t idx = base + threadIdx.x;
        uint32_t x = idx < count ? sums[idx] : 0, total;
        uint32_t ex = block_excl_scan_u32(x, tmp, &total);
        if (idx < count) sums[idx] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0 && grand_total) *grand_total = carry;
}

struct Scratch {
    std::vector<void*> ptrs;
    cudaStream_t st;
    explicit Scratch(cudaStream_t s) : st(s) {}
    template <typename T>
    cudaError_t alloc(T** p, size_t count) {
        cudaError_t e = cudaMallocAsync((void**)p, std::max<size_t>(count, 1) * sizeof(T), st);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
    ~Scratch() {
        for (void* p : ptrs) cudaFreeAsync(p, st);
    }
};

// ------------------------------------------------------------ radix sort
// Stable LSD radix sort of 64-bit keys, up to RS_BITS bits a pass.  Per pass:
//   upsweep   a CTA counts the digits of a chunk of consecutive tiles and leaves
//             each tile's counts before it within the chunk;
//   chunk scan  the chunks' totals become prefixes, digit by digit;
//   downsweep a CTA ranks a tile's keys (warp by warp in key order, equal
//             digits found with ballots), puts them in digit order in shared
//             memory and stores each digit's run contiguously.
// 9 bits and 6144 keys a tile: a run is 96 bytes on average, and 44 bits (2^22
// vertices) take five passes.  A tile needs 48 KB of shared memory for the
// exchange and 32 KB of per-warp counts; at 64 registers two CTAs fit an SM.
// RMAT-22 builds by tile: 8192 keys (spills) 6.7 ms, 6144 6.4, 4096 6.5, 2048
// 7.1; match-any in place of the ballots 0.6 ms more.
constexpr int RS_T = 512;
constexpr int RS_WARPS = RS_T / 32;
constexpr int RS_ITEMS = 12;
constexpr int RS_OCC = 2;
constexpr int RS_TILE = RS_T * RS_ITEMS;
constexpr int RS_BITS = 9;
constexpr int RS_BINS = 1 << RS_BITS;
constexpr int RS_CHUNK = 8;  // tiles a counting CTA takes, where there are enough of them
static_assert(RS_BINS == RS_T, "a thread per digit");

// Where a pass reads its keys.
enum { KEYS_ARRAY = 0, KEYS_DIRECTED = 1, KEYS_UNDIRECTED = 2, KEYS_BOTH = 3 };
struct KeySrc {
    const uint64_t* keys;  // KEYS_ARRAY
    const int32_t* src;    // the others: key s << bits | d of edge i (KEYS_DIRECTED), of its ends in
    const int32_t* dst;    // order (KEYS_UNDIRECTED), or of both directions of edge i / 2 (KEYS_BOTH)
    int bits;
};

template <int MODE>
__device__ __forceinline__ uint64_t load_key(const KeySrc& k, int64_t i, uint32_t n, bool& wrong) {
    if constexpr (MODE == KEYS_ARRAY) {
        return __ldcs((const unsigned long long*)k.keys + i);
    } else {
        const int64_t e = MODE == KEYS_BOTH ? i >> 1 : i;
        uint32_t s = (uint32_t)__ldg(k.src + e), d = (uint32_t)__ldg(k.dst + e);
        wrong |= s >= n || d >= n;  // negative ids too
        if ((MODE == KEYS_BOTH && (i & 1)) || (MODE == KEYS_UNDIRECTED && s > d)) {
            const uint32_t x = s;
            s = d;
            d = x;
        }
        return ((uint64_t)s << k.bits) | d;
    }
}

// hist[tile][digit] = keys of the tile's chunk before the tile, chunk[c][digit] =
// keys of the chunk.  Reading edges, it also checks their ids (*bad); an id
// out of range only makes a wrong digit here, and the build stops before
// anything is indexed by it.
template <int MODE>
__global__ void __launch_bounds__(RS_T)
    radix_upsweep_kernel(KeySrc ks, int64_t count, int shift, uint32_t mask, int per, uint32_t* __restrict__ hist,
                         uint32_t* __restrict__ chunk, int32_t n, int* bad) {
    __shared__ uint32_t h[RS_BINS];
    h[threadIdx.x] = 0;
    __syncthreads();
    bool wrong = false;
    for (int t = 0; t < per; ++t) {
        const int64_t tile = (int64_t)blockIdx.x * per + t, base = tile * RS_TILE;
        if (base >= count) break;  // CTA-uniform
        hist[tile * RS_BINS + threadIdx.x] = h[threadIdx.x];
        __syncthreads();
        uint64_t key[RS_ITEMS];
#pragma unroll
        for (int i = 0; i < RS_ITEMS; ++i) {
            const int64_t at = base + i * RS_T + threadIdx.x;
            key[i] = at < count ? load_key<MODE>(ks, at, (uint32_t)n, wrong) : 0;
        }
#pragma unroll
        for (int i = 0; i < RS_ITEMS; ++i) {
            if (base + i * RS_T + threadIdx.x < count) atomicAdd(&h[(uint32_t)(key[i] >> shift) & mask], 1u);
        }
        __syncthreads();
    }
    chunk[(int64_t)blockIdx.x * RS_BINS + threadIdx.x] = h[threadIdx.x];
    if (MODE != KEYS_ARRAY && wrong) atomicExch(bad, 1);
}

// Prefix over the chunks of each digit, in place; total[digit].  A CTA takes
// 32 digits, 32 groups of chunks side by side.
__global__ void __launch_bounds__(1024) radix_chunk_scan_kernel(uint32_t* chunk, int64_t nchunks, uint32_t* total) {
    __shared__ uint32_t s[32][33];
    const int dl = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int d = blockIdx.x * 32 + dl;
    const int64_t per = div_up(nchunks, 32), c0 = g * per, c1 = min(nchunks, c0 + per);
    uint32_t sum = 0;
#pragma unroll 8
    for (int64_t c = c0; c < c1; ++c) sum += chunk[c * RS_BINS + d];
    s[g][dl] = sum;
    __syncthreads();
    uint32_t before = 0;
    for (int i = 0; i < g; ++i) before += s[i][dl];
    if (g == 31) total[d] = before + sum;
#pragma unroll 4
    for (int64_t c = c0; c < c1; ++c) {
        const uint32_t x = chunk[c * RS_BINS + d];
        chunk[c * RS_BINS + d] = before;
        before += x;
    }
}

struct alignas(16) RadixSmem {
    uint64_t key[RS_TILE];
    uint32_t cnt[RS_WARPS][RS_BINS];  // keys of the digit in the warps before, then their place in the tile
    uint32_t out[RS_BINS];            // global place of the digit's run less its place in the tile
    uint32_t tmp[33];
};

// NB: bits of the digit (at most; one ballot each)
template <int MODE, int NB>
__global__ void __launch_bounds__(RS_T, RS_OCC)
    radix_downsweep_kernel(KeySrc ks, uint64_t* __restrict__ keys_out, int64_t count, int shift, uint32_t mask,
                           int per, const uint32_t* __restrict__ hist, const uint32_t* __restrict__ chunk,
                           const uint32_t* __restrict__ total) {
    extern __shared__ __align__(16) unsigned char radix_dyn[];
    RadixSmem& sm = *reinterpret_cast<RadixSmem*>(radix_dyn);
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile = blockIdx.x, base = tile * RS_TILE;
    const int tn = (int)min((int64_t)RS_TILE, count - base);
    // a warp's keys are consecutive: item i of lane l is key warp * 512 + i * 32 + l
    const int w0 = (int)warp * 32 * RS_ITEMS + (int)lane;
    uint64_t key[RS_ITEMS];
    bool wrong = false;  // the upsweep has looked
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i)
        key[i] = w0 + i * 32 < tn ? load_key<MODE>(ks, base + w0 + i * 32, 0u, wrong) : 0;
#pragma unroll
    for (int d = 0; d < RS_BINS; d += 128) *reinterpret_cast<uint4*>(&sm.cnt[warp][d + 4 * lane]) = make_uint4(0, 0, 0, 0);
    const uint32_t td = total[threadIdx.x];  // thread t: digit t
    uint32_t gstart = chunk[(tile / per) * RS_BINS + threadIdx.x] + hist[tile * RS_BINS + threadIdx.x];
    uint32_t all;
    gstart += block_excl_scan_u32(td, sm.tmp, &all);
    __syncwarp();
    uint16_t rank[RS_ITEMS];
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const bool valid = w0 + i * 32 < tn;
        const uint32_t d = (uint32_t)(key[i] >> shift) & mask;
        unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const bool set = (d >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, set);
            peers &= set ? m : ~m;
        }
        const unsigned below = peers & lanemask_lt();
        uint32_t before = 0;
        if (valid && below == 0) {  // the first of its digit: count them all
            before = sm.cnt[warp][d];
            sm.cnt[warp][d] = before + __popc(peers);
        }
        before = __shfl_sync(0xffffffffu, before, valid ? __ffs(peers) - 1 : 0);
        rank[i] = (uint16_t)(before + __popc(below));
        __syncwarp();
    }
    __syncthreads();
    {
        uint32_t run = 0;
#pragma unroll 4
        for (int w = 0; w < RS_WARPS; ++w) run += sm.cnt[w][threadIdx.x];
        uint32_t tt;
        uint32_t at = block_excl_scan_u32(run, sm.tmp, &tt);
        sm.out[threadIdx.x] = gstart - at;
#pragma unroll 4
        for (int w = 0; w < RS_WARPS; ++w) {
            const uint32_t c = sm.cnt[w][threadIdx.x];
            sm.cnt[w][threadIdx.x] = at;
            at += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        if (w0 + i * 32 < tn) {
            const uint32_t d = (uint32_t)(key[i] >> shift) & mask;
            sm.key[sm.cnt[warp][d] + rank[i]] = key[i];
        }
    }
    __syncthreads();
    for (int at = threadIdx.x; at < tn; at += RS_T) {
        const uint64_t k = sm.key[at];
        keys_out[(uint32_t)(sm.out[(uint32_t)(k >> shift) & mask] + (uint32_t)at)] = k;
    }
}

// Tiles a counting CTA takes: one while that leaves SMs idle (a chunk of eight
// tiles of a 65,000-edge list took its one CTA 15 us), then up to RS_CHUNK.
int64_t radix_ctas() { return (int64_t)num_sms() * 4; }
int radix_chunk(int64_t tiles) { return (int)std::max<int64_t>(1, std::min<int64_t>(RS_CHUNK, tiles / radix_ctas())); }

// Counters of a sort of up to `count` keys (kept over the passes and sorts of one build).
struct RadixScratch {
    uint32_t *hist = nullptr, *chunk = nullptr, *total = nullptr;
    static int64_t hist_words(int64_t count) { return div_up(std::max<int64_t>(count, 1), RS_TILE) * RS_BINS; }
    // The chunks of any sort of at most `count` keys, not of `count` alone: with
    // c < RS_CHUNK tiles a chunk there are fewer than (c + 1) * radix_ctas()
    // tiles, so at most 2 * radix_ctas() chunks (1215 tiles take 1215 at 608
    // CTAs, 1216 take 608).
    static int64_t chunk_words(int64_t count) {
        const int64_t tiles = div_up(std::max<int64_t>(count, 1), RS_TILE);
        return std::max(div_up(tiles, RS_CHUNK), std::min(tiles, 2 * radix_ctas())) * RS_BINS;
    }
    template <typename S>
    cudaError_t alloc(S& sc, int64_t count) {
        cudaError_t e = sc.alloc(&hist, hist_words(count));
        if (e == cudaSuccess) e = sc.alloc(&chunk, chunk_words(count));
        if (e == cudaSuccess) e = sc.alloc(&total, RS_BINS);
        return e;
    }
};

template <int MODE>
cudaError_t radix_pass(const KeySrc& ks, uint64_t* out, int64_t count, int shift, int nb, const RadixScratch& rs,
                       int32_t n, int* bad, cudaStream_t st) {
    const uint32_t mask = (1u << nb) - 1;
    const int64_t tiles = div_up(count, RS_TILE);
    const int per = radix_chunk(tiles);
    const int64_t chunks = div_up(tiles, per);
    auto down = nb <= 7 ? radix_downsweep_kernel<MODE, 7>
                        : nb == 8 ? radix_downsweep_kernel<MODE, 8> : radix_downsweep_kernel<MODE, 9>;
    cudaError_t e = cudaFuncSetAttribute(down, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RadixSmem));
    if (e != cudaSuccess) return e;
    radix_upsweep_kernel<MODE><<<(unsigned)chunks, RS_T, 0, st>>>(ks, count, shift, mask, per, rs.hist, rs.chunk, n, bad);
    radix_chunk_scan_kernel<<<RS_BINS / 32, 1024, 0, st>>>(rs.chunk, chunks, rs.total);
    down<<<(unsigned)tiles, RS_T, sizeof(RadixSmem), st>>>(ks, out, count, shift, mask, per, rs.hist, rs.chunk, rs.total);
    return cudaGetLastError();
}

// Sort by bits [0, bits): the first pass reads `ks` and writes a, later ones
// alternate between a and b; *result = where the keys end.  ks.keys may be b.
cudaError_t radix_sort(int mode, const KeySrc& ks, uint64_t* a, uint64_t* b, int64_t count, int bits,
                       const RadixScratch& rs, int32_t n, int* bad, cudaStream_t st, uint64_t** result) {
    const int passes = std::max(1, (bits + RS_BITS - 1) / RS_BITS);
    int shift = 0;
    for (int p = 0; p < passes; ++p) {
        const int nb = (bits - shift + passes - p - 1) / (passes - p);  // bits dealt evenly
        cudaError_t e;
        if (count == 0) e = cudaSuccess;
        else if (p > 0) e = radix_pass<KEYS_ARRAY>(KeySrc{b, nullptr, nullptr, 0}, a, count, shift, nb, rs, n, bad, st);
        else if (mode == KEYS_DIRECTED) e = radix_pass<KEYS_DIRECTED>(ks, a, count, shift, nb, rs, n, bad, st);
        else if (mode == KEYS_UNDIRECTED) e = radix_pass<KEYS_UNDIRECTED>(ks, a, count, shift, nb, rs, n, bad, st);
        else if (mode == KEYS_BOTH) e = radix_pass<KEYS_BOTH>(ks, a, count, shift, nb, rs, n, bad, st);
        else e = radix_pass<KEYS_ARRAY>(ks, a, count, shift, nb, rs, n, bad, st);
        if (e != cudaSuccess) return e;
        shift += nb;
        std::swap(a, b);
    }
    *result = b;
    return cudaSuccess;
}

// keys sorted by bits [0, bits), in keys or tmp (reordering and hubs-first rows)
cudaError_t radix_sort_u64(uint64_t* keys, uint64_t* tmp, int64_t count, int bits, const RadixScratch& rs,
                           cudaStream_t st, uint64_t** result) {
    return radix_sort(KEYS_ARRAY, KeySrc{keys, nullptr, nullptr, 0}, tmp, keys, count, bits, rs, 0, nullptr, st, result);
}

int grid_for(int64_t count, int threads) {
    int64_t b = div_up(std::max<int64_t>(count, 1), threads);
    return (int)std::min<int64_t>(b, (int64_t)num_sms() * 32);
}

// ------------------------------------------------------------ build steps
__device__ __forceinline__ bool keep_key(uint64_t k, uint64_t prev, bool first, int bits, int dedup, int drop_self) {
    if (drop_self && (k >> bits) == (k & ((1ull << bits) - 1))) return false;
    return !(dedup && !first && prev == k);
}

// first[lo .. hi] = val for each lane (hi < lo: none); a lane's long run, the
// rows without a key between two rows with one, is stored by the whole warp
// (on RMAT-22 one lane at a time took 0.5 ms: half the vertices have no larger
// neighbour).  Warp-uniform.
__device__ __forceinline__ void fill_rows(int32_t* first, int32_t lo, int32_t hi, int32_t val) {
    const bool wide = hi - lo >= 16;
    if (!wide)
        for (int32_t r = lo; r <= hi; ++r) first[r] = val;
    for (unsigned m = __ballot_sync(0xffffffffu, wide); m; m &= m - 1) {
        const int l = __ffs(m) - 1;
        const int32_t a = __shfl_sync(0xffffffffu, lo, l), b = __shfl_sync(0xffffffffu, hi, l),
                      v = __shfl_sync(0xffffffffu, val, l);
        for (int64_t r = (int64_t)a + (threadIdx.x & 31); r <= b; r += 32) first[r] = v;
    }
}

// keys of each tile that stay: no self-loops (drop_self), one of equal keys (dedup)
__global__ void __launch_bounds__(RS_T)
    unique_count_kernel(const uint64_t* __restrict__ keys, int64_t count, int bits, int dedup, int drop_self,
                        uint32_t* __restrict__ tile_cnt) {
    __shared__ uint32_t tmp[33];
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    uint32_t c = 0;
#pragma unroll 8
    for (int i = 0; i < RS_ITEMS; ++i) {
        const int64_t at = base + i * RS_T + threadIdx.x;
        if (at < count) c += keep_key(keys[at], at > 0 ? keys[at - 1] : 0, at == 0, bits, dedup, drop_self) ? 1u : 0u;
    }
    uint32_t total;
    block_excl_scan_u32(c, tmp, &total);
    if (threadIdx.x == 0) tile_cnt[blockIdx.x] = total;
}

// The kept keys in order, and first[r] = kept keys before the first key of a
// row >= r, r in [0, n]: every key, kept or not, whose row is not the previous
// key's writes the rows in between.  tile_off: prefix of the tiles' counts.
__global__ void __launch_bounds__(RS_T)
    unique_write_kernel(const uint64_t* __restrict__ keys, int64_t count, int bits, int dedup, int drop_self,
                        const uint32_t* __restrict__ tile_off, int32_t n, uint64_t* __restrict__ out,
                        int32_t* __restrict__ first) {
    __shared__ uint32_t s_warp[RS_WARPS];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w0 = (int64_t)blockIdx.x * RS_TILE + (int64_t)warp * 32 * RS_ITEMS + lane;
    uint64_t key[RS_ITEMS];
    unsigned keep = 0;  // bit i: this lane's item i stays
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const int64_t at = w0 + i * 32;
        key[i] = at < count ? keys[at] : 0;
    }
    // the key before lane 0's first (the warp's later ones are in lane 31)
    const uint64_t before = lane == 0 && w0 > 0 && w0 < count ? keys[w0 - 1] : 0;
    const uint64_t low = (1ull << bits) - 1;
    unsigned start = 0;  // bit i: this lane's item i is not in the previous key's row
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const int64_t at = w0 + i * 32;
        uint64_t prev = __shfl_up_sync(0xffffffffu, key[i], 1);
        const uint64_t last = i > 0 ? __shfl_sync(0xffffffffu, key[i > 0 ? i - 1 : 0], 31) : before;
        if (lane == 0) prev = last;
        const uint64_t x = key[i] ^ prev;
        const bool self = drop_self && (key[i] >> bits) == (key[i] & low);
        const bool in = at < count;
        keep |= (in && !self && !(dedup && x == 0 && at > 0) ? 1u : 0u) << i;
        start |= (in && ((x >> bits) != 0 || at == 0) ? 1u : 0u) << i;
    }
    const uint32_t wsum = __reduce_add_sync(0xffffffffu, (unsigned)__popc(keep));
    if (lane == 0) s_warp[warp] = wsum;
    __syncthreads();
    uint32_t pos = tile_off[blockIdx.x];
    for (unsigned w = 0; w < warp; ++w) pos += s_warp[w];
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const bool k = (keep >> i) & 1u, s = (start >> i) & 1u;
        const unsigned m = __ballot_sync(0xffffffffu, k);
        const uint32_t p = pos + __popc(m & lanemask_lt());
        if (k) out[p] = key[i];
        pos += __popc(m);
        if (!__any_sync(0xffffffffu, s)) continue;
        uint64_t prev = __shfl_up_sync(0xffffffffu, key[i], 1);
        const uint64_t last = i > 0 ? __shfl_sync(0xffffffffu, key[i > 0 ? i - 1 : 0], 31) : before;
        if (lane == 0) prev = last;
        const int64_t at = w0 + i * 32;
        fill_rows(first, s ? (at > 0 ? (int32_t)(prev >> bits) + 1 : 0) : 0, s ? (int32_t)(key[i] >> bits) : -1,
                  (int32_t)p);
    }
    if (blockIdx.x == gridDim.x - 1) {  // the rows after the last key's
#pragma unroll
        for (int i = 0; i < RS_ITEMS; ++i) {
            const int64_t at = w0 + i * 32;
            const int32_t hi = at == count - 1 ? n : -1;
            fill_rows(first, hi >= 0 ? (int32_t)(key[i] >> bits) + 1 : 0, hi, (int32_t)pos);
        }
    }
}

// first[r] = keys whose lower part is < r (keys ordered by it), r in [0, n]
__global__ void low_rows_kernel(const uint64_t* __restrict__ keys, int64_t mm, int32_t n, int bits,
                                int32_t* __restrict__ first) {
    const uint64_t mask = (1ull << bits) - 1;
    const int64_t lane = threadIdx.x & 31;
    for (int64_t p0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; p0 <= mm; p0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = p0 + lane;  // the loop is warp-uniform
        int32_t lo = 0, hi = -1;
        if (p <= mm) {
            lo = p > 0 ? (int32_t)(keys[p - 1] & mask) + 1 : 0;
            hi = p < mm ? (int32_t)(keys[p] & mask) : n;
        }
        fill_rows(first, lo, hi, (int32_t)p);
    }
}

// col[i] = lower (high = 0) or upper part of key i
__global__ void key_part_kernel(const uint64_t* __restrict__ keys, int64_t mm, int bits, int high,
                                int32_t* __restrict__ col) {
    const uint64_t mask = (1ull << bits) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < mm; i += (int64_t)gridDim.x * blockDim.x)
        col[i] = (int32_t)(high ? keys[i] >> bits : keys[i] & mask);
}

// Columns of a symmetric graph from E and L (see the head of this file).
__global__ void merge_parts_kernel(const uint64_t* __restrict__ E, const uint64_t* __restrict__ L, int64_t mu, int bits,
                                   const int32_t* __restrict__ firstE, const int32_t* __restrict__ firstL,
                                   int32_t* __restrict__ col) {
    const uint64_t mask = (1ull << bits) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < mu; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t e = E[i], l = L[i];
        col[(int64_t)__ldg(firstL + (e >> bits) + 1) + i] = (int32_t)(e & mask);
        col[(int64_t)__ldg(firstE + (l & mask)) + i] = (int32_t)(l >> bits);
    }
}

__global__ void add_rows_kernel(const int32_t* __restrict__ a, const int32_t* __restrict__ b, int64_t count,
                                int32_t* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = a[i] + b[i];
}

struct DegStats {
    unsigned long long sum;
    double sumsq;
    int max;
    int isolated;
};

// A warp per word of the bitmap, lane = vertex.
__global__ void __launch_bounds__(256)
    degree_stats_kernel(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ in_ptr, int32_t n, DegStats* st,
                        uint32_t* __restrict__ isolated) {
    __shared__ unsigned long long s_sum[8];
    __shared__ double s_sq[8];
    __shared__ int s_mx[8], s_iso[8];
    const int64_t words = div_up(n, 32), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long sum = 0;
    double sq = 0;
    int mx = 0, iso = 0;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < words; w += nwarps) {
        const int64_t v = w * 32 + lane;
        int d = 0, din = 1;
        if (v < n) {
            d = row_ptr[v + 1] - row_ptr[v];
            din = in_ptr[v + 1] - in_ptr[v];
        }
        sum += (unsigned long long)d;
        sq += (double)d * d;
        mx = max(mx, d);
        const unsigned m = __ballot_sync(0xffffffffu, din == 0);
        if (lane == 0) {
            isolated[w] = m;
            iso += __popc(m);
        }
    }
    sum = warp_sum(sum);
    sq = warp_sum(sq);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) {
        s_sum[warp] = sum;
        s_sq[warp] = sq;
        s_mx[warp] = mx;
        s_iso[warp] = iso;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int i = 1; i < 8; ++i) {
        sum += s_sum[i];
        sq += s_sq[i];
        mx = max(mx, s_mx[i]);
        iso += s_iso[i];
    }
    atomicAdd(&st->sum, sum);
    atomicAdd(&st->sumsq, sq);
    atomicMax(&st->max, mx);
    atomicAdd(&st->isolated, iso);
}

// One allocation for everything a build needs while it runs.  Large ones by
// cudaMalloc: 1.1 GB from the stream-ordered pool costs 0.9 to 1.1 ms to map and
// 1.5 ms to trim at the next synchronisation.  They go back by cudaFreeAsync,
// in the stream's order (0.6 ms, paid in the stream's next wait): cudaFree, 0.45
// ms, waits for the work of every stream, and a build beside a search on another
// stream waited for that too.  Up to 32 MB, the least the pool maps, from the
// pool: builds that follow one another find it still mapped (117 us by
// cudaMalloc), if it is given back after the last wait of a build (a wait trims
// the pool: 45 us).
struct Arena {
    cudaStream_t st;
    unsigned char* base = nullptr;
    size_t need = 0, used = 0;
    explicit Arena(cudaStream_t s) : st(s) {}
    Arena(const Arena&) = delete;
    Arena& operator=(const Arena&) = delete;
    bool pooled() const { return need <= ((size_t)32 << 20); }
    static size_t pad(size_t bytes) { return (bytes + 255) & ~(size_t)255; }
    template <typename T>
    void want(int64_t count) { need += pad(std::max<size_t>((size_t)count, 1) * sizeof(T)); }
    bool make() {
        const size_t b = std::max<size_t>(need, 256);
        const cudaError_t e = pooled() ? cudaMallocAsync((void**)&base, b, st) : cudaMalloc((void**)&base, b);
        if (e != cudaSuccess) base = nullptr;
        return e == cudaSuccess;
    }
    template <typename T>
    T* take(int64_t count) {
        T* p = reinterpret_cast<T*>(base + used);
        used += pad(std::max<size_t>((size_t)count, 1) * sizeof(T));
        return p;
    }
    void drop() {
        if (base) cudaFreeAsync(base, st);
        base = nullptr;
        need = used = 0;
    }
    ~Arena() { drop(); }
};

enum { ROWS_CSR = 0, ROWS_CSR_CSC = 1, ROWS_SYMMETRIC = 2 };
// A graph's arrays, in one allocation (each cost a build about 120 us to make and free).
struct RowsOut {
    void* block = nullptr;
    int32_t *row_ptr = nullptr, *col = nullptr, *csc_ptr = nullptr, *csc_col = nullptr;
    uint32_t* isolated = nullptr;  // filled in later; a DegStats lies behind it
    int64_t m = 0;
    bool make(int32_t n, int64_t mm, bool csc) {
        const size_t rowb = Arena::pad(((size_t)n + 1) * 4), colb = Arena::pad((size_t)std::max<int64_t>(mm, 1) * 4);
        const size_t isob = Arena::pad((size_t)div_up(n, 32) * 4);
        if (cudaMalloc(&block, (csc ? 2 : 1) * (rowb + colb) + isob + sizeof(DegStats)) != cudaSuccess) return false;
        unsigned char* p = static_cast<unsigned char*>(block);
        row_ptr = reinterpret_cast<int32_t*>(p);
        col = reinterpret_cast<int32_t*>(p += rowb);
        p += colb;
        if (csc) {
            csc_ptr = reinterpret_cast<int32_t*>(p);
            csc_col = reinterpret_cast<int32_t*>(p += rowb);
            p += colb;
        }
        isolated = reinterpret_cast<uint32_t*>(p);
        m = mm;
        return true;
    }
    void drop() {
        cudaFree(block);
        *this = RowsOut();
    }
};

// Device arrays of the rows of `count` keys (shape: ROWS_*; ROWS_SYMMETRIC
// takes KEYS_UNDIRECTED with dedup and drop_self).  With KEYS_ARRAY the key
// array is used as sort space.  `ar`, empty, takes the scratch: nothing uses
// it any more when the call returns.  `out` owns nothing after an error.
bfs_status build_rows(int mode, KeySrc ks, int64_t count, int bits, int dedup, int drop_self, int shape, int32_t n,
                      cudaStream_t st, Arena& ar, RowsOut* out) {
    const int64_t tiles = div_up(std::max<int64_t>(count, 1), RS_TILE);
    ar.want<uint64_t>(count);
    if (mode != KEYS_ARRAY) ar.want<uint64_t>(count);
    ar.want<uint32_t>(RadixScratch::hist_words(count));
    ar.want<uint32_t>(RadixScratch::chunk_words(count));
    ar.want<uint32_t>(RS_BINS);
    ar.want<uint32_t>(tiles);
    ar.want<uint32_t>(2);
    if (shape == ROWS_SYMMETRIC) ar.want<int32_t>(2 * ((int64_t)n + 1));
    if (!ar.make()) {
        cudaGetLastError();
        return fail(BFS_ENOMEM, "build scratch of %lld keys", (long long)count);
    }
    uint64_t* a = ar.take<uint64_t>(count);
    uint64_t* b = mode == KEYS_ARRAY ? const_cast<uint64_t*>(ks.keys) : ar.take<uint64_t>(count);
    RadixScratch rs;
    rs.hist = ar.take<uint32_t>(RadixScratch::hist_words(count));
    rs.chunk = ar.take<uint32_t>(RadixScratch::chunk_words(count));
    rs.total = ar.take<uint32_t>(RS_BINS);
    uint32_t* tile_cnt = ar.take<uint32_t>(tiles);
    uint32_t* d_res = ar.take<uint32_t>(2);  // {keys kept, an id out of range}
    int32_t* firstE = shape == ROWS_SYMMETRIC ? ar.take<int32_t>(2 * ((int64_t)n + 1)) : nullptr;
    int32_t* firstL = firstE ? firstE + n + 1 : nullptr;

    BFS_CUDA(cudaMemsetAsync(d_res, 0, 8, st));
    uint64_t* sorted = a;
    BFS_CUDA(radix_sort(mode, ks, a, b, count, 2 * bits, rs, n, (int*)d_res + 1, st, &sorted));
    if (count > 0) {
        unique_count_kernel<<<(unsigned)tiles, RS_T, 0, st>>>(sorted, count, bits, dedup, drop_self, tile_cnt);
        scan_sums_kernel<<<1, SCAN_THREADS, 0, st>>>(tile_cnt, tiles, d_res);
    }
    uint32_t res[2] = {0, 0};
    BFS_CUDA(cudaMemcpyAsync(res, d_res, 8, cudaMemcpyDeviceToHost, st));
    BFS_CUDA(cudaStreamSynchronize(st));
    if (res[1]) return fail(BFS_EINVAL, "edge list has a vertex id outside [0, %d)", n);
    const int64_t mu = res[0], mm = shape == ROWS_SYMMETRIC ? 2 * mu : mu;
    if (mm > INT32_MAX) return fail(BFS_ERANGE, "graph has %lld directed entries (> 2^31-1)", (long long)mm);
    RowsOut o;
    if (!o.make(n, mm, shape == ROWS_CSR_CSC)) {
        cudaGetLastError();
        return fail(BFS_ENOMEM, "cannot allocate the rows of %lld entries, n=%d", (long long)mm, n);
    }
    uint64_t* E = sorted == a ? b : a;  // kept keys, ordered
    cudaError_t e = cudaSuccess;
    int32_t* rp = shape == ROWS_SYMMETRIC ? firstE : o.row_ptr;
    if (count > 0)
        unique_write_kernel<<<(unsigned)tiles, RS_T, 0, st>>>(sorted, count, bits, dedup, drop_self, tile_cnt, n, E, rp);
    else
        e = cudaMemsetAsync(rp, 0, ((size_t)n + 1) * sizeof(int32_t), st);
    if (shape != ROWS_SYMMETRIC && mm > 0) key_part_kernel<<<grid_for(mm, 256), 256, 0, st>>>(E, mm, bits, 0, o.col);
    if (e == cudaSuccess && shape != ROWS_CSR) {
        // L: E sorted, stable, by the lower part alone.  The merge below reads
        // both, and the column array of 2 * mu entries is exactly one more
        // key array to sort through, as long as L does not end in it; a
        // directed graph is done with E.
        uint64_t *x = sorted, *y = E, *L = nullptr;
        if (shape == ROWS_SYMMETRIC) {
            y = reinterpret_cast<uint64_t*>(o.col);
            if (((bits + RS_BITS - 1) / RS_BITS) % 2 == 0) std::swap(x, y);
        }
        e = radix_sort(KEYS_ARRAY, KeySrc{E, nullptr, nullptr, 0}, x, y, mu, bits, rs, n, nullptr, st, &L);
        int32_t* fl = shape == ROWS_SYMMETRIC ? firstL : o.csc_ptr;
        if (e == cudaSuccess) {
            low_rows_kernel<<<grid_for(mu + 1, 256), 256, 0, st>>>(L, mu, n, bits, fl);
            if (shape == ROWS_SYMMETRIC) {
                if (mu > 0) merge_parts_kernel<<<grid_for(mu, 256), 256, 0, st>>>(E, L, mu, bits, firstE, firstL, o.col);
                add_rows_kernel<<<grid_for(n + 1ll, 256), 256, 0, st>>>(firstE, firstL, n + 1ll, o.row_ptr);
            } else if (mu > 0) {
                key_part_kernel<<<grid_for(mu, 256), 256, 0, st>>>(L, mu, bits, 1, o.csc_col);
            }
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        o.drop();
        return cuda_fail(e, "build rows");
    }
    *out = o;
    return BFS_OK;
}

// ------------------------------------------------------------ RCM
// Reverse Cuthill-McKee numbering (Section 7.1), computed level by level.
// rank(v) = position of v in (degree, id) order.  A component starts at its
// lowest-ranked vertex; the vertices first reached from the level whose
// positions are [lb, le) form the next level, ordered by (lowest position of
// a neighbour in [lb, le), rank) -- the order in which a FIFO queue numbering
// each dequeued vertex's unnumbered neighbours in rank order numbers them.

constexpr int RCM_SMALL_SORT = 4096;       // levels up to this size are sorted by one CTA
constexpr int64_t RCM_FIND_CHUNK = 1 << 20;  // rank-order window scanned per start search

// key = degree << bits | v
__global__ void rcm_rank_keys_kernel(const int32_t* row_ptr, int32_t n, int bits, uint64_t* keys) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        keys[v] = ((uint64_t)(uint32_t)(row_ptr[v + 1] - row_ptr[v]) << bits) | (uint64_t)v;
}

// byrank[i] = vertex of rank i, rank[v]; pos = -1, minpos = INT32_MAX; the
// degree-0 vertices (the lowest ranks, each its own component) are numbered
// at once in rank order; *n0 = their count
__global__ void rcm_init_kernel(const uint64_t* sorted, const int32_t* row_ptr, int32_t n, int bits, int32_t* byrank,
                                int32_t* rank, int32_t* pos, int32_t* order, int32_t* minpos, int* n0) {
    const uint64_t mask = (1ull << bits) - 1;
    int cnt = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = (int32_t)(sorted[i] & mask);
        byrank[i] = v;
        rank[v] = (int32_t)i;
        minpos[v] = INT32_MAX;
        const bool iso = row_ptr[v + 1] == row_ptr[v];
        pos[v] = iso ? (int32_t)i : -1;
        if (iso) order[i] = v;
        cnt += iso ? 1 : 0;
    }
    cnt = __reduce_add_sync(0xffffffffu, (unsigned)cnt);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(n0, cnt);
}

// lowest rank index in [lo, hi) whose vertex is not numbered yet
__global__ void rcm_find_start_kernel(const int32_t* byrank, const int32_t* pos, int64_t lo, int64_t hi, int* found) {
    for (int64_t i = lo + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < hi; i += (int64_t)gridDim.x * blockDim.x)
        if (pos[byrank[i]] < 0) atomicMin(found, (int)i);
}

__global__ void rcm_place_start_kernel(const int32_t* byrank, const int* found, int32_t next, int32_t* pos,
                                       int32_t* order) {
    const int32_t s = byrank[*found];
    pos[s] = next;
    order[next] = s;
}

// one warp per vertex of the level [lb, le): every unnumbered neighbour v
// takes the lowest such position as its key and joins the next level once
__global__ void rcm_expand_kernel(const int32_t* row_ptr, const int32_t* col, const int32_t* order, int32_t lb,
                                  int32_t le, const int32_t* pos, int32_t* minpos, uint32_t* seen, int32_t* list,
                                  int* cnt) {
    const unsigned lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = lb + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); p < le; p += nwarps) {
        const int32_t u = order[p];
        const int32_t b = row_ptr[u], e = row_ptr[u + 1];
        for (int32_t j = b + (int32_t)lane; j < e; j += 32) {
            const int32_t v = col[j];
            if (pos[v] >= 0) continue;
            atomicMin(minpos + v, (int32_t)p);
            const uint32_t bit = 1u << (v & 31);
            if (!(atomicOr(seen + (v >> 5), bit) & bit)) list[atomicAdd(cnt, 1)] = v;
        }
    }
}

// key = minpos << bits | rank
__global__ void rcm_level_keys_kernel(const int32_t* list, int32_t cnt, const int32_t* minpos, const int32_t* rank,
                                      int bits, uint64_t* keys) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = list[i];
        keys[i] = ((uint64_t)(uint32_t)minpos[v] << bits) | (uint64_t)(uint32_t)rank[v];
    }
}

// ascending bitonic sort of up to RCM_SMALL_SORT keys in one CTA
__global__ void rcm_small_sort_kernel(uint64_t* keys, int32_t cnt) {
    __shared__ uint64_t s[RCM_SMALL_SORT];
    for (int i = threadIdx.x; i < RCM_SMALL_SORT; i += blockDim.x) s[i] = i < cnt ? keys[i] : ~0ull;
    __syncthreads();
    for (int k = 2; k <= RCM_SMALL_SORT; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < RCM_SMALL_SORT; i += blockDim.x) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const bool up = (i & k) == 0;
                    const uint64_t a = s[i], c = s[ixj];
                    if ((a > c) == up) {
                        s[i] = c;
                        s[ixj] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) keys[i] = s[i];
}

__global__ void rcm_assign_kernel(const uint64_t* sorted, int32_t cnt, int bits, const int32_t* byrank, int32_t next,
                                  int32_t* pos, int32_t* order) {
    const uint64_t mask = (1ull << bits) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = byrank[sorted[i] & mask];
        pos[v] = next + (int32_t)i;
        order[next + i] = v;
    }
}

__global__ void rcm_newid_identity_kernel(int32_t n, int32_t* newid) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        newid[v] = (int32_t)v;
}

__global__ void rcm_newid_kernel(const int32_t* pos, int32_t n, int32_t* newid) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        newid[v] = n - 1 - pos[v];
}

// (newid[s] << bits) | newid[d] for every CSR entry, one warp per row
__global__ void relabel_keys_kernel(const int32_t* row_ptr, const int32_t* col, int32_t n, const int32_t* newid,
                                    int bits, uint64_t* keys) {
    const unsigned lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += nwarps) {
        const uint64_t hi = (uint64_t)(uint32_t)newid[v] << bits;
        for (int32_t j = row_ptr[v] + (int32_t)lane; j < row_ptr[v + 1]; j += 32)
            keys[j] = hi | (uint64_t)(uint32_t)newid[col[j]];
    }
}

template <typename T>
bfs_status read_scalar(const T* d, T* h, cudaStream_t st) {
    BFS_CUDA(cudaMemcpyAsync(h, d, sizeof(T), cudaMemcpyDeviceToHost, st));
    BFS_CUDA(cudaStreamSynchronize(st));
    return BFS_OK;
}

// newid (device [n]) of the Reverse Cuthill-McKee numbering of a symmetric CSR
bfs_status rcm_newid(const int32_t* row_ptr, const int32_t* col, int32_t n, int bits, cudaStream_t st,
                     int32_t* newid) {
    Scratch sc(st);
    uint64_t *keys, *tmp;
    int32_t *byrank, *rank, *pos, *order, *minpos, *list;
    uint32_t* seen;
    int *d_n0, *d_cnt, *d_found;
    RadixScratch rs;  // of the rank sort, and of every level's
    const int64_t words = div_up(n, 32);
    if (sc.alloc(&keys, n) || sc.alloc(&tmp, n) || sc.alloc(&byrank, n) || sc.alloc(&rank, n) || sc.alloc(&pos, n) ||
        sc.alloc(&order, n) || sc.alloc(&minpos, n) || sc.alloc(&list, n) || sc.alloc(&seen, words) ||
        sc.alloc(&d_n0, 1) || sc.alloc(&d_cnt, 1) || sc.alloc(&d_found, 1) || rs.alloc(sc, n)) {
        cudaGetLastError();
        return fail(BFS_ENOMEM, "RCM scratch for n=%d", n);
    }
    rcm_rank_keys_kernel<<<grid_for(n, 256), 256, 0, st>>>(row_ptr, n, bits, keys);
    uint64_t* sorted;
    BFS_CUDA(radix_sort_u64(keys, tmp, n, bits + 32, rs, st, &sorted));
    BFS_CUDA(cudaMemsetAsync(d_n0, 0, 4, st));
    BFS_CUDA(cudaMemsetAsync(seen, 0, words * 4, st));
    rcm_init_kernel<<<grid_for(n, 256), 256, 0, st>>>(sorted, row_ptr, n, bits, byrank, rank, pos, order, minpos, d_n0);
    int n0 = 0;
    bfs_status s = read_scalar(d_n0, &n0, st);
    if (s != BFS_OK) return s;
    int32_t next = n0;
    int64_t cursor = n0;
    while (cursor < n) {
        const int64_t hi = std::min<int64_t>(n, cursor + RCM_FIND_CHUNK);
        const int none = INT32_MAX;
        BFS_CUDA(cudaMemcpyAsync(d_found, &none, 4, cudaMemcpyHostToDevice, st));
        rcm_find_start_kernel<<<grid_for(hi - cursor, 256), 256, 0, st>>>(byrank, pos, cursor, hi, d_found);
        int found = none;
        if ((s = read_scalar(d_found, &found, st)) != BFS_OK) return s;
        if (found == none) {
            cursor = hi;
            continue;
        }
        cursor = (int64_t)found + 1;
        rcm_place_start_kernel<<<1, 1, 0, st>>>(byrank, d_found, next, pos, order);
        int32_t lb = next, le = next + 1;
        next += 1;
        for (;;) {
            BFS_CUDA(cudaMemsetAsync(d_cnt, 0, 4, st));
            rcm_expand_kernel<<<grid_for((int64_t)(le - lb) * 32, 256), 256, 0, st>>>(row_ptr, col, order, lb, le, pos,
                                                                                     minpos, seen, list, d_cnt);
            int cnt = 0;
            if ((s = read_scalar(d_cnt, &cnt, st)) != BFS_OK) return s;
            if (cnt == 0) break;
            if (next + (int64_t)cnt > n) return fail(BFS_EVALIDATE, "RCM numbered more than n vertices");
            rcm_level_keys_kernel<<<grid_for(cnt, 256), 256, 0, st>>>(list, cnt, minpos, rank, bits, keys);
            uint64_t* lsorted = keys;
            if (cnt <= RCM_SMALL_SORT) {
                rcm_small_sort_kernel<<<1, 1024, 0, st>>>(keys, cnt);
            } else {
                BFS_CUDA(radix_sort_u64(keys, tmp, cnt, 2 * bits, rs, st, &lsorted));
            }
            rcm_assign_kernel<<<grid_for(cnt, 256), 256, 0, st>>>(lsorted, cnt, bits, byrank, next, pos, order);
            lb = le;
            le = next + cnt;
            next += cnt;
        }
    }
    if (next != n) return fail(BFS_EVALIDATE, "RCM numbered %d of %d vertices", next, n);
    rcm_newid_kernel<<<grid_for(n, 256), 256, 0, st>>>(pos, n, newid);
    BFS_CUDA(cudaGetLastError());
    BFS_CUDA(cudaStreamSynchronize(st));
    return BFS_OK;
}

// ------------------------------------------------------------ hubs-first rows
// key = (INT32_MAX - degree) << bits | v: ascending = degree descending, id ascending
__global__ void hub_rank_keys_kernel(const int32_t* row_ptr, int32_t n, int bits, uint64_t* keys) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        keys[v] = ((uint64_t)(uint32_t)(INT32_MAX - (row_ptr[v + 1] - row_ptr[v])) << bits) | (uint64_t)v;
}

__global__ void rank_of_kernel(const uint64_t* sorted, int32_t n, int bits, int32_t* byrank, int32_t* rank) {
    const uint64_t mask = (1ull << bits) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = (int32_t)(sorted[i] & mask);
        byrank[i] = v;
        rank[v] = (int32_t)i;
    }
}

// (row << bits) | rank of the entry, one warp per row
__global__ void hub_row_keys_kernel(const int32_t* ptr, const int32_t* col, int32_t n, const int32_t* rank, int bits,
                                    uint64_t* keys) {
    const unsigned lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += nwarps)
        for (int32_t j = ptr[v] + (int32_t)lane; j < ptr[v + 1]; j += 32)
            keys[j] = ((uint64_t)v << bits) | (uint64_t)(uint32_t)rank[col[j]];
}

__global__ void hub_col_kernel(const uint64_t* sorted, int64_t m, int bits, const int32_t* byrank, int32_t* col) {
    const uint64_t mask = (1ull << bits) - 1;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x)
        col[j] = byrank[sorted[j] & mask];
}

// Replace the d-major column array by one whose rows are ordered by the
// entries' out-degree, highest first (ties by id); row bounds are unchanged.
bfs_status pull_hubs_first(bfs_graph* g, int bits, cudaStream_t st) {
    const int32_t n = g->n;
    const int64_t m = g->m;
    Scratch sc(st);
    uint64_t *rk, *rt, *keys, *tmp;
    int32_t *byrank, *rank, *col;
    RadixScratch rs;
    if (sc.alloc(&rk, n) || sc.alloc(&rt, n) || sc.alloc(&byrank, n) || sc.alloc(&rank, n) || sc.alloc(&keys, m) ||
        sc.alloc(&tmp, m) || rs.alloc(sc, std::max<int64_t>(n, m))) {
        cudaGetLastError();
        return fail(BFS_ENOMEM, "hubs-first scratch");
    }
    // a directed graph's d-major columns are its own and are reordered in place
    const bool own = g->csc_col != g->col;
    if (own) {
        col = g->csc_col;
    } else if (cudaMalloc(&g->hub_col, (size_t)std::max<int64_t>(m, 1) * sizeof(int32_t)) != cudaSuccess) {
        cudaGetLastError();
        g->hub_col = nullptr;
        return fail(BFS_ENOMEM, "hubs-first column array of %lld entries", (long long)m);
    } else {
        col = g->hub_col;
    }
    hub_rank_keys_kernel<<<grid_for(n, 256), 256, 0, st>>>(g->row_ptr, n, bits, rk);
    uint64_t* ranked;
    cudaError_t e = radix_sort_u64(rk, rt, n, bits + 32, rs, st, &ranked);
    if (e == cudaSuccess) {
        rank_of_kernel<<<grid_for(n, 256), 256, 0, st>>>(ranked, n, bits, byrank, rank);
        hub_row_keys_kernel<<<grid_for((int64_t)n * 32, 256), 256, 0, st>>>(g->csc_ptr, g->csc_col, n, rank, bits, keys);
        uint64_t* ks;
        e = radix_sort_u64(keys, tmp, m, 2 * bits, rs, st, &ks);
        if (e == cudaSuccess) {
            hub_col_kernel<<<grid_for(m, 256), 256, 0, st>>>(ks, m, bits, byrank, col);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "hubs-first rows");
    g->csc_col = col;
    return BFS_OK;
}

// The graph's arrays are `r`'s from now on.
void take_rows(bfs_graph* g, const RowsOut& r, bool sym) {
    cudaFree(g->rows);
    g->rows = r.block;
    g->row_ptr = r.row_ptr;
    g->col = r.col;
    g->csc_ptr = sym ? r.row_ptr : r.csc_ptr;
    g->csc_col = sym ? r.col : r.csc_col;
    g->isolated = r.isolated;
    g->m = r.m;
}

// Renumber a built symmetric graph in RCM order: g->perm, then the CSR again
bfs_status rcm_reorder(bfs_graph* g, int bits, cudaStream_t st) {
    if (cudaMalloc(&g->perm, (size_t)g->n * sizeof(int32_t)) != cudaSuccess) {
        cudaGetLastError();
        return fail(BFS_ENOMEM, "permutation of n=%d", g->n);
    }
    bfs_status s = rcm_newid(g->row_ptr, g->col, g->n, bits, st, g->perm);
    if (s != BFS_OK) return s;
    Scratch sc(st);
    uint64_t* keys;
    if (sc.alloc(&keys, g->m) != cudaSuccess) {
        cudaGetLastError();
        return fail(BFS_ENOMEM, "relabel keys");
    }
    relabel_keys_kernel<<<grid_for((int64_t)g->n * 32, 256), 256, 0, st>>>(g->row_ptr, g->col, g->n, g->perm, bits, keys);
    BFS_CUDA(cudaGetLastError());
    RowsOut r;
    Arena ar(st);
    s = build_rows(KEYS_ARRAY, KeySrc{keys, nullptr, nullptr, bits}, g->m, bits, 0, 0, ROWS_CSR, g->n, st, ar, &r);
    if (s != BFS_OK) return s;
    take_rows(g, r, true);
    return BFS_OK;
}

}  // namespace

}  // namespace bfsgb

using namespace bfsgb;

extern "C" bfs_status bfs_build_graph(int32_t n, int64_t m, const int32_t* src, const int32_t* dst, uint32_t flags,
                                      void* cuda_stream, bfs_graph** out) {
    if (!out) return fail(BFS_EINVAL, "out is NULL");
    *out = nullptr;
    if (n <= 0) return fail(BFS_EINVAL, "n must be positive (got %d)", n);
    if (m < 0) return fail(BFS_EINVAL, "m must be >= 0");
    if (m > 0 && (!src || !dst)) return fail(BFS_EINVAL, "src/dst is NULL");
    int sym = (flags & BFS_SYMMETRIZE) != 0;
    if ((flags & BFS_REORDER_RCM) && !sym) return fail(BFS_EINVAL, "BFS_REORDER_RCM needs BFS_SYMMETRIZE");
    int64_t count = sym ? 2 * m : m;
    if (count > INT32_MAX) return fail(BFS_ERANGE, "%lld directed entries before deduplication (> 2^31-1)", (long long)count);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    int bits = 1;
    while ((1ll << bits) < (int64_t)n) ++bits;

    const int dedup = (flags & BFS_DEDUP) != 0, drop_self = (flags & BFS_DROP_SELF) != 0;
    KeySrc ks{nullptr, src, dst, bits};
    Arena in(st);  // copies of an edge list in host memory
    const bool host_src = m > 0 && !is_device_ptr(src), host_dst = m > 0 && !is_device_ptr(dst);
    if (host_src || host_dst) {
        if (host_src) in.want<int32_t>(m);
        if (host_dst) in.want<int32_t>(m);
        if (!in.make()) {
            cudaGetLastError();
            return fail(BFS_ENOMEM, "edge list of %lld entries", (long long)m);
        }
        if (host_src) {
            int32_t* p = in.take<int32_t>(m);
            BFS_CUDA(cudaMemcpyAsync(p, src, m * 4, cudaMemcpyHostToDevice, st));
            ks.src = p;
        }
        if (host_dst) {
            int32_t* p = in.take<int32_t>(m);
            BFS_CUDA(cudaMemcpyAsync(p, dst, m * 4, cudaMemcpyHostToDevice, st));
            ks.dst = p;
        }
    }

    bfs_graph* g = new (std::nothrow) bfs_graph();
    if (!g) return fail(BFS_ENOMEM, "host allocation");
    g->n = n;
    g->device = device_id();
    // one sort of every edge where both directions hold the same entries;
    // a kept self-loop of a symmetric graph is two entries, repeats stay
    const bool once = sym && dedup && drop_self;
    RowsOut r;
    Arena ar(st);
    bfs_status s = build_rows(once ? KEYS_UNDIRECTED : sym ? KEYS_BOTH : KEYS_DIRECTED, ks, once ? m : count, bits, dedup,
                              drop_self, once ? ROWS_SYMMETRIC : sym ? ROWS_CSR : ROWS_CSR_CSC, n, st, ar, &r);
    if (s != BFS_OK) {
        delete g;
        return s;
    }
    take_rows(g, r, sym);
    g->symmetric = sym;
    const bool more = (flags & (BFS_REORDER_RCM | BFS_PULL_HUBS_FIRST)) != 0;
    if (!ar.pooled()) {
        ar.drop();
        // back before the steps below take theirs (they wait too)
        const cudaError_t e = more ? cudaStreamSynchronize(st) : cudaSuccess;
        if (e != cudaSuccess) {
            bfs_free_graph(g);
            return cuda_fail(e, "build scratch");
        }
    } else if (more) {
        ar.drop();
    }
    if (sym && (flags & BFS_REORDER_RCM)) {
        bfs_status sr = rcm_reorder(g, bits, st);
        if (sr != BFS_OK) {
            bfs_free_graph(g);
            return sr;
        }
    }
    if (flags & BFS_PULL_HUBS_FIRST) {
        bfs_status sh = pull_hubs_first(g, bits, st);
        if (sh != BFS_OK) {
            bfs_free_graph(g);
            return sh;
        }
    }
    int64_t words = div_up(n, 32);
    DegStats h{};
    // behind the bitmap, see RowsOut
    DegStats* d_st = reinterpret_cast<DegStats*>((unsigned char*)g->isolated + Arena::pad((size_t)words * 4));
    cudaError_t e = cudaMemsetAsync(d_st, 0, sizeof(DegStats), st);
    degree_stats_kernel<<<std::min(grid_for(words * 32, 256), num_sms() * 8), 256, 0, st>>>(g->row_ptr, g->csc_ptr, n, d_st, g->isolated);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d_st, sizeof(DegStats), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        bfs_free_graph(g);
        return cuda_fail(e, "degree statistics");
    }
    g->deg_max = h.max;
    g->deg_mean = (double)h.sum / n;
    g->deg_var = h.sumsq / n - g->deg_mean * g->deg_mean;
    g->n_isolated = h.isolated;
    *out = g;
    return BFS_OK;
}

extern "C" bfs_status bfs_graph_info(const bfs_graph* g, bfs_graph_stats* out) {
    if (!g || !out) return fail(BFS_EINVAL, "null argument");
    out->n = g->n;
    out->m = g->m;
    out->symmetric = g->symmetric;
    out->n_isolated = g->n_isolated;
    out->deg_max = g->deg_max;
    out->deg_mean = g->deg_mean;
    out->deg_var = g->deg_var;
    return BFS_OK;
}

extern "C" bfs_status bfs_graph_csr(const bfs_graph* g, int32_t csc, int32_t* row_ptr, int32_t* col, void* cuda_stream) {
    if (!g) return fail(BFS_EINVAL, "graph is NULL");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int32_t* rp = csc ? g->csc_ptr : g->row_ptr;
    const int32_t* cl = csc ? g->csc_col : g->col;
    if (row_ptr) BFS_CUDA(cudaMemcpyAsync(row_ptr, rp, ((int64_t)g->n + 1) * 4, cudaMemcpyDefault, st));
    if (col && g->m > 0) BFS_CUDA(cudaMemcpyAsync(col, cl, g->m * 4, cudaMemcpyDefault, st));
    if ((row_ptr && !is_device_ptr(row_ptr)) || (col && !is_device_ptr(col))) BFS_CUDA(cudaStreamSynchronize(st));
    return BFS_OK;
}

extern "C" void bfs_free_graph(bfs_graph* g) {
    if (!g) return;
    free_ws1(g->ws1);
    free_wsms(g->wsms);
    free_wsms(g->wsmix);
    cudaFree(g->rows);
    cudaFree(g->hub_col);
    cudaFree(g->perm);
    cudaFree(g->cc_scratch);
    delete g;
}

extern "C" bfs_status bfs_graph_permutation(const bfs_graph* g, int32_t* newid, void* cuda_stream) {
    if (!g || !newid) return fail(BFS_EINVAL, "null argument");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const bool host = !is_device_ptr(newid);
    if (g->perm) {
        BFS_CUDA(cudaMemcpyAsync(newid, g->perm, (size_t)g->n * 4, host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st));
        if (host) BFS_CUDA(cudaStreamSynchronize(st));
        return BFS_OK;
    }
    if (host) {
        for (int32_t v = 0; v < g->n; ++v) newid[v] = v;
        return BFS_OK;
    }
    rcm_newid_identity_kernel<<<grid_for(g->n, 256), 256, 0, st>>>(g->n, newid);
    BFS_CUDA(cudaGetLastError());
    return BFS_OK;
}
