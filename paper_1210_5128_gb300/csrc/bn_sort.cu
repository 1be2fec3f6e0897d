// bn_sort.cu -- per-node ranking of the table entries for the scan.
//
// Every entry (i, rho) gets spos[i][rho]: its position when node i's entries are ordered
// by score descending, ties by rank ascending.  spos is unique within a node and
// "smaller spos" means "higher score, or equal score and lower rank", so the order-score
// scan's (max score, lowest rank) reduction becomes a single unsigned min over spos.
// srank[i][p] is the inverse (the rank at sorted position p), sset[i][p] its parent nodes.
//
// The order is total (no two entries of a node share score and rank), so no pass has to be
// stable.  A node's entries are split by sampled splitters -- (score, rank) pairs, so ties
// split too -- into buckets of about 1,024, and a block sorts each bucket in shared memory
// and writes all three arrays: the keys are read twice and the pairs written and read once,
// against nine read-and-scatter passes of a byte-digit radix sort.  Measured at n = 60,
// k = 4 (60 times 489,406 entries): radix sort and set words 5.43 ms, buckets 0.91 ms
// (splitters 0.07, bucket of every entry 0.11, scatter 0.15, sorting and writing 0.57);
// HBM would allow about 0.25 ms.  What made the difference between that and a first 1.73 ms:
// the count pass looks a key's cell up and searches the few splitters there (0.30 with a
// binary search of all), the scatter orders a tile in shared memory and writes runs (0.51
// entry by entry), the sort takes a bucket's range from its splitters and 2,048 evenly cut
// sub-buckets (0.84 with a reduction and 256 to 512 of them).  The sort is bound by its
// instructions, of which the fixed work of a block is a large part.  Tables of more than
// BS_MAX_BUCKETS * 2,048 sets a node keep the radix sort: their buckets would outgrow a
// block's shared memory.
#include <algorithm>
#include <vector>

#include "bn_table.cuh"

namespace bn {

static constexpr int RS_THREADS = 256;
static constexpr int RS_ROUNDS = 16;
static constexpr int RS_TILE = RS_THREADS * RS_ROUNDS;   // 4096 elements per tile

struct RsPass {
    const uint64_t* kin;
    const uint32_t* vin;
    uint64_t* kout;
    uint32_t* vout;
    int64_t N;
    int shift;          // digit = (key >> shift) & 255, or the node (value / S) when < 0
    int64_t S;
    int node0;          // first node of this batch
    uint32_t* counts;   // [256][T]
    uint32_t* totals;   // [256]
    int T;
};

__device__ __forceinline__ int rs_digit(const RsPass& P, uint64_t k, uint32_t v)
{
    return P.shift >= 0 ? (int)((k >> P.shift) & 255ull) : (int)(v / (uint32_t)P.S);
}

__global__ void k_rs_init(const int64_t* __restrict__ keys, int64_t Sp, int64_t S, int node0, int64_t N,
                          uint64_t* __restrict__ kout, uint32_t* __restrict__ vout)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= N) return;
    const int64_t i = g / S, r = g - i * S;
    const uint64_t u = (uint64_t)keys[(node0 + i) * Sp + r] ^ 0x8000000000000000ull;  // ascending as unsigned
    kout[g] = ~u;                                                                        // descending score
    vout[g] = (uint32_t)g;
}

__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(RsPass P)
{
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const int64_t e = base + (int64_t)r * RS_THREADS + threadIdx.x;
        if (e < P.N) atomicAdd(&h[rs_digit(P, P.kin[e], P.vin[e])], 1u);
    }
    __syncthreads();
    P.counts[(size_t)threadIdx.x * P.T + blockIdx.x] = h[threadIdx.x];
}

// exclusive scan of counts[d][0..T) for one digit d per block; totals[d] = the sum
__global__ void __launch_bounds__(1024) k_rs_scan(uint32_t* __restrict__ counts, int T, uint32_t* __restrict__ totals)
{
    __shared__ uint32_t part[1024];
    uint32_t* c = counts + (size_t)blockIdx.x * T;
    const int per = (T + 1023) / 1024;
    const int b = threadIdx.x * per, e = min(T, b + per);
    uint32_t s = 0;
    for (int j = b; j < e; ++j) s += c[j];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        uint32_t v = threadIdx.x >= off ? part[threadIdx.x - off] : 0u;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    uint32_t run = part[threadIdx.x] - s;   // exclusive prefix of this thread's range
    for (int j = b; j < e; ++j) {
        const uint32_t v = c[j];
        c[j] = run;
        run += v;
    }
    if (threadIdx.x == 1023) totals[blockIdx.x] = part[1023];
}

// stable scatter of one tile: round-major order (element base + r*256 + t), ranks
// within a round from warp match groups plus the earlier warps' counts of the digit
__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(RsPass P)
{
    __shared__ uint32_t s_run[256];
    __shared__ uint32_t s_w[RS_THREADS / 32][256];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        // digit base = exclusive scan of totals (256 values, Hillis-Steele in shared)
        __shared__ uint32_t t[256];
        const uint32_t mine = P.totals[threadIdx.x];
        t[threadIdx.x] = mine;
        __syncthreads();
        for (int off = 1; off < 256; off <<= 1) {
            uint32_t v = threadIdx.x >= off ? t[threadIdx.x - off] : 0u;
            __syncthreads();
            t[threadIdx.x] += v;
            __syncthreads();
        }
        s_run[threadIdx.x] = t[threadIdx.x] - mine + P.counts[(size_t)threadIdx.x * P.T + blockIdx.x];
    }
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    const unsigned lt = (1u << lane) - 1u;
    for (int r = 0; r < RS_ROUNDS; ++r) {
        for (int j = threadIdx.x; j < (RS_THREADS / 32) * 256; j += RS_THREADS) (&s_w[0][0])[j] = 0u;
        __syncthreads();
        const int64_t e = base + (int64_t)r * RS_THREADS + threadIdx.x;
        const bool valid = e < P.N;
        uint64_t k = 0;
        uint32_t v = 0;
        int d = 256;                                  // sentinel for the tail
        if (valid) {
            k = P.kin[e];
            v = P.vin[e];
            d = rs_digit(P, k, v);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t lrank = (uint32_t)__popc(peers & lt);
        if (valid && lrank == 0) s_w[warp][d] = (uint32_t)__popc(peers);
        __syncthreads();
        if (valid) {
            uint32_t off = s_run[d] + lrank;
            for (int w = 0; w < warp; ++w) off += s_w[w][d];
            P.kout[off] = k;
            P.vout[off] = v;
        }
        __syncthreads();
        {
            uint32_t add = 0;
            for (int w = 0; w < RS_THREADS / 32; ++w) add += s_w[w][threadIdx.x];
            s_run[threadIdx.x] += add;
        }
        __syncthreads();
    }
}

__global__ void k_rs_finish(const uint32_t* __restrict__ vals, int64_t N, int64_t S, int64_t Sp, int node0,
                            uint32_t* __restrict__ srank, uint32_t* __restrict__ spos)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= N) return;
    const int64_t i = g / S, p = g - i * S;      // sorted by node first: position p of node i
    const uint32_t v = vals[g];
    const int64_t r = (int64_t)v - i * S;
    srank[(node0 + i) * Sp + p] = (uint32_t)r;
    spos[(node0 + i) * Sp + r] = (uint32_t)p;
}

// ---------------------------------------------------------------------------------
// bucket sort
// ---------------------------------------------------------------------------------
static constexpr int BS_MAX_BUCKETS = 1024;
static constexpr int BS_AVG = 1024;                  // entries a bucket on average (2,048 above 1 M sets)
static constexpr int BS_CAP = 4096;                  // entries a block sorts in shared memory
static constexpr int BS_THREADS = 512;
static constexpr int BS_PER = BS_CAP / BS_THREADS;
static constexpr int BS_NSUB = 2048;                 // sub-buckets of a bucket
static constexpr uint32_t BS_CROWD = 128;            // entries of four sub-buckets above which a block sorts its bucket
                                                     // by a network, which takes as long as that many compares an entry
static constexpr int BS_CELLS = 2048;                // cells of a node's key range, for the count pass
static constexpr int BS_TILE = 8192;                 // entries of a partition tile
static constexpr int BS_SAMPLES = 8192;              // at most, of a node

// ascending <=> score descending
__device__ __forceinline__ uint64_t bs_key(int64_t key) { return (uint64_t)key ^ 0x7FFFFFFFFFFFFFFFull; }
__device__ __forceinline__ bool bs_less(uint64_t xa, uint32_t ra, uint64_t xb, uint32_t rb)
{
    return xa < xb || (xa == xb && ra < rb);
}

// Monotone map of the keys of [lo, hi] to N cells of equal width (keys outside: the first or
// the last cell).  The float's error only moves the cells' ends: 0.999998 keeps the last
// key below cell N.
struct BsCells {
    uint64_t lo, hi, scale;
    int sh;
    __device__ __forceinline__ BsCells(uint64_t lo_, uint64_t hi_, int N) : lo(lo_), hi(hi_)
    {
        const uint64_t range = hi - lo;
        sh = max(0, 32 - __clzll((long long)range));
        scale = __float2ull_rd((float)N * 4294967296.0f / ((float)(uint32_t)(range >> sh) + 1.0f) * 0.999998f);
    }
    __device__ __forceinline__ uint32_t operator()(uint64_t x) const
    {
        const uint64_t y = min(max(x, lo), hi);
        return (uint32_t)(((y - lo) >> sh) * scale >> 32);
    }
};

struct BsArgs {
    const int64_t* keys;      // [n][Sp]
    const uint64_t* pst;
    int64_t S, Sp;
    int node0;                // first node of this batch
    int NB, tiles;            // buckets and tiles a node
    int M;                    // samples a node (a power of two, at least 2 NB)
    uint64_t* split_x;        // [nb][NB] splitters; bucket b holds [splitter b - 1, splitter b)
    uint32_t* split_r;
    uint32_t* cells;          // [nb][BS_CELLS] splitters below a cell | splitters below the next << 16
    uint32_t* counts;         // [nb][NB] entries, then [nb][NB] first entries of the buckets
    uint32_t* tile_base;      // [nb][tiles][NB] the tile's first entry within each bucket
    uint16_t* bid;            // [nb][S] bucket of each entry
    uint64_t* bx;             // [nb][S] the entries by bucket
    uint32_t* br;
    uint32_t* srank;          // [n][Sp]
    uint32_t* spos;           // [n][Sp]
    uint32_t* sset;           // [n][Ssp] or null
    int64_t Ssp;
};

// splitters of one node a block: a stratified pseudo-random sample, sorted in shared memory
// (bitonic), every (M / NB)-th element.  The result of the sort does not depend on them.
__global__ void __launch_bounds__(1024) k_bs_split(BsArgs A)
{
    extern __shared__ __align__(16) uint8_t bs_sm[];
    uint64_t* x = (uint64_t*)bs_sm;
    uint32_t* r = (uint32_t*)(x + A.M);
    const int i = blockIdx.x;
    const int64_t* K = A.keys + (size_t)(A.node0 + i) * A.Sp;
    for (int j = threadIdx.x; j < A.M; j += blockDim.x) {
        const int64_t lo = A.S * j / A.M, hi = A.S * (j + 1) / A.M;      // hi > lo: S >= M
        uint32_t h = (uint32_t)j * 0x9E3779B9u;
        h ^= h >> 15;
        h *= 0x85EBCA6Bu;
        h ^= h >> 13;
        const int64_t e = lo + (int64_t)(h % (uint32_t)(hi - lo));
        x[j] = bs_key(K[e]);
        r[j] = (uint32_t)e;
    }
    for (int len = 2; len <= A.M; len <<= 1)
        for (int d = len >> 1; d > 0; d >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < A.M / 2; t += blockDim.x) {
                const int lo = 2 * t - (t & (d - 1)), hi = lo + d;       // bit d of lo is 0
                const bool up = (lo & len) == 0;
                const uint64_t xa = x[lo], xb = x[hi];
                const uint32_t ra = r[lo], rb = r[hi];
                if (bs_less(xb, rb, xa, ra) == up) {
                    x[lo] = xb; x[hi] = xa;
                    r[lo] = rb; r[hi] = ra;
                }
            }
        }
    __syncthreads();
    for (int b = threadIdx.x; b + 1 < A.NB; b += blockDim.x) {
        const int q = (int)((int64_t)A.M * (b + 1) / A.NB);
        A.split_x[(size_t)i * A.NB + b] = x[q];
        A.split_r[(size_t)i * A.NB + b] = r[q];
    }
    // where the splitters of every cell of the key range begin and end
    const int ns = A.NB - 1;
    auto splitter = [&](int b) { return x[(int)((int64_t)A.M * (b + 1) / A.NB)]; };
    const BsCells cell(splitter(0), splitter(ns - 1), BS_CELLS);
    for (uint32_t c = threadIdx.x; c < BS_CELLS; c += blockDim.x) {
        int e[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int lo = 0, hi = ns;                        // splitters of the cells before c + h
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (cell(splitter(mid)) < c + h) lo = mid + 1;
                else hi = mid;
            }
            e[h] = lo;
        }
        A.cells[(size_t)i * BS_CELLS + c] = (uint32_t)e[0] | (uint32_t)e[1] << 16;
    }
}

// bucket of every entry of a tile, and the tile's place within each bucket (the tiles take
// their places in the order they arrive)
__global__ void __launch_bounds__(512) k_bs_count(BsArgs A)
{
    __shared__ uint64_t sx[BS_MAX_BUCKETS];
    __shared__ uint32_t sr[BS_MAX_BUCKETS];
    __shared__ uint32_t h[BS_MAX_BUCKETS];
    __shared__ uint32_t sc[BS_CELLS];
    const int i = blockIdx.y, tile = blockIdx.x, ns = A.NB - 1;
    for (int c = threadIdx.x; c < BS_CELLS; c += blockDim.x) sc[c] = A.cells[(size_t)i * BS_CELLS + c];
    for (int b = threadIdx.x; b < BS_MAX_BUCKETS; b += blockDim.x) {
        sx[b] = b < ns ? A.split_x[(size_t)i * A.NB + b] : ~0ull;
        sr[b] = b < ns ? A.split_r[(size_t)i * A.NB + b] : ~0u;
        h[b] = 0;
    }
    __syncthreads();
    const BsCells cell(sx[0], sx[ns - 1], BS_CELLS);
    const int64_t* K = A.keys + (size_t)(A.node0 + i) * A.Sp;
    uint16_t* B = A.bid + (size_t)i * A.S;
    const int64_t e1 = min((int64_t)(tile + 1) * BS_TILE, A.S);
#pragma unroll 4
    for (int64_t e = (int64_t)tile * BS_TILE + threadIdx.x; e < e1; e += 512) {
        const uint64_t x = bs_key(K[e]);
        const uint32_t range = sc[cell(x)];
        int b = (int)(range & 0xffffu), b1 = (int)(range >> 16);        // splitters below x ...
        while (b < b1) {
            const int mid = (b + b1) >> 1;
            if (sx[mid] < x) b = mid + 1;
            else b1 = mid;
        }
        if (b < ns && sx[b] == x) {                                     // ... and ties at or below e
            b1 = (int)(range >> 16);
            while (b < b1) {
                const int mid = (b + b1) >> 1;
                if (sx[mid] == x && sr[mid] <= (uint32_t)e) b = mid + 1;
                else b1 = mid;
            }
        }
        B[e] = (uint16_t)b;
        atomicAdd(&h[b], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < A.NB; b += blockDim.x)
        A.tile_base[((size_t)i * A.tiles + tile) * A.NB + b] = h[b] ? atomicAdd(&A.counts[(size_t)i * A.NB + b], h[b]) : 0u;
}

// first entry of every bucket (one block a node; the second half of `counts`)
__global__ void __launch_bounds__(BS_MAX_BUCKETS) k_bs_scan(BsArgs A, int nb)
{
    __shared__ uint32_t w[32];
    const int i = blockIdx.x, b = threadIdx.x, lane = b & 31;
    const uint32_t c = b < A.NB ? A.counts[(size_t)i * A.NB + b] : 0u;
    uint32_t s = c;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, s, d);
        if (lane >= d) s += y;
    }
    if (lane == 31) w[b >> 5] = s;
    __syncthreads();
    if (b < 32) {
        uint32_t v = w[b], t = v;
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, d);
            if (b >= d) t += y;
        }
        w[b] = t - v;
    }
    __syncthreads();
    if (b < A.NB) A.counts[(size_t)(nb + i) * A.NB + b] = s - c + w[b >> 5];
}

// Moves a tile's entries to their buckets.  They are put in bucket order in shared memory
// first: the tile's entries of one bucket (17 on average at n = 60) then leave as one run of
// 8-byte and one of 4-byte words instead of one by one.
static constexpr int BS_ROUNDS = BS_TILE / 512;
static constexpr size_t BS_SCATTER_SMEM = (size_t)BS_TILE * 12;
__global__ void __launch_bounds__(512) k_bs_scatter(BsArgs A, int nb)
{
    extern __shared__ __align__(16) uint8_t bs_sm[];
    uint64_t* sx = (uint64_t*)bs_sm;                    // [TILE] keys in bucket order
    uint32_t* sv = (uint32_t*)(sx + BS_TILE);           // [TILE] entry of the tile | bucket << 16
    __shared__ uint32_t h[BS_MAX_BUCKETS];              // entries of a bucket, then its first place here
    __shared__ uint32_t to[BS_MAX_BUCKETS];             // its first place among the node's, less that
    __shared__ uint32_t w[16];
    const int i = blockIdx.y, tile = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t e0 = (int64_t)tile * BS_TILE;
    const int cnt = (int)min((int64_t)BS_TILE, A.S - e0);
    const int64_t* K = A.keys + (size_t)(A.node0 + i) * A.Sp + e0;
    const uint16_t* B = A.bid + (size_t)i * A.S + e0;
    h[tid] = 0;
    h[tid + 512] = 0;
    __syncthreads();
    uint32_t v[BS_ROUNDS];                              // bucket << 16 | place within the tile's bucket
#pragma unroll
    for (int u = 0; u < BS_ROUNDS; ++u) {
        const int e = u * 512 + tid;
        v[u] = e < cnt ? (uint32_t)B[e] << 16 : 0u;
    }
#pragma unroll
    for (int u = 0; u < BS_ROUNDS; ++u)
        if (u * 512 + tid < cnt) v[u] |= atomicAdd(&h[v[u] >> 16], 1u);
    __syncthreads();
    // exclusive scan of the 1,024 counts, two a thread
    const uint32_t c0 = h[2 * tid], c1 = h[2 * tid + 1];
    uint32_t s = c0 + c1;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, s, d);
        if (lane >= d) s += y;
    }
    if (lane == 31) w[warp] = s;
    __syncthreads();
    s += __reduce_add_sync(0xffffffffu, lane < warp ? w[lane] : 0u) - (c0 + c1);
    h[2 * tid] = s;
    h[2 * tid + 1] = s + c0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int b = 2 * tid + q;
        if (b < A.NB)
            to[b] = A.counts[(size_t)(nb + i) * A.NB + b] + A.tile_base[((size_t)i * A.tiles + tile) * A.NB + b] -
                    (q ? s + c0 : s);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < BS_ROUNDS; ++u) {
        const int e = u * 512 + tid;
        if (e < cnt) {
            const uint32_t b = v[u] >> 16, p = h[b] + (v[u] & 0xffffu);
            sx[p] = bs_key(K[e]);
            sv[p] = (uint32_t)e | b << 16;
        }
    }
    __syncthreads();
    uint64_t* X = A.bx + (size_t)i * A.S;
    uint32_t* R = A.br + (size_t)i * A.S;
#pragma unroll 4
    for (int p = tid; p < cnt; p += 512) {
        const uint32_t y = sv[p], at = to[y >> 16] + (uint32_t)p;
        X[at] = sx[p];
        R[at] = (uint32_t)e0 + (y & 0xffffu);
    }
}

// the outputs of one entry: sorted position p of node i holds rank r
__device__ __forceinline__ void bs_write(const BsArgs& A, int i, uint32_t p, uint32_t r)
{
    A.srank[(size_t)i * A.Sp + p] = r;
    A.spos[(size_t)i * A.Sp + r] = p;
    if (A.sset) A.sset[(size_t)i * A.Ssp + p] = sset_word(A.pst[r], i);
}

// A bucket whose cnt entries in sx, sr tie or crowd: put in order by a bitonic network, then
// written.  All its comparators put the lower entry first (the first step of a merge mirrors
// its second half), so entries past cnt count as larger than any without being there.  Not
// inlined: it would cost k_bs_sort registers where nothing crowds (574 -> 597 us at n = 60).
__device__ __noinline__ void bs_sort_crowded(const BsArgs& A, int i, uint32_t p0, int cnt, uint64_t* sx, uint32_t* sr)
{
    int half = 1;                                       // half the power of two that holds cnt
    while (2 * half < cnt) half *= 2;
    for (int len = 2; len <= 2 * half; len *= 2)
        for (int d = len / 2; d > 0; d /= 2) {
            __syncthreads();
            for (int t = threadIdx.x; t < half; t += BS_THREADS) {
                const int o = t & (d - 1), lo = 2 * t - o, hi = 2 * d == len ? lo + len - 1 - 2 * o : lo + d;
                if (hi >= cnt) continue;
                const uint64_t xa = sx[lo], xb = sx[hi];
                const uint32_t ra = sr[lo], rb = sr[hi];
                if (bs_less(xb, rb, xa, ra)) {
                    sx[lo] = xb; sx[hi] = xa;
                    sr[lo] = rb; sr[hi] = ra;
                }
            }
        }
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += BS_THREADS) bs_write(A, i, p0 + t, sr[t]);
}

// One block a bucket.  The entries are spread over BS_NSUB sub-buckets of equal width (the
// keys of one bucket are close to evenly spread), and an entry's place is its sub-bucket's
// start plus the entries of it that come before (one compare on average).  Where scores tie or
// crowd (more than BS_CROWD entries in four sub-buckets), the block sorts the bucket by a
// bitonic network instead: 60 nodes, k = 4, all scores equal rank in 3.1 ms, by the compares
// in 15.3, by the radix sort in 4.6 (all different: 1.2, 1.2 and 7.7).  The last pass takes
// the entries by sub-bucket, so that its writes of srank and sset stay nearly in order.
// Three blocks an SM (two spill nothing and take 10 % longer).  WHOLE: a node's entries are
// one bucket, read straight from the table.  Buckets above BS_CAP are placed by counting, tile
// by tile.  Eight samples a bucket let hardly any reach four times the average of 1,024; from
// 1 M sets a node on the average grows to 2,048 and about one bucket in a hundred is above
// (49 nodes, k = 5, 1.9 M sets a node: ranked in 9.6 ms, by the radix sort in 29.4).
template <bool WHOLE>
__global__ void __launch_bounds__(BS_THREADS, 3) k_bs_sort(BsArgs A, int nb)
{
    extern __shared__ __align__(16) uint8_t bs_sm[];
    uint64_t* sx = (uint64_t*)bs_sm;                    // [CAP] by sub-bucket
    uint32_t* sr = (uint32_t*)(sx + BS_CAP);            // [CAP]
    uint32_t* sub = sr + BS_CAP;                        // [NSUB + 1]
    __shared__ uint64_t s_min[BS_THREADS / 32], s_max[BS_THREADS / 32];
    __shared__ uint32_t s_w[BS_THREADS / 32];
    __shared__ int s_crowd;                             // four sub-buckets side by side have more than BS_CROWD entries
    const int i = blockIdx.y, b = blockIdx.x, node = A.node0 + i;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t p0 = 0;
    int cnt = (int)A.S;
    const uint64_t* gx = nullptr;
    const uint32_t* gr = nullptr;
    if (!WHOLE) {
        cnt = (int)A.counts[(size_t)i * A.NB + b];
        p0 = A.counts[(size_t)(nb + i) * A.NB + b];
        gx = A.bx + (size_t)i * A.S + p0;
        gr = A.br + (size_t)i * A.S + p0;
        if (cnt > BS_CAP) {
            for (int e0 = 0; e0 < cnt; e0 += BS_THREADS) {                       // (block-uniform)
                const int e = e0 + threadIdx.x;
                const uint64_t x = e < cnt ? gx[e] : 0;
                const uint32_t r = e < cnt ? gr[e] : 0;
                uint32_t q = 0;
                for (int t0 = 0; t0 < cnt; t0 += BS_CAP) {
                    const int m = min(BS_CAP, cnt - t0);
                    __syncthreads();
                    for (int t = threadIdx.x; t < m; t += BS_THREADS) {
                        sx[t] = gx[t0 + t];
                        sr[t] = gr[t0 + t];
                    }
                    __syncthreads();
                    for (int t = 0; t < m; ++t) q += bs_less(sx[t], sr[t], x, r);
                }
                if (e < cnt) bs_write(A, node, p0 + q, r);
            }
            return;
        }
    }
    uint64_t x[BS_PER], lo = ~0ull, hi = 0ull;
    uint32_t at[BS_PER];                                // sub-bucket << 16 | place within it
#pragma unroll
    for (int u = 0; u < BS_PER; ++u) {
        const int e = u * BS_THREADS + threadIdx.x;
        x[u] = 0;
        if (e < cnt) x[u] = WHOLE ? bs_key(A.keys[(size_t)node * A.Sp + e]) : gx[e];
    }
    for (int q = threadIdx.x; q < BS_NSUB; q += BS_THREADS) sub[q] = 0;
    if (threadIdx.x == 0) s_crowd = 0;
    if (!WHOLE && b > 0 && b + 1 < A.NB) {              // between two splitters
        lo = A.split_x[(size_t)i * A.NB + b - 1];
        hi = A.split_x[(size_t)i * A.NB + b];
    } else {
#pragma unroll
        for (int u = 0; u < BS_PER; ++u)
            if (u * BS_THREADS + (int)threadIdx.x < cnt) {
                lo = min(lo, x[u]);
                hi = max(hi, x[u]);
            }
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, d));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, d));
        }
        if (lane == 0) {
            s_min[warp] = lo;
            s_max[warp] = hi;
        }
        __syncthreads();
        for (int w = 0; w < BS_THREADS / 32; ++w) {
            lo = min(lo, s_min[w]);
            hi = max(hi, s_max[w]);
        }
    }
    __syncthreads();
    if (hi < lo) return;                                                         // an empty bucket
    const BsCells cell(lo, hi, BS_NSUB);
#pragma unroll
    for (int u = 0; u < BS_PER; ++u)
        if (u * BS_THREADS + (int)threadIdx.x < cnt) {
            const uint32_t d = cell(x[u]);
            at[u] = d << 16 | atomicAdd(&sub[d], 1u);
        }
    __syncthreads();
    {
        // exclusive scan of the sub-bucket counts, four a thread
        static_assert(BS_NSUB == 4 * BS_THREADS, "four sub-buckets a thread");
        uint32_t c[4], s = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            c[q] = sub[4 * threadIdx.x + q];
            s += c[q];
        }
        const uint32_t mine = s;
        if (mine > BS_CROWD) s_crowd = 1;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, s, d);
            if (lane >= d) s += y;
        }
        if (lane == 31) s_w[warp] = s;
        __syncthreads();
        s += __reduce_add_sync(0xffffffffu, lane < warp ? s_w[lane] : 0u) - mine;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            sub[4 * threadIdx.x + q] = s;
            s += c[q];
        }
        if (threadIdx.x == 0) sub[BS_NSUB] = (uint32_t)cnt;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < BS_PER; ++u) {
        const int e = u * BS_THREADS + threadIdx.x;
        if (e < cnt) {
            const uint32_t q = sub[at[u] >> 16] + (at[u] & 0xffffu);
            sx[q] = x[u];
            sr[q] = WHOLE ? (uint32_t)e : gr[e];
        }
    }
    __syncthreads();
    if (s_crowd) {                                      // (block-uniform)
        bs_sort_crowded(A, node, p0, cnt, sx, sr);
        return;
    }
    for (int t = threadIdx.x; t < cnt; t += BS_THREADS) {
        const uint64_t y = sx[t];
        const uint32_t r = sr[t], d = cell(y);
        const uint32_t s0 = sub[d], s1 = sub[d + 1];
        uint32_t q = s0;
        for (uint32_t o = s0; o < s1; ++o) q += bs_less(sx[o], sr[o], y, r);
        bs_write(A, node, p0 + q, r);
    }
}

static constexpr size_t BS_SMEM = (size_t)BS_CAP * 12 + 4 * (BS_NSUB + 1);

// sorted positions at or past S of the parent-node words (padding up to the row stride, a
// whole number of the sliced scan's stages): never consistent with an order
__global__ void k_sset_pad(uint32_t* __restrict__ sset, int64_t S, int64_t Ssp)
{
    const int64_t p = S + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < Ssp) sset[(size_t)blockIdx.y * Ssp + p] = SSET_NEVER;
}

// the empty set's sorted position of every node, plus 1
__global__ void k_cut(const uint32_t* __restrict__ spos, int64_t Sp, int n, uint32_t* __restrict__ cut)
{
    if ((int)threadIdx.x < n) cut[threadIdx.x] = spos[(size_t)threadIdx.x * Sp] + 1;
}

// spos_t[r / 2][i][r % 2] = spos[i][r]: 32 x 32 tiles through shared memory, a thread
// storing the two positions of a rank pair of one node as one 8-byte word (coalesced both
// ways)
__global__ void k_spos_transpose(const uint32_t* __restrict__ spos, int n, int64_t Sp, uint32_t* __restrict__ spos_t)
{
    __shared__ uint32_t tile[32][33];                      // [node][rank]
    const int64_t r0 = (int64_t)blockIdx.x * 32;
    const int i0 = blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;          // 32 x 8 threads
    for (int y = ty; y < 32; y += 8) {
        const int i = i0 + y;
        if (i < n) tile[y][tx] = spos[(size_t)i * Sp + r0 + tx];
    }
    __syncthreads();
    uint2* out = (uint2*)spos_t;
    for (int y2 = ty; y2 < 16; y2 += 8) {
        const int i = i0 + tx;
        if (i < n) out[(size_t)(r0 / 2 + y2) * n + i] = make_uint2(tile[tx][2 * y2], tile[tx][2 * y2 + 1]);
    }
}

__global__ void k_spos_pad(uint32_t* __restrict__ spos, uint32_t* __restrict__ srank, int n, int64_t S, int64_t Sp)
{
    const int64_t pad = Sp - S;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)n * pad) return;
    const int64_t i = idx / pad, e = idx - i * pad;
    spos[i * Sp + S + e] = 0xffffffffu;
    srank[i * Sp + S + e] = 0u;
}

// stream-ordered temporaries of one call
struct SortTemps {
    cudaStream_t s;
    std::vector<void*> p;
    ~SortTemps()
    {
        for (void* q : p) dev_free(q, s);
    }
    template <class T>
    int get(T** out, size_t count)
    {
        void* q = nullptr;
        cudaError_t e = dev_alloc(&q, std::max<size_t>(count, 1) * sizeof(T), s);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return set_error(BN_ENOMEM, "rank_entries: %zu bytes of sort buffers: %s", count * sizeof(T),
                             cudaGetErrorString(e));
        }
        p.push_back(q);
        *out = (T*)q;
        return BN_OK;
    }
};

static int rank_by_buckets(bn_table* t, cudaStream_t s)
{
    const int64_t S = t->S;
    const int per = (int)std::max<int64_t>(1, std::min<int64_t>(t->n, 0x7fffffffLL / S));
    BsArgs A;
    A.keys = t->keys;
    A.pst = t->pst;
    A.S = S;
    A.Sp = t->Sp;
    A.srank = t->srank;
    A.spos = t->spos;
    A.sset = t->sset;
    A.Ssp = t->sset_stride;
    const bool whole = S <= BS_CAP;
    A.NB = whole ? 1 : (int)std::min<int64_t>(BS_MAX_BUCKETS, (S + BS_AVG - 1) / BS_AVG);
    A.tiles = (int)((S + BS_TILE - 1) / BS_TILE);
    A.M = 32;
    while (A.M < 8 * A.NB && A.M < BS_SAMPLES) A.M *= 2;
    SortTemps tmp{s, {}};
    int rc;
    if (!whole &&
        ((rc = tmp.get(&A.split_x, (size_t)per * A.NB)) || (rc = tmp.get(&A.split_r, (size_t)per * A.NB)) ||
         (rc = tmp.get(&A.cells, (size_t)per * BS_CELLS)) ||
         (rc = tmp.get(&A.counts, (size_t)2 * per * A.NB)) ||
         (rc = tmp.get(&A.tile_base, (size_t)per * A.tiles * A.NB)) || (rc = tmp.get(&A.bid, (size_t)per * S)) ||
         (rc = tmp.get(&A.bx, (size_t)per * S)) || (rc = tmp.get(&A.br, (size_t)per * S))))
        return rc;
    static ContextOnce once;
    rc = once_in_context(once, [&]() -> int {
        BN_CUDA(cudaFuncSetAttribute(k_bs_split, cudaFuncAttributeMaxDynamicSharedMemorySize, BS_SAMPLES * 12));
        BN_CUDA(cudaFuncSetAttribute(k_bs_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BS_SCATTER_SMEM));
        BN_CUDA(cudaFuncSetAttribute(k_bs_sort<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BS_SMEM));
        BN_CUDA(cudaFuncSetAttribute(k_bs_sort<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BS_SMEM));
        return BN_OK;
    });
    if (rc) return rc;
    for (A.node0 = 0; A.node0 < t->n; A.node0 += per) {
        const int nb = std::min(per, t->n - A.node0);
        if (whole) {
            k_bs_sort<true><<<dim3(1, (unsigned)nb), BS_THREADS, BS_SMEM, s>>>(A, nb);
            BN_LAUNCH_CHECK("k_bs_sort");
            continue;
        }
        BN_CUDA(cudaMemsetAsync(A.counts, 0, sizeof(uint32_t) * (size_t)nb * A.NB, s));
        k_bs_split<<<nb, 1024, (size_t)A.M * 12, s>>>(A);
        BN_LAUNCH_CHECK("k_bs_split");
        k_bs_count<<<dim3((unsigned)A.tiles, (unsigned)nb), 512, 0, s>>>(A);
        BN_LAUNCH_CHECK("k_bs_count");
        k_bs_scan<<<nb, BS_MAX_BUCKETS, 0, s>>>(A, nb);
        BN_LAUNCH_CHECK("k_bs_scan");
        k_bs_scatter<<<dim3((unsigned)A.tiles, (unsigned)nb), 512, BS_SCATTER_SMEM, s>>>(A, nb);
        BN_LAUNCH_CHECK("k_bs_scatter");
        k_bs_sort<false><<<dim3((unsigned)A.NB, (unsigned)nb), BS_THREADS, BS_SMEM, s>>>(A, nb);
        BN_LAUNCH_CHECK("k_bs_sort");
    }
    return BN_OK;
}

static int rank_by_radix(bn_table* t, cudaStream_t s)
{
    const int64_t S = t->S;
    // nodes per batch so that batch * S fits the 32-bit value
    const int per = (int)std::max<int64_t>(1, std::min<int64_t>(t->n, 0x7fffffffLL / S));
    const int64_t Nmax = (int64_t)per * S;
    const int Tmax = (int)((Nmax + RS_TILE - 1) / RS_TILE);
    uint64_t *k0 = nullptr, *k1 = nullptr;
    uint32_t *v0 = nullptr, *v1 = nullptr, *counts = nullptr, *totals = nullptr;
    cudaError_t e = dev_alloc((void**)&k0, 8 * (size_t)Nmax, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&k1, 8 * (size_t)Nmax, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&v0, 4 * (size_t)Nmax, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&v1, 4 * (size_t)Nmax, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&counts, 4 * (size_t)256 * Tmax, s);
    if (e == cudaSuccess) e = dev_alloc((void**)&totals, 4 * 256, s);
    struct F {
        cudaStream_t s;
        void* p[6];
        ~F()
        {
            for (void* q : p)
                if (q) dev_free(q, s);
        }
    } fr{s, {k0, k1, v0, v1, counts, totals}};
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(BN_ENOMEM, "rank_entries: %zu bytes of sort buffers: %s", (size_t)Nmax * 24,
                         cudaGetErrorString(e));
    }
    for (int node0 = 0; node0 < t->n; node0 += per) {
        const int nb = std::min(per, t->n - node0);
        const int64_t N = (int64_t)nb * S;
        const int T = (int)((N + RS_TILE - 1) / RS_TILE);
        k_rs_init<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(t->keys, t->Sp, S, node0, N, k0, v0);
        BN_LAUNCH_CHECK("k_rs_init");
        uint64_t *ki = k0, *ko = k1;
        uint32_t *vi = v0, *vo = v1;
        for (int pass = 0; pass < 9; ++pass) {
            RsPass P;
            P.kin = ki;
            P.vin = vi;
            P.kout = ko;
            P.vout = vo;
            P.N = N;
            P.shift = pass < 8 ? 8 * pass : -1;
            P.S = S;
            P.node0 = node0;
            P.counts = counts;
            P.totals = totals;
            P.T = T;
            if (pass == 8 && nb == 1) break;        // a single node needs no node pass
            k_rs_hist<<<T, RS_THREADS, 0, s>>>(P);
            BN_LAUNCH_CHECK("k_rs_hist");
            k_rs_scan<<<256, 1024, 0, s>>>(counts, T, totals);
            BN_LAUNCH_CHECK("k_rs_scan");
            k_rs_scatter<<<T, RS_THREADS, 0, s>>>(P);
            BN_LAUNCH_CHECK("k_rs_scatter");
            std::swap(ki, ko);
            std::swap(vi, vo);
        }
        k_rs_finish<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(vi, N, S, t->Sp, node0, t->srank, t->spos);
        BN_LAUNCH_CHECK("k_rs_finish");
    }
    return BN_OK;
}

// Ranks every node's entries (see the file comment) and lays out what the scans read:
// srank, spos, its entry-major copy spos_t and (k <= 4) the parent nodes by sorted
// position.  d_cut receives each node's empty-set position + 1 (device, n words; the caller
// copies it to t->cut).  Temporaries are stream-ordered.  The parent nodes' memory is taken here
// and not with the rest of the table, though that may wait for the counting kernels (whose
// freed sums it can reuse): taken before them, the host's 10 to 20 us come before the first
// kernel instead of behind it (37 nodes learned end to end 2.34 -> 2.35 ms, twelve networks
// 19.2 -> 19.3).
int rank_entries(bn_table* t, uint32_t* d_cut, cudaStream_t s)
{
    const int64_t S = t->S;
    if (S > 0xffffffffLL) return set_error(BN_EUNSUPPORTED, "rank_entries: too many sets per node");
    int rc = alloc_sset(t);
    if (rc) return rc;
    if (S <= (int64_t)BS_MAX_BUCKETS * 2 * BS_AVG) {
        if ((rc = rank_by_buckets(t, s))) return rc;
    } else {
        if ((rc = rank_by_radix(t, s))) return rc;
        if (t->sset && (rc = build_sset(t, s))) return rc;
    }
    if (t->sset && t->sset_stride > S) {
        k_sset_pad<<<dim3((unsigned)((t->sset_stride - S + 255) / 256), (unsigned)t->n), 256, 0, s>>>(t->sset, S,
                                                                                                 t->sset_stride);
        BN_LAUNCH_CHECK("k_sset_pad");
    }
    if (t->Sp > S) {
        const int64_t tot = (int64_t)t->n * (t->Sp - S);
        k_spos_pad<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(t->spos, t->srank, t->n, S, t->Sp);
        BN_LAUNCH_CHECK("k_spos_pad");
    }
    k_spos_transpose<<<dim3((unsigned)(t->Sp / 32), (unsigned)((t->n + 31) / 32)), dim3(32, 8), 0, s>>>(t->spos, t->n, t->Sp,
                                                                                                    t->spos_t);
    BN_LAUNCH_CHECK("k_spos_transpose");
    k_cut<<<1, MAXN, 0, s>>>(t->spos, t->Sp, t->n, d_cut);
    BN_LAUNCH_CHECK("k_cut");
    return BN_OK;
}

}  // namespace bn
