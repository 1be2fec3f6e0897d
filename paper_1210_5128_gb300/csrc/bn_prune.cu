// bn_prune.cu -- exact pruning of the table and the scan over what is left.
//
// An entry (i, pi) can never be the answer of Eq. (6) if some proper subset pi' of pi
// scores at least as well: whenever pi lies inside a node's predecessors so does pi',
// and pi' wins (a higher score, or an equal score at a lower rank -- ranks are
// size-ascending).  Removing every such "dominated" entry leaves every order's result
// unchanged.  For each node the surviving entries are kept in sorted-position order
// (score descending, rank ascending), so a scan over them can stop at its first
// consistent entry.
//
// best_le(pi) = max over all subsets of pi (pi included) of the entry key, computed size
// class by size class from the j immediate subsets; pi survives iff key(pi) >
// max_t best_le(pi minus its t-th element).
#include <algorithm>
#include <cstring>
#include <vector>

#include "bn_table.cuh"

namespace bn {

static constexpr int PR_CHUNK = 4096;     // sorted positions per compaction block
static constexpr int PR_WORDS = PR_CHUNK / 32;
static constexpr int PS_CHUNK = 2048;     // surviving entries per pruned-scan block
static constexpr int PR_MAX_K = 7;
static constexpr int PR_BLOCK = 2048;     // entries of a dominance block (its binomial table is paid once)

struct DomArgs {
    const int64_t* keys;       // [n][Sp]
    const uint64_t* pst;
    const uint32_t* spos;      // [n][Sp]
    int64_t Sp;
    int64_t base, count;       // first rank and number of the size class's sets
    int64_t sub_base;          // first rank of the next smaller class
    int64_t below;             // sets smaller than the largest class: best_le's row stride
    int64_t* best_le;          // [n][below]; the largest class is not stored
    uint32_t* alive;           // [n][words] survivors by sorted position, one bit each
    int64_t words;
    unsigned long long* maxabs;   // largest |entry| among the survivors, as bits
};

// One thread per entry of size class J (consecutive threads, consecutive ranks: neighbours
// differ in their lowest element, so the key and the J subset reads are coalesced or
// broadcast).  The rank of the set without its t-th element is a prefix sum of C(a_s, s)
// over s < t plus a suffix sum of C(a_s, s - 1) over s > t.  Bound by the 8 bytes of key an
// entry from HBM and the subset reads from L2: the largest class
// of n = 37, k = 4 takes 20 us, all five classes 45 us, against 448 us with one thread per
// 64 consecutive ranks.
template <int J>
__global__ void __launch_bounds__(256) k_dominance(DomArgs A)
{
    __shared__ uint32_t bin[64 * (J + 1)];                       // C(a, t), t <= J (ranks are below 2^31)
    for (int q = threadIdx.x; q < 64 * (J + 1); q += blockDim.x) bin[q] = (uint32_t)g_binom.v[q / (J + 1)][q % (J + 1)];
    __syncthreads();
    const int i = blockIdx.y;
    const int64_t r1 = min((int64_t)(blockIdx.x + 1) * PR_BLOCK, A.count);
    unsigned long long mag = 0;
#pragma unroll 2
    for (int64_t r = (int64_t)blockIdx.x * PR_BLOCK + threadIdx.x; r < r1; r += 256) {
        const int64_t key = A.keys[(size_t)i * A.Sp + A.base + r];
        int64_t sub_max = KEY_NONE;
        if (J > 0) {
            const int64_t* BL = A.best_le + (size_t)i * A.below + A.sub_base;
            uint64_t m = A.pst[A.base + r];
            uint32_t lo[J + 1], up[J + 1];                       // C(a_s, s), C(a_s, s - 1)
            uint32_t suf = 0;
#pragma unroll
            for (int t = 0; t < J; ++t) {
                const int a = __ffsll((long long)m) - 1;
                m &= m - 1;
                lo[t] = bin[a * (J + 1) + t + 1];
                up[t] = bin[a * (J + 1) + t];
                suf += up[t];
            }
            uint32_t pre = 0;
#pragma unroll
            for (int t = 0; t < J; ++t) {
                suf -= up[t];
                sub_max = max(sub_max, BL[pre + suf]);
                pre += lo[t];
            }
        }
        if (A.base + r < A.below) A.best_le[(size_t)i * A.below + A.base + r] = max(key, sub_max);
        if (J == 0 || key > sub_max) {
            const uint32_t p = A.spos[(size_t)i * A.Sp + A.base + r];
            atomicOr(&A.alive[(size_t)i * A.words + (p >> 5)], 1u << (p & 31));
            // (positive doubles order like their bits)
            mag = max(mag, (unsigned long long)__double_as_longlong(fabs(key_to_double(key))));
        }
    }
    if (__any_sync(0xffffffffu, mag != 0)) {
#pragma unroll
        for (int d = 16; d; d >>= 1) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, d));
        if ((threadIdx.x & 31) == 0) atomicMax(A.maxabs, mag);
    }
}

// survivors per (node, chunk of sorted positions)
__global__ void __launch_bounds__(PR_WORDS) k_alive_count(const uint32_t* __restrict__ alive, int64_t words, int nch,
                                                          uint32_t* __restrict__ counts)
{
    __shared__ uint32_t s[PR_WORDS / 32];
    const int64_t w = (int64_t)blockIdx.x * PR_WORDS + threadIdx.x;
    const uint32_t c = w < words ? (uint32_t)__popc(alive[(size_t)blockIdx.y * words + w]) : 0u;
    const uint32_t v = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t tot = 0;
        for (int q = 0; q < PR_WORDS / 32; ++q) tot += s[q];
        counts[(size_t)blockIdx.y * nch + blockIdx.x] = tot;
    }
}

// first survivor of every chunk (in place) and every node, and the nodes' counts
__global__ void __launch_bounds__(1024) k_alive_scan(uint32_t* __restrict__ counts, int n, int nch,
                                                     uint32_t* __restrict__ aoff, uint32_t* __restrict__ acnt)
{
    __shared__ uint32_t part[1024];
    const int64_t tot = (int64_t)n * nch, per = (tot + 1023) / 1024;
    const int64_t b = min(tot, threadIdx.x * per), e = min(tot, b + per);
    uint32_t s = 0;
    for (int64_t j = b; j < e; ++j) s += counts[j];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const uint32_t v = (int)threadIdx.x >= off ? part[threadIdx.x - off] : 0u;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    uint32_t run = part[threadIdx.x] - s;
    for (int64_t j = b; j < e; ++j) {
        const uint32_t c = counts[j];
        counts[j] = run;
        run += c;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += 1024) {
        const uint32_t o = counts[(size_t)i * nch];
        aoff[i] = o;
        acnt[i] = (i + 1 < n ? counts[(size_t)(i + 1) * nch] : part[1023]) - o;
    }
}

// the survivors of a chunk in sorted-position order
__global__ void __launch_bounds__(PR_WORDS) k_alive_write(const uint32_t* __restrict__ alive, int64_t words, int nch,
                                                          const uint32_t* __restrict__ first,
                                                          const uint32_t* __restrict__ srank, int64_t Sp,
                                                          const uint64_t* __restrict__ pst, uint64_t* __restrict__ amask,
                                                          uint32_t* __restrict__ aspos)
{
    __shared__ uint32_t wsum[PR_WORDS / 32];
    const int i = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * PR_WORDS + threadIdx.x;
    uint32_t bits = w < words ? alive[(size_t)i * words + w] : 0u;
    const uint32_t c = (uint32_t)__popc(bits);
    uint32_t s = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, s, d);
        if (lane >= d) s += y;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    uint32_t at = first[(size_t)i * nch + blockIdx.x] + s - c;
    for (int q = 0; q < warp; ++q) at += wsum[q];
    while (bits) {
        const uint32_t p = (uint32_t)(w * 32) + (uint32_t)__ffs((int)bits) - 1u;
        bits &= bits - 1;
        amask[at] = pst[srank[(size_t)i * Sp + p]];
        aspos[at++] = p;
    }
}

struct PrunedArgs {
    const uint64_t* amask;
    const uint32_t* aspos;
    const uint32_t* aoff;      // [n] first survivor of node i
    const uint32_t* acnt;      // [n]
    int max_chunks;
    const uint32_t* list_count;
    const uint64_t* list_pc;
    uint32_t* list_best;
    int cap;
};

// scan over a node's survivors in sorted-position order, staged in shared memory: each
// thread stops at its first consistent entry (the minimum sorted position within this
// chunk); warps leave when all their items have one; chunks combine with atomicMin
// (4,096 orders of 60 nodes, 24 survivors a node: 51 -> 24 us against reading each survivor
// from global memory in turn)
__global__ void __launch_bounds__(256) k_scan_pruned(PrunedArgs A)
{
    __shared__ uint64_t s_m[PS_CHUNK];
    const int node = blockIdx.x / A.max_chunks, ch = blockIdx.x - node * A.max_chunks;
    const int cnt = (int)A.list_count[node];
    const int g0 = blockIdx.y * 256;
    if (g0 >= cnt) return;                                                  // block-uniform
    const int64_t acount = A.acnt[node];
    const int64_t e0 = (int64_t)ch * PS_CHUNK;
    if (e0 >= acount) return;
    const int m = (int)min((int64_t)PS_CHUNK, acount - e0);
    const int item = g0 + (int)threadIdx.x;
    const bool active = item < cnt;
    const uint32_t off = A.aoff[node] + (uint32_t)e0;
    const uint64_t npc = active ? ~A.list_pc[(size_t)node * A.cap + item] : 0ull;
    for (int e = threadIdx.x; e < m; e += 256) s_m[e] = A.amask[off + e];
    __syncthreads();
    int best = active ? -1 : 0;
    for (int e = 0; e < m; e += 8) {
        uint32_t hit = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (e + u < m) hit |= (uint32_t)((s_m[e + u] & npc) == 0ull) << u;
        if (best < 0 && hit) best = e + __ffs((int)hit) - 1;
        if (__all_sync(0xffffffffu, best >= 0)) break;
    }
    if (active && best >= 0) atomicMin(&A.list_best[(size_t)node * A.cap + item], A.aspos[off + best]);
}

int launch_scan_pruned(const bn_table* t, const uint32_t* list_count, const uint64_t* list_pc, uint32_t* list_best,
                       int cap, cudaStream_t s)
{
    PrunedArgs A;
    A.amask = t->amask;
    A.aspos = t->aspos;
    A.aoff = t->aoff;
    A.acnt = t->acnt;
    A.max_chunks = t->alive_chunks;
    A.list_count = list_count;
    A.list_pc = list_pc;
    A.list_best = list_best;
    A.cap = cap;
    dim3 grid((unsigned)(t->n * t->alive_chunks), (unsigned)((cap + 255) / 256));
    k_scan_pruned<<<grid, 256, 0, s>>>(A);
    BN_LAUNCH_CHECK("k_scan_pruned");
    return BN_OK;
}

template <int J>
static int launch_dominance(const DomArgs& A, int n, cudaStream_t s)
{
    k_dominance<J><<<dim3((unsigned)((A.count + PR_BLOCK - 1) / PR_BLOCK), (unsigned)n), 256, 0, s>>>(A);
    BN_LAUNCH_CHECK("k_dominance");
    return BN_OK;
}

int prune_table(bn_table* t, cudaStream_t s)
{
    if (t->amask) return BN_OK;
    const int n = t->n, N = n - 1, k = t->k;
    if (k > PR_MAX_K) return set_error(BN_EUNSUPPORTED, "prune: k=%d above %d", k, PR_MAX_K);
    const int64_t S = t->S, words = (S + 31) / 32;
    const int nch = (int)((S + PR_CHUNK - 1) / PR_CHUNK);
    const int64_t below = S - (int64_t)h_binom.v[N][k];          // k <= n - 1
    // one work block: best_le | alive bits | largest |entry| | node offsets, counts | chunks
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = (size_t)round_up((int64_t)(off + bytes), 256);
        return o;
    };
    const size_t o_bits = take(4 * (size_t)n * words), o_max = take(8), o_aoff = take(4 * (size_t)n),
                 o_acnt = take(4 * (size_t)n), o_cnt = take(4 * (size_t)n * nch), o_le = take(8 * (size_t)n * below);
    uint8_t* work = nullptr;
    cudaError_t e = dev_alloc((void**)&work, off, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(BN_ENOMEM, "prune: %zu bytes of work space", off);
    }
    struct F {
        void* p;
        cudaStream_t s;
        ~F() { dev_free(p, s); }
    } fr{work, s};
    uint32_t* alive = (uint32_t*)(work + o_bits);
    uint32_t* counts = (uint32_t*)(work + o_cnt);
    BN_CUDA(cudaMemsetAsync(work, 0, o_max + 8, s));             // the bits and the maximum
    DomArgs A{t->keys, t->pst, t->spos, t->Sp, 0, 0, 0, below, (int64_t*)(work + o_le), alive, words,
              (unsigned long long*)(work + o_max)};
    for (int j = 0; j <= k; ++j) {
        A.count = (int64_t)h_binom.v[N][j];
        int rc = BN_OK;
        switch (j) {
            case 0: rc = launch_dominance<0>(A, n, s); break;
            case 1: rc = launch_dominance<1>(A, n, s); break;
            case 2: rc = launch_dominance<2>(A, n, s); break;
            case 3: rc = launch_dominance<3>(A, n, s); break;
            case 4: rc = launch_dominance<4>(A, n, s); break;
            case 5: rc = launch_dominance<5>(A, n, s); break;
            case 6: rc = launch_dominance<6>(A, n, s); break;
            default: rc = launch_dominance<7>(A, n, s); break;
        }
        if (rc) return rc;
        A.sub_base = A.base;
        A.base += A.count;
    }
    k_alive_count<<<dim3((unsigned)nch, (unsigned)n), PR_WORDS, 0, s>>>(alive, words, nch, counts);
    BN_LAUNCH_CHECK("k_alive_count");
    k_alive_scan<<<1, 1024, 0, s>>>(counts, n, nch, (uint32_t*)(work + o_aoff), (uint32_t*)(work + o_acnt));
    BN_LAUNCH_CHECK("k_alive_scan");
    // one read-back (the maximum, offsets and counts lie side by side) sizes the survivors
    std::vector<uint8_t> h(o_cnt - o_max);
    BN_CUDA(cudaMemcpyAsync(h.data(), work + o_max, h.size(), cudaMemcpyDeviceToHost, s));
    BN_CUDA(cudaStreamSynchronize(s));
    const uint32_t* hcnt = (const uint32_t*)(h.data() + (o_acnt - o_max));
    uint64_t run = 0;
    uint32_t mx = 0;
    for (int i = 0; i < n; ++i) {
        run += hcnt[i];
        mx = std::max(mx, hcnt[i]);
    }
    if (run >= 0xffffffffull) return set_error(BN_EUNSUPPORTED, "prune: too many surviving entries");
    uint8_t* blk = nullptr;
    const size_t m1 = (size_t)std::max<uint64_t>(run, 1);
    BN_CUDA(obj_alloc((void**)&blk, 12 * m1 + 8 * (size_t)n + 64));
    t->alive_block = blk;
    t->aspos = (uint32_t*)(blk + 8 * m1);
    t->aoff = (uint32_t*)(blk + 12 * m1);
    t->acnt = t->aoff + n;
    t->alive_total = (int64_t)run;
    t->alive_max = mx;
    t->alive_chunks = (int)std::max<uint32_t>(1, (mx + PS_CHUNK - 1) / PS_CHUNK);
    memcpy(&t->max_abs_survivor, h.data(), 8);
    BN_CUDA(cudaMemcpyAsync(t->aoff, work + o_aoff, 4 * (size_t)n, cudaMemcpyDeviceToDevice, s));
    BN_CUDA(cudaMemcpyAsync(t->acnt, work + o_acnt, 4 * (size_t)n, cudaMemcpyDeviceToDevice, s));
    t->amask = (uint64_t*)blk;
    k_alive_write<<<dim3((unsigned)nch, (unsigned)n), PR_WORDS, 0, s>>>(alive, words, nch, counts, t->srank, t->Sp, t->pst,
                                                                t->amask, t->aspos);
    BN_LAUNCH_CHECK("k_alive_write");
    int rc = build_survivor_cache(t, s);
    if (rc) return rc;
    BN_CUDA(cudaStreamSynchronize(s));
    return BN_OK;
}

}  // namespace bn

using namespace bn;

extern "C" int bn_table_set_scan(bn_table* t, int mode, void* stream)
{
    set_error(BN_OK, "");
    if (!t) return set_error(BN_EINVAL, "bn_table_set_scan: NULL table");
    if (mode != BN_SCAN_FULL && mode != BN_SCAN_PRUNED && mode != BN_SCAN_UNRANK && mode != BN_SCAN_SLICED &&
        mode != BN_SCAN_SORTED)
        return set_error(BN_EINVAL, "bn_table_set_scan: mode %d", mode);
    if ((mode == BN_SCAN_SLICED || mode == BN_SCAN_SORTED) && !t->sset)
        return set_error(BN_EUNSUPPORTED, "bn_table_set_scan: the bit-sliced scans need k <= 4 (k = %d)", t->k);
    if (mode == BN_SCAN_PRUNED) {
        int rc = prune_table(t, (cudaStream_t)stream);
        if (rc) return rc;
    }
    t->scan_mode = mode;
    return BN_OK;
}

extern "C" int bn_table_pruned(const bn_table* t, int64_t* survivors_per_node)
{
    set_error(BN_OK, "");
    if (!t || !survivors_per_node) return set_error(BN_EINVAL, "bn_table_pruned: NULL argument");
    if (!t->amask) return set_error(BN_EINVAL, "bn_table_pruned: the table has not been pruned");
    std::vector<uint32_t> h(t->n);
    BN_CUDA(cudaMemcpy(h.data(), t->acnt, 4 * (size_t)t->n, cudaMemcpyDeviceToHost));
    for (int i = 0; i < t->n; ++i) survivors_per_node[i] = h[i];
    return BN_OK;
}
