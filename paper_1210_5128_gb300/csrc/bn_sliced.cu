// bn_sliced.cu -- the order score of Eq. (6) with the orders bit-sliced.
//
// In a node's entries ordered by sorted position (score descending, rank ascending; see
// bn_sort.cu) the answer for an order is the FIRST entry whose parent set lies inside
// the node's predecessors.  So the (entry, order) tests need not each keep a running
// minimum: slice the orders into 32-bit words instead.  For node i, group g of 32 work
// items and node v, the word P[v][g] has bit r set when v precedes i in item 32g + r.
// An entry with parent nodes {v1, .., vj} (j <= k <= 4) is consistent with exactly the
// items of P[v1][g] & .. & P[vj][g]: four shared-memory words and three ANDs test one
// entry against 32 orders at once.  Of those items, the ones this warp has not found
// yet take the entry's sorted position (a shared-memory atomicMin, by the lowest lane of
// a step that hits the item), and a warp-wide OR marks them found.  Every later entry of
// the warp lies further down the sorted list, so it can only lose.  A node's stages (2,048
// entries) go round its blocks, so all of them walk from the top of the list to its end
// together, and they trade positions through the work list: an item that holds a position
// above a block's next stage is not tested there any more.
//
// The entries reach shared memory as one 4-byte word each (the parent node ids, a byte
// apiece, in sorted-position order; `sset`), streamed by 1-D bulk (TMA) copies, so a
// full pass reads 4 B per (node, entry) -- as the mask-test scan does -- but tests 32
// items per shared-memory word instead of one.  The per-lane copies of the P words
// (each lane reads its own bank) keep the four loads free of bank conflicts.
//
// Two modes.  The full pass reads every entry of the table.  The sorted mode
// (BN_SCAN_SORTED) stops early, with identical results: nothing past the empty set's
// sorted position can be chosen (the empty set is consistent with every order), and a
// block stops streaming once each of its items holds a position above the next stage
// (every entry still unread lies further down the list).
#include <algorithm>

#include "bn_table.cuh"

namespace bn {

static constexpr int SL_CWARPS = 8;                 // consumer warps
static constexpr int SL_THREADS = 32 * (SL_CWARPS + 1);   // and one producer warp
static constexpr int SL_SUB = 2048;                 // entries per stage
static constexpr int SL_STAGES = 4;
static constexpr int SL_PER_WARP = SL_SUB / SL_CWARPS;  // 256 entries of a stage per consumer warp
static constexpr int SL_ROWS = 66;                  // nodes 0..63, "no parent" (64), "never" (65)
static constexpr int SL_ROW_BYTES = 256;            // two groups' 32 lanes per row
static_assert(SSET_ONES == 64 && SSET_NEVER == 0x41414141u, "rows 64 (all ones) and 65 (all zero)");
static constexpr int SL_MAX_K = 4;

// The P copies of up to four groups sit in static shared memory, whose address the
// compiler knows, so a byte-permute result addresses a row directly; eight groups do not
// fit the static limit and use the dynamic region.
__host__ __device__ constexpr bool sl_static_p(int G) { return G <= 4; }
__host__ __device__ constexpr size_t sl_p_bytes(int G) { return (size_t)((G + 1) / 2) * SL_ROWS * SL_ROW_BYTES; }
// dynamic shared memory of a block
__host__ __device__ constexpr size_t sl_smem(int G)
{
    return (size_t)SL_STAGES * SL_SUB * 4            // staged entry words
           + (sl_static_p(G) ? 0 : sl_p_bytes(G))    // per-lane copies of P[v][g]
           + (size_t)32 * G * 4                      // per-item best sorted position
           + 16 * SL_STAGES + 64;                    // full/empty mbarriers, flags, skip words
}


struct SlicedArgs {
    const uint32_t* sset;          // [n][Ssp] parent node ids of the entry at each sorted position
    const uint32_t* spos;          // [n][Sp] sorted position of each rank (rank 0 = empty set)
    int64_t Sp, S;
    int64_t Ssp;                   // sset row stride: S rounded up to whole stages
    int n;
    int nchunk;                    // blocks per node and item set
    int per;                       // sorted mode: consecutive stages per block
    const uint32_t* list_count;
    const uint64_t* list_pc;
    uint32_t* list_best;
    int cap;
    uint32_t* status;
};

// ---------------------------------------------------------------------------------
// sset[i][p]: the parent nodes of the entry at sorted position p of node i (sset_word);
// positions at or past S (padding up to the row stride Ssp, a whole number of stages) hold
// SSET_NEVER.
// ---------------------------------------------------------------------------------
__global__ void k_sset(const uint32_t* __restrict__ srank, const uint64_t* __restrict__ pst, int n, int64_t S,
                       int64_t Sp, int64_t Ssp, uint32_t* __restrict__ sset)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (int64_t)n * S) return;
    const int i = (int)(g / S);
    const int64_t p = g - (int64_t)i * S;
    sset[(size_t)i * Ssp + p] = sset_word(pst[srank[(size_t)i * Sp + p]], i);
}

int alloc_sset(bn_table* t)
{
    if (t->k > SL_MAX_K || t->n > 64 || t->sset) return BN_OK;   // the mask-test scans serve larger k
    const int64_t Ssp = round_up(t->S, SL_SUB);
    cudaError_t e = obj_alloc(&t->sset, sizeof(uint32_t) * (size_t)t->n * (size_t)Ssp);
    if (e != cudaSuccess) {
        t->sset = nullptr;
        cudaGetLastError();
        return set_error(BN_ENOMEM, "sorted parent sets: %zu bytes: %s",
                         sizeof(uint32_t) * (size_t)t->n * (size_t)Ssp, cudaGetErrorString(e));
    }
    t->sset_stride = Ssp;
    t->bytes += sizeof(uint32_t) * (size_t)t->n * (size_t)Ssp;
    return BN_OK;
}

int build_sset(bn_table* t, cudaStream_t s)
{
    const int64_t tot = (int64_t)t->n * t->S;
    k_sset<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(t->srank, t->pst, t->n, t->S, t->Sp, t->sset_stride, t->sset);
    BN_LAUNCH_CHECK("k_sset");
    return BN_OK;
}

// word index of P[v][g] for lane 0
__device__ __forceinline__ int Pw(int g, int v)
{
    return (g >> 1) * SL_ROWS * (SL_ROW_BYTES / 4) + v * (SL_ROW_BYTES / 4) + (g & 1) * 32;
}

// bit l of lane r's result = bit r of lane l's x (five exchange steps)
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane)
{
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        const uint32_t m = d == 16 ? 0x0000ffffu : d == 8 ? 0x00ff00ffu : d == 4 ? 0x0f0f0f0fu : d == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, d);
        x = (lane & d) ? (x & ~m) | ((y & ~m) >> d) : (x & m) | ((y & m) << d);
    }
    return x;
}

// Records a step's new items of one group: `hit` = the items that this lane's four entries w
// match, `items` = the OR over the lanes.  Positions run lane-major (lane l holds pos0 +
// 4 l .. + 3).  A ballot per new item, or a bit-matrix transpose where there are many, hands
// lane r the lanes that hit item r; it takes the lowest of them, fetches that lane's four
// words and records the first that holds the item: one conflict-free atomicMin a lane,
// however dense the hits.
__device__ __forceinline__ void record_items(uint32_t hit, uint32_t items, uint4 w4, const uint8_t* P,
                                             uint32_t* best, uint32_t pos0, int lane)
{
    uint32_t lanes = 0;
    if (__popc(items) > 16) {
        lanes = transpose32(hit, lane);
    } else {
        for (uint32_t t = items; t; t &= t - 1) {
            const int r = __ffs(t) - 1;
            const uint32_t b = __ballot_sync(0xffffffffu, (hit >> r) & 1u);
            if (lane == r) lanes = b;
        }
    }
    const int src = lanes ? __ffs(lanes) - 1 : 0;
    const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
    const uint32_t lane4 = (uint32_t)lane * 4u;
    int u = 3;
#pragma unroll
    for (int v = 3; v >= 0; --v) {
        uint32_t m = 0xffffffffu;
#pragma unroll
        for (int j = 0; j < 4; ++j) m &= *(const uint32_t*)(P + __byte_perm(w[v], lane4, 0x5504u + 0x10u * j));
        if ((__shfl_sync(0xffffffffu, m, src) >> lane) & 1u) u = v;
    }
    if (lanes) atomicMin(best + lane, pos0 + 4 * src + u);
}

// Block (c, node i) = blockIdx.x = c * n + i, item set blockIdx.y: items 32 G y .. 32 G y +
// 32 G - 1 of node i, stages c, c + nchunk, c + 2 nchunk, .. of the node's list (sorted
// mode: stages c per .. c per + per - 1).  Eight
// consumer warps and one producer warp: consumer warp w tests entries w * 256 .. w * 256 +
// 255 of every stage, 128 a step, so each warp walks its entries in increasing sorted
// position; the producer refills a stage as soon as every consumer has released it (an
// empty mbarrier per stage), so no consumer waits for a refill.
//
// With contiguous chunks the lower blocks of a full pass test all their items although the
// top one finds most of them.  Round-robin stages, the recording of a step's items by one
// atomicMin a lane and the producer's early end of its trades took the full pass at n = 60
// from 154 to 60 us for 256 orders and from 533 to 164 for 777.  The sorted mode keeps
// contiguous chunks (its lower blocks stop as soon as the top one has found everything, and
// every block that holds some of the top pays for its dense hits): 83 -> 36 us and 132 -> 70
// by the recording alone.
template <int G, bool CUT>
__global__ void __launch_bounds__(SL_THREADS) k_scan_sliced(SlicedArgs A)
{
    extern __shared__ __align__(128) uint8_t smem[];
    uint32_t* s_ent = (uint32_t*)smem;                                            // [STAGES][SUB]
    // P[v][g] for lane l at word (g / 2) * ROWS * 64 + v * 64 + (g % 2) * 32 + l: a row of
    // 256 bytes per node, so an entry's byte v and the lane's offset make the row address
    // in one byte permute
    __shared__ __align__(256) uint32_t s_Pst[sl_static_p(G) ? sl_p_bytes(G) / 4 : 1];
    uint32_t* s_P = sl_static_p(G) ? s_Pst : s_ent + SL_STAGES * SL_SUB;
    uint32_t* s_best = s_ent + SL_STAGES * SL_SUB + (sl_static_p(G) ? 0 : sl_p_bytes(G) / 4);   // [32 G]
    uint64_t* bar = (uint64_t*)(s_best + 32 * G);                                 // full, per stage
    uint64_t* ebar = bar + SL_STAGES;                                             // empty, per stage
    int* s_flags = (int*)(ebar + SL_STAGES);                                      // abort, first stage not issued, done
    uint32_t* s_skip = (uint32_t*)(s_flags + 4);                                  // [G]

    const int node = blockIdx.x % A.n;
    const int chunk = blockIdx.x / A.n;
    const int cnt = (int)A.list_count[node];
    const int g0 = blockIdx.y * 32 * G;
    if (g0 >= cnt) return;                                                        // block-uniform
    int64_t end = A.S;
    if (CUT) end = min(end, (int64_t)A.spos[(size_t)node * A.Sp] + 1);            // the empty set's position
    const int total = (int)((end + SL_SUB - 1) / SL_SUB);                         // the node's stages
    const int first = CUT ? chunk * A.per : chunk, stride = CUT ? 1 : A.nchunk;   // this block's
    if (first >= total) return;
    const int nsub = CUT ? min(A.per, total - first) : (total - first + stride - 1) / stride;
    auto stage_base = [&](int it) { return ((int64_t)it * stride + first) * SL_SUB; };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nvalid = min(cnt - g0, 32 * G);
    const bool producer = warp == SL_CWARPS;
    const uint32_t* src = A.sset + (size_t)node * A.Ssp;
    uint64_t pol_stream = 0;
    // the producer stages `it` into buffer st: always a whole stage (the row stride Ssp is
    // a whole number of stages).  Words past S are SSET_NEVER; in the sorted mode the
    // last stage may run past the empty set's position, and those entries cannot win
    // (the empty set, in the same stage, is consistent with every item and ranks above
    // them), so no lane needs a bounds test.
    auto issue = [&](int it, int st) {
        mbar_arrive_expect_tx(&bar[st], SL_SUB * 4u);
        bulk_g2s(s_ent + st * SL_SUB, src + stage_base(it), SL_SUB * 4u, &bar[st], pol_stream);
    };

    if (producer) {
        // items that hold a position above this block's first stage already (from blocks that
        // ran before it) are not tested; then the first copies go out while the consumers
        // set up
        int pre = 0;
        for (int g = 0; g < G; ++g) {
            const int item = g0 + 32 * g + lane;
            const bool done = item < cnt && *(volatile const uint32_t*)&A.list_best[(size_t)node * A.cap + item] <
                                                (uint32_t)stage_base(0);
            const uint32_t d = __ballot_sync(0xffffffffu, done);
            if (lane == 0) s_skip[g] = d;
            pre += __popc(d);
        }
        if (lane == 0) {
            s_flags[0] = 0;                                                       // abort
            s_flags[1] = 0x7fffffff;                                              // first stage never issued
            s_flags[2] = CUT && pre == nvalid;                                    // nothing to do
            pol_stream = l2_policy_evict_first();
            for (int s = 0; s < SL_STAGES; ++s) {
                mbar_init(&bar[s], 1);
                mbar_init(&ebar[s], SL_CWARPS);
            }
            fence_mbar_init();
            if (!s_flags[2])
                for (int it = 0; it < SL_STAGES && it < nsub; ++it) issue(it, it);
        }
    } else {
        // the items' predecessor words, the consumer warps spread over (group, node): rows of
        // the nodes from ballots of the group's masks, row 64 all ones, row 65 zero
        constexpr int PARTS = SL_CWARPS / G;                                      // warps a group
        const int g = warp / PARTS, part = warp % PARTS;
        const int item = g0 + g * 32 + lane;
        const uint64_t pc = item < cnt ? A.list_pc[(size_t)node * A.cap + item] : 0ull;
#pragma unroll 4
        for (int v = part; v < A.n; v += PARTS) {
            const bool bit = v != node && ((pc >> (v - (v > node))) & 1ull);
            s_P[Pw(g, v) + lane] = __ballot_sync(0xffffffffu, bit);
        }
        if (part == 0) {
            s_P[Pw(g, 64) + lane] = 0xffffffffu;
            s_P[Pw(g, 65) + lane] = 0u;
        }
        for (int j = threadIdx.x; j < 32 * G; j += 32 * SL_CWARPS) s_best[j] = SPOS_NONE;
    }
    __syncthreads();
    if (CUT && s_flags[2]) return;                                      // block-uniform; nothing issued

    if (producer) {
        // Lane 0 refills each stage once every consumer has released it.  Then, while the
        // copy is in flight, the whole warp trades positions with the node's other blocks: it
        // publishes this block's new positions (atomicMin), marks as skipped every item that
        // holds a position above the next stage, and (sorted mode) sees whether all of them
        // hold one above the stage that would be issued next.
        int issued = min(SL_STAGES, nsub);
        bool all_done = false, settled = false;
        uint32_t pub[G], known[G];         // last published position; items already skipped
#pragma unroll
        for (int g = 0; g < G; ++g) {
            pub[g] = SPOS_NONE;
            known[g] = s_skip[g];
        }
        for (int it = 0; it + SL_STAGES < nsub; ++it) {
            const int st = it % SL_STAGES;
            int go = 1;
            if (lane == 0) {
                if (*(volatile int*)&s_flags[0]) {
                    go = 0;
                } else if (!mbar_wait_bounded(&ebar[st], (uint32_t)((it / SL_STAGES) & 1), WAIT_TIMEOUT_NS)) {
                    *(volatile int*)&s_flags[0] = 1;
                    atomicOr(A.status, STATUS_TIMEOUT);
                    go = 0;
                } else if (CUT && all_done) {
                    // no unread entry can win; release the consumers of this buffer's next
                    // phase without a copy
                    *(volatile int*)&s_flags[1] = it + SL_STAGES;
                    mbar_arrive(&bar[st]);
                    issued = it + SL_STAGES + 1;
                    go = 0;
                } else {
                    issue(it + SL_STAGES, st);
                    issued = it + SL_STAGES + 1;
                }
            }
            if (!__shfl_sync(0xffffffffu, go, 0)) break;
            if (settled) continue;         // (a trade's round trip would outlast a stage's copy)
            // every load first (one round trip for all groups), then the updates
            uint32_t mine[G], other[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int item = g0 + 32 * g + lane;
                const bool live = item < cnt && !((known[g] >> lane) & 1u);
                mine[g] = live ? *(volatile const uint32_t*)&s_best[g * 32 + lane] : SPOS_NONE;
                other[g] = live ? *(volatile const uint32_t*)&A.list_best[(size_t)node * A.cap + item] : SPOS_NONE;
            }
            const uint32_t next = (uint32_t)stage_base(it + 1), after = (uint32_t)stage_base(it + 1 + SL_STAGES);
            bool open = false;             // an item that the stage to be issued next may serve
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int item = g0 + 32 * g + lane;
                if (mine[g] < pub[g] && mine[g] < other[g]) {
                    atomicMin(&A.list_best[(size_t)node * A.cap + item], mine[g]);
                    pub[g] = mine[g];
                }
                const uint32_t pos = min(mine[g], other[g]);
                open |= item < cnt && !((known[g] >> lane) & 1u) && pos >= after;
                const uint32_t bits = __ballot_sync(0xffffffffu, pos < next);
                known[g] |= bits;
                if (lane == 0 && bits) *(volatile uint32_t*)&s_skip[g] |= bits;
            }
            all_done = !__any_sync(0xffffffffu, open);
            settled = true;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int nv = min(max(cnt - g0 - 32 * g, 0), 32);
                settled &= (known[g] | (nv >= 32 ? 0u : 0xffffffffu << nv)) == 0xffffffffu;
            }
        }
        if (lane == 0) {
            // no copy may still be in flight when the block's shared memory goes away
            for (int j = max(0, issued - SL_STAGES); j < issued; ++j)
                mbar_wait_bounded(&bar[j % SL_STAGES], (uint32_t)((j / SL_STAGES) & 1), WAIT_TIMEOUT_NS);
        }
    } else {
        uint32_t found[G];                 // items of group g this warp no longer tests
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int nv = min(max(cnt - g0 - 32 * g, 0), 32);
            found[g] = nv >= 32 ? 0u : (0xffffffffu << nv);
            found[g] |= s_skip[g];
        }
        const uint32_t lane4 = (uint32_t)lane * 4u;
        const uint8_t* Pb = (const uint8_t*)s_P;
        for (int it = 0; it < nsub; ++it) {
            const int st = it % SL_STAGES;
            const uint32_t parity = (uint32_t)((it / SL_STAGES) & 1);
            if (__shfl_sync(0xffffffffu, *(volatile int*)&s_flags[0], 0)) break;
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&bar[st], parity, WAIT_TIMEOUT_NS))) {
                if (lane == 0) {
                    *(volatile int*)&s_flags[0] = 1;
                    atomicOr(A.status, STATUS_TIMEOUT);
                }
                break;
            }
            if (CUT && it >= __shfl_sync(0xffffffffu, *(volatile int*)&s_flags[1], 0)) break;
            const int64_t base = stage_base(it) + warp * SL_PER_WARP;
            const uint4* E4 = (const uint4*)(s_ent + st * SL_SUB + warp * SL_PER_WARP);
            uint32_t all_found = 0xffffffffu;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                found[g] |= *(volatile const uint32_t*)&s_skip[g];
                all_found &= found[g];
            }
            if (all_found != 0xffffffffu) {
                // a step: 128 entries, four consecutive ones a lane (one 16-byte load); one
                // warp vote per step, then one warp-wide OR per group marks the step's new
                // items found (two records of an item in one step: the atomicMin keeps the
                // earlier position)
#pragma unroll 1
                for (int q = 0; q < SL_PER_WARP / 128; ++q) {
                    const uint4 w4 = E4[q * 32 + lane];
                    const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
                    // byte 1 = the parent's node id, byte 0 = this lane's offset: the byte
                    // address of P[v][g] minus the group's constant part
                    auto word = [&](uint32_t wu, uint32_t sel, int g) {
                        return *(const uint32_t*)(Pb + 4 * Pw(g, 0) + __byte_perm(wu, lane4, sel));
                    };
                    uint32_t raw[G];
#pragma unroll
                    for (int g = 0; g < G; ++g) raw[g] = 0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
#pragma unroll
                        for (int g = 0; g < G; ++g)
                            raw[g] |= word(w[u], 0x5504, g) & word(w[u], 0x5514, g) & word(w[u], 0x5524, g) &
                                      word(w[u], 0x5534, g);
                    }
                    uint32_t any = 0;
#pragma unroll
                    for (int g = 0; g < G; ++g) any |= raw[g] & ~found[g];
                    if (__any_sync(0xffffffffu, any != 0)) {
                        // rare past the top of a list, where one entry matches many orders
                        const uint32_t pos0 = (uint32_t)(base + q * 128);
#pragma unroll
                        for (int g = 0; g < G; ++g) {
                            const uint32_t hit = raw[g] & ~found[g];
                            const uint32_t items = __reduce_or_sync(0xffffffffu, hit);
                            if (!items) continue;                                 // warp-uniform
                            found[g] |= items;
                            record_items(hit, items, w4, Pb + 4 * Pw(g, 0), &s_best[g * 32], pos0, lane);
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&ebar[st]);
        }
    }
    __syncthreads();
    if (s_flags[0]) return;                                                       // block-uniform
    for (int j = threadIdx.x; j < nvalid; j += SL_THREADS) {
        const uint32_t b = s_best[j];
        if (b != SPOS_NONE) atomicMin(&A.list_best[(size_t)node * A.cap + g0 + j], b);
    }
}

// Launch shape: as many blocks as are resident at once (the occupancy calculator: threads,
// registers and shared memory), one wave of long blocks, so each block's set-up is paid
// once; the sorted mode counts on at least four stages a block over the nodes' live ranges
// [0, cut), and the blocks past a node's live stages leave at once.
template <int G, bool CUT>
static int sliced_launch(const bn_table* t, const uint32_t* list_count, const uint64_t* list_pc,
                         uint32_t* list_best, int cap, int sets, uint32_t* status, cudaStream_t s)
{
    static ContextOnce once;
    static int resident[64] = {0};
    const int d = device_id();
    const int rc = once_in_context(once, [&]() -> int {
        BN_CUDA(cudaFuncSetAttribute(k_scan_sliced<G, CUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sl_smem(G)));
        int nb = 0;
        BN_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_scan_sliced<G, CUT>, SL_THREADS, sl_smem(G)));
        if (d >= 0 && d < 64) resident[d] = std::max(1, nb);
        return BN_OK;
    });
    if (rc) return rc;
    const int per_sm = (d >= 0 && d < 64 && resident[d] > 0) ? resident[d] : 1;
    const int64_t want = (int64_t)sm_count() * per_sm;
    int64_t nchunk, per = 0;
    if (!CUT) {
        nchunk = std::max<int64_t>(1, want / ((int64_t)t->n * sets));
        nchunk = std::min<int64_t>(nchunk, (t->S + SL_SUB - 1) / SL_SUB);
    } else {
        int64_t live = 0, longest = 0;
        for (int i = 0; i < t->n; ++i) {
            live += t->cut[i];
            longest = std::max<int64_t>(longest, t->cut[i]);
        }
        const int64_t chunk = std::max<int64_t>(4 * SL_SUB, round_up((live * sets + want - 1) / want, SL_SUB));
        nchunk = (longest + chunk - 1) / chunk;
        per = chunk / SL_SUB;
    }
    SlicedArgs A{t->sset, t->spos, t->Sp, t->S, t->sset_stride, t->n, (int)nchunk, (int)per, list_count,
                 list_pc, list_best, cap, status};
    dim3 grid((unsigned)(nchunk * t->n), (unsigned)sets);
    k_scan_sliced<G, CUT><<<grid, SL_THREADS, sl_smem(G), s>>>(A);
    BN_LAUNCH_CHECK("k_scan_sliced");
    return BN_OK;
}

int launch_scan_sliced(const bn_table* t, const uint32_t* list_count, const uint64_t* list_pc, uint32_t* list_best,
                       int cap, bool cut, uint32_t* status, cudaStream_t s)
{
    if (!t->sset) return set_error(BN_EUNSUPPORTED, "sliced scan: needs k <= 4 (k = %d)", t->k);
    if (cap < 1) return BN_OK;
    const int per = std::min(cap, 256);
    const int G = per <= 32 ? 1 : (per <= 64 ? 2 : (per <= 128 ? 4 : 8));
    const int sets = (cap + 32 * G - 1) / (32 * G);
    if (sets > 65535) return set_error(BN_EUNSUPPORTED, "sliced scan: %d items per node (at most %d)", cap, 65535 * 256);
#define BN_SL(GG)                                                                                               \
    return cut ? sliced_launch<GG, true>(t, list_count, list_pc, list_best, cap, sets, status, s)               \
               : sliced_launch<GG, false>(t, list_count, list_pc, list_best, cap, sets, status, s)
    switch (G) {
        case 1: BN_SL(1);
        case 2: BN_SL(2);
        case 4: BN_SL(4);
        default: BN_SL(8);
    }
#undef BN_SL
}

}  // namespace bn
