// bn_sum.cu -- the sum-based order score of the prior scorer the paper compares its own
// against (Sec. III.B): log10 of the sum over every graph consistent with an order of
// 10^(graph score), which factorises over nodes into
//     sum_i log10 sum_{parent sets pi of i drawn from its predecessors} 10^entry(i, pi).
// The paper's argument against it is its cost (exponentials and logarithms instead of
// comparisons) and that its best order need not carry the best graph; this scan makes the
// first point measurable on the same table and the same hardware.
//
// Only the entries near the top of a node's list count.  The best consistent entry m of an
// (order, node) comes from the max-based scan; then the entries are walked by sorted
// position (score descending) from the best one down to m - D, D = log10(S 2^60) decades:
// the entries below sum to less than S 10^-D = 2^-60 of the sum, 1/128 of its last bit, so
// leaving their terms out changes the result by less than its rounding does.  A block owns a
// chunk of a node's list and up to SUM_OB orders; blocks outside every order's window
// leave at once.  The shift is the same for every partial sum of an (order, node), and the
// partials merge in a fixed order, so results are deterministic for a given launch shape.
#include <algorithm>
#include <cmath>

#include "bn_table.cuh"

namespace bn {

static constexpr int SUM_OB = 8;          // orders per block
static constexpr int SUM_THREADS = 256;
static constexpr int SUM_WARPS = SUM_THREADS / 32;
static constexpr int SUM_CHUNK = 2048;    // sorted positions per block
static constexpr int SUM_BATCH = 256;     // orders whose partials are held at a time

struct SumScanArgs {
    const int64_t* keys;
    const uint64_t* pst;
    const uint32_t* srank;
    int64_t S, Sp;
    int n, B, b0, b1;                     // all orders; the batch [b0, b1)
    int nchunk;
    double reach;                         // D
    const uint64_t* list_pc;              // [n][B] candidate-space predecessor masks
    const uint32_t* list_best;            // [n][B] sorted position of the best consistent entry
    double* part;                         // [n][b1 - b0][nchunk] sums of 10^(entry - best)
};

__device__ __forceinline__ int64_t sorted_key(const SumScanArgs& A, int i, int64_t p)
{
    return A.keys[(size_t)i * A.Sp + A.srank[(size_t)i * A.Sp + p]];
}

// Terms wait in a short queue per (warp, order) so that the exponentials -- the cost of this
// score: some forty FP64 operations each -- run on full warps: at n = 60 about one entry in
// five is consistent with an order, and a warp takes the exponential for one lane as for 32.
__global__ void __launch_bounds__(SUM_THREADS) k_sum_window(SumScanArgs A)
{
    __shared__ double s_q[SUM_WARPS][SUM_OB][64];
    __shared__ uint64_t s_npc[SUM_OB];
    __shared__ int64_t s_thr[SUM_OB];
    __shared__ double s_m[SUM_OB], s_s[SUM_WARPS][SUM_OB];
    __shared__ uint32_t s_p0[SUM_OB];
    const int chunk = blockIdx.x, node = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b0 = A.b0 + (int)blockIdx.z * SUM_OB, nb = min(SUM_OB, A.b1 - b0);
    const int64_t e0 = (int64_t)chunk * SUM_CHUNK, e1 = min(e0 + SUM_CHUNK, A.S);
    if (tid < SUM_OB) {
        uint32_t p0 = SPOS_NONE;
        int64_t thr = 0x7fffffffffffffffLL;
        double m = -INFINITY;
        uint64_t npc = ~0ull;
        if (tid < nb) {
            const size_t at = (size_t)node * A.B + b0 + tid;
            npc = ~A.list_pc[at];
            p0 = A.list_best[at];
            if ((int64_t)p0 >= A.S) p0 = SPOS_NONE;                     // only after a timed-out scan
            else m = key_to_double(sorted_key(A, node, p0));
            // (a best entry of -inf: every consistent one is, the sum stays empty)
            if (m > -INFINITY) thr = double_to_key(__dsub_rn(m, A.reach));
            else p0 = SPOS_NONE;
        }
        s_npc[tid] = npc;
        s_p0[tid] = p0;
        s_thr[tid] = thr;
        s_m[tid] = m;
    }
    __syncthreads();
    uint32_t first = SPOS_NONE;
    int64_t low = 0x7fffffffffffffffLL;
#pragma unroll
    for (int b = 0; b < SUM_OB; ++b) {
        first = min(first, s_p0[b]);
        low = min(low, s_thr[b]);
    }
    double acc[SUM_OB];
#pragma unroll
    for (int b = 0; b < SUM_OB; ++b) acc[b] = 0.0;
    if (e1 > (int64_t)first && sorted_key(A, node, e0) >= low) {        // block-uniform
        int cnt[SUM_OB];
#pragma unroll
        for (int b = 0; b < SUM_OB; ++b) cnt[b] = 0;
        const uint32_t lt = (1u << lane) - 1u;
        for (int64_t p = e0 + tid; p - lane < e1; p += SUM_THREADS) {
            uint32_t ok = 0;
            uint32_t r = 0;
            if (p < e1) {
                r = A.srank[(size_t)node * A.Sp + p];
                const uint64_t mask = A.pst[r];
#pragma unroll
                for (int b = 0; b < SUM_OB; ++b)
                    ok |= (uint32_t)((uint32_t)p >= s_p0[b] && (mask & s_npc[b]) == 0ull) << b;
            }
            const int64_t key = ok ? A.keys[(size_t)node * A.Sp + r] : KEY_NONE;
            const double v = key_to_double(key);
#pragma unroll
            for (int b = 0; b < SUM_OB; ++b) {
                const bool take = ((ok >> b) & 1u) && key >= s_thr[b];
                const uint32_t bal = __ballot_sync(0xffffffffu, take);
                if (bal) {
                    double* q = s_q[warp][b];
                    if (take) q[cnt[b] + __popc(bal & lt)] = __dsub_rn(v, s_m[b]);
                    cnt[b] += __popc(bal);
                    if (cnt[b] >= 32) {
                        __syncwarp();
                        acc[b] += exp10(q[lane]);
                        cnt[b] -= 32;
                        const double rest = q[32 + lane];
                        __syncwarp();
                        if (lane < cnt[b]) q[lane] = rest;
                        __syncwarp();
                    }
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < SUM_OB; ++b)
            if (lane < cnt[b]) acc[b] += exp10(s_q[warp][b][lane]);
    }
#pragma unroll
    for (int b = 0; b < SUM_OB; ++b) {
        double s = acc[b];
#pragma unroll
        for (int off = 16; off; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (lane == 0) s_s[warp][b] = s;
    }
    __syncthreads();
    if (tid < nb) {
        double s = 0.0;
        for (int w = 0; w < SUM_WARPS; ++w) s += s_s[w][tid];
        A.part[((size_t)node * (A.b1 - A.b0) + (b0 - A.b0) + tid) * A.nchunk + chunk] = s;
    }
}

// One block an order: a warp per node sums the chunks (lane-strided, then a fixed tree), the
// node terms, then their sum in ascending node id.
__global__ void __launch_bounds__(SUM_THREADS) k_sum_finish(SumScanArgs A, double* __restrict__ node_score,
                                                            double* __restrict__ order_score)
{
    __shared__ double s_v[MAXN];
    const int b = A.b0 + blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < A.n; i += SUM_WARPS) {
        const double* p = A.part + ((size_t)i * (A.b1 - A.b0) + blockIdx.x) * A.nchunk;
        double s = 0.0;
        for (int c = lane; c < A.nchunk; c += 32) s += p[c];
#pragma unroll
        for (int off = 16; off; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (lane == 0) {
            uint32_t best = A.list_best[(size_t)i * A.B + b];
            if ((int64_t)best >= A.S) best = 0;                        // only after a timed-out scan
            const double v = key_to_double(sorted_key(A, i, best)) + log10(s);
            s_v[i] = v;
            if (node_score) node_score[(size_t)b * A.n + i] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && order_score) {
        double total = 0.0;
        for (int i = 0; i < A.n; ++i) total += s_v[i];
        order_score[b] = total;
    }
}

}  // namespace bn

using namespace bn;

extern "C" int bn_score_orders_sum(const bn_table* t, const uint8_t* orders, int B, double* order_score,
                                   double* node_score, int mem, void* stream)
{
    set_error(BN_OK, "");
    if (!t) return set_error(BN_EINVAL, "bn_score_orders_sum: NULL table");
    if (B < 0) return set_error(BN_EINVAL, "bn_score_orders_sum: B=%d", B);
    if (mem != BN_MEM_HOST && mem != BN_MEM_DEVICE) return set_error(BN_EINVAL, "bn_score_orders_sum: bad mem");
    if (B == 0) return BN_OK;
    if (!orders) return set_error(BN_EINVAL, "bn_score_orders_sum: orders is NULL");
    cudaStream_t s = (cudaStream_t)stream;
    const int n = t->n;
    const int nchunk = (int)((t->S + SUM_CHUNK - 1) / SUM_CHUNK);
    const int batch = std::min(B, SUM_BATCH);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = (size_t)round_up((int64_t)(off + bytes), 256);
        return o;
    };
    const size_t o_orders = take(mem == BN_MEM_HOST ? (size_t)B * n : 0);
    const size_t o_pc = take(sizeof(uint64_t) * (size_t)n * B);
    const size_t o_best = take(sizeof(uint32_t) * (size_t)n * B);
    const size_t o_cnt = take(sizeof(uint32_t) * n);
    const size_t o_st = take(sizeof(uint32_t));
    const size_t o_part = take(sizeof(double) * (size_t)n * batch * nchunk);
    const size_t o_os = take(mem == BN_MEM_HOST && order_score ? sizeof(double) * B : 0);
    const size_t o_ns = take(mem == BN_MEM_HOST && node_score ? sizeof(double) * (size_t)B * n : 0);
    uint8_t* base = nullptr;
    cudaError_t e = dev_alloc((void**)&base, off, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(BN_ENOMEM, "bn_score_orders_sum: scratch of %zu bytes: %s", off, cudaGetErrorString(e));
    }
    struct Free {
        uint8_t* p;
        cudaStream_t s;
        ~Free() { dev_free(p, s); }
    } fr{base, s};
    const uint8_t* d_orders = orders;
    if (mem == BN_MEM_HOST) {
        BN_CUDA(cudaMemcpyAsync(base + o_orders, orders, (size_t)B * n, cudaMemcpyHostToDevice, s));
        d_orders = base + o_orders;
    }
    uint64_t* d_pc = (uint64_t*)(base + o_pc);
    uint32_t* d_st = (uint32_t*)(base + o_st);
    double* d_part = (double*)(base + o_part);
    uint32_t* d_best = (uint32_t*)(base + o_best);
    uint32_t* d_cnt = (uint32_t*)(base + o_cnt);
    double* d_os = mem == BN_MEM_HOST ? (order_score ? (double*)(base + o_os) : nullptr) : order_score;
    double* d_ns = mem == BN_MEM_HOST ? (node_score ? (double*)(base + o_ns) : nullptr) : node_score;
    BN_CUDA(cudaMemsetAsync(d_st, 0, sizeof(uint32_t), s));
    int rc = launch_pred_lists(d_orders, B, n, d_pc, d_best, d_cnt, d_st, s);
    if (rc) return rc;
    // the best consistent entries, by the fastest scan the table has (all give the same)
    if (t->amask) rc = launch_scan_pruned(t, d_cnt, d_pc, d_best, B, s);
    else if (t->sset) rc = launch_scan_sliced(t, d_cnt, d_pc, d_best, B, true, d_st, s);
    else rc = launch_scan(t, plan_scan(t, B), d_cnt, d_pc, d_best, B, d_st, s);
    if (rc) return rc;
    const double reach = std::log10((double)t->S) + 60.0 * 0.30102999566398120;
    for (int b0 = 0; b0 < B; b0 += batch) {
        SumScanArgs A{t->keys, t->pst, t->srank, t->S, t->Sp, n, B, b0, std::min(B, b0 + batch), nchunk, reach, d_pc,
                      d_best, d_part};
        const int groups = (A.b1 - b0 + SUM_OB - 1) / SUM_OB;
        k_sum_window<<<dim3((unsigned)nchunk, (unsigned)n, (unsigned)groups), SUM_THREADS, 0, s>>>(A);
        BN_LAUNCH_CHECK("k_sum_window");
        k_sum_finish<<<(unsigned)(A.b1 - b0), SUM_THREADS, 0, s>>>(A, d_ns, d_os);
        BN_LAUNCH_CHECK("k_sum_finish");
    }
    if (mem == BN_MEM_HOST) {
        if (order_score) BN_CUDA(cudaMemcpyAsync(order_score, d_os, sizeof(double) * B, cudaMemcpyDeviceToHost, s));
        if (node_score)
            BN_CUDA(cudaMemcpyAsync(node_score, d_ns, sizeof(double) * (size_t)B * n, cudaMemcpyDeviceToHost, s));
    }
    uint32_t st = 0;
    BN_CUDA(cudaMemcpyAsync(&st, d_st, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    BN_CUDA(cudaStreamSynchronize(s));
    if (st & STATUS_BADINPUT) return set_error(BN_EINVAL, "bn_score_orders_sum: an order is not a permutation of 0..n-1");
    if (st & STATUS_TIMEOUT) return set_error(BN_ETIMEOUT, "bn_score_orders_sum: a bounded device wait expired");
    return BN_OK;
}
