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
// leaving their terms out changes the result by less than its rounding does.  A warp owns a
// run of a node's list for up to SUM_OB orders; runs outside every order's window are
// skipped.  Partials merge in a fixed order, so results are deterministic for a given
// launch shape.
//
// The cost is the exponentials: most consistent entries lie within D of the best, and an
// FP64 exp10 is some thirty instructions on a pipe that takes 64 cycles for a warp's one.  So
// an entry's 10^(entry - ref) is formed once for all orders of the block, in 64-bit integer
// arithmetic (exp10_fx), relative to the first entry ref of a stretch of the list no longer
// than one decade; a consistent order adds it as an integer, and only the stretch's sums
// are brought to FP64 and scaled by 10^(ref - m) -- one exp10 on eight lanes per 1,024
// entries.  Every term is good to 2^-55 of itself.  Steps of 32 entries that
// span more than a decade or two binades of scores (short lists, the ends of long ones)
// take FP64 exponentials per (entry, order).  8 orders at n = 60: 484 us with one exp10 per
// (entry, order), 208 so; 6.1 ms with every entry's.
#include <algorithm>
#include <cmath>

#include "bn_fx.cuh"
#include "bn_table.cuh"

namespace bn {

static constexpr int SUM_OB = 8;          // orders per block
static constexpr int SUM_THREADS = 256;
static constexpr int SUM_WARPS = SUM_THREADS / 32;
static constexpr int SUM_BATCH = 256;     // orders whose partials are held at a time
static constexpr int SUM_SLICE = 65535 * 256;   // orders whose lists are: as many as every scan's grid takes

struct SumScanArgs {
    const int64_t* keys;
    const uint64_t* pst;
    const uint32_t* srank;
    int64_t S, Sp;
    int n, B, b0, b1;                     // all orders; the batch [b0, b1)
    int run;                              // sorted positions per warp (256 or 1,024)
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

static __device__ const Exp2Tables g_exp2 = make_exp2();

__global__ void __launch_bounds__(SUM_THREADS) k_sum_window(SumScanArgs A)
{
    __shared__ uint64_t s_T[3][64];
    __shared__ double s_slow[SUM_WARPS][SUM_OB][32];      // FP64 terms of a lane's wide steps
    __shared__ uint64_t s_npc[SUM_OB];
    __shared__ int64_t s_thr[SUM_OB];
    __shared__ double s_m[SUM_OB], s_s[SUM_WARPS][SUM_OB];
    __shared__ uint32_t s_p0[SUM_OB];
    const int chunk = blockIdx.x, node = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b0 = A.b0 + (int)blockIdx.z * SUM_OB, nb = min(SUM_OB, A.b1 - b0);
    if (tid < 192) s_T[tid >> 6][tid & 63] = g_exp2.v[tid >> 6][tid & 63];
    if (tid < SUM_OB) {
        uint32_t p0 = SPOS_NONE;
        int64_t thr = 0x7fffffffffffffffLL;
        double m = -INFINITY;
        uint64_t npc = ~0ull;
        if (tid < nb) {
            const size_t at = (size_t)node * A.B + b0 + tid;
            p0 = A.list_best[at];
            if ((int64_t)p0 >= A.S) p0 = SPOS_NONE;                     // only after a timed-out scan
            else m = key_to_double(sorted_key(A, node, p0));
            // (a best entry of -inf: every consistent one is, the sum stays empty)
            if (m > -INFINITY) {
                thr = double_to_key(__dsub_rn(m, A.reach));
                npc = ~A.list_pc[at];
            } else {
                p0 = SPOS_NONE;
            }
        }
        s_npc[tid] = npc;
        s_p0[tid] = p0;
        s_thr[tid] = thr;
        s_m[tid] = m;
    }
    __syncthreads();
    uint32_t first = SPOS_NONE;
    int64_t low = 0x7fffffffffffffffLL;
    uint64_t npc[SUM_OB];
#pragma unroll
    for (int b = 0; b < SUM_OB; ++b) {
        first = min(first, s_p0[b]);
        low = min(low, s_thr[b]);
        npc[b] = s_npc[b];
    }
    const int64_t e0 = ((int64_t)chunk * SUM_WARPS + warp) * A.run, e1 = min(e0 + A.run, A.S);
    double acc = 0.0;                                     // lane b: order b's sum over this run
    if (e0 < e1 && e1 > (int64_t)first && sorted_key(A, node, e0) >= low) {          // warp-uniform
        const double my_m = lane < SUM_OB ? s_m[lane] : 0.0;
        uint64_t sum[SUM_OB];
#pragma unroll
        for (int b = 0; b < SUM_OB; ++b) sum[b] = 0;
        int64_t ref = 0;
        int ref_exp = 0, held = 0;                        // steps summed relative to ref
        bool slow_used = false;
        // the stretch's sums over the warp, 22 bits at a time, to lane b's FP64 sum
        auto flush = [&]() {
            uint64_t mine = 0;
            uint32_t top = 0;
#pragma unroll
            for (int b = 0; b < SUM_OB; ++b) {
                const uint32_t l0 = __reduce_add_sync(0xffffffffu, (uint32_t)sum[b] & 0x3fffffu);
                const uint32_t l1 = __reduce_add_sync(0xffffffffu, (uint32_t)(sum[b] >> 22) & 0x3fffffu);
                const uint32_t l2 = __reduce_add_sync(0xffffffffu, (uint32_t)(sum[b] >> 44));
                if (lane == b) {
                    mine = ((uint64_t)l1 << 22) + l0;
                    top = l2;
                }
                sum[b] = 0;
            }
            if (lane < nb && my_m > -INFINITY) {
                const double t = __fma_rn((double)top, 0x1p44, (double)mine) * 0x1p-59;
                if (t != 0.0) acc += t * exp10(key_to_double(ref) - my_m);
            }
            held = 0;
        };
        for (int64_t p = e0 + lane; p - lane < e1; p += 32) {
            uint32_t ok = 0;
            int64_t key = KEY_NONE;
            const bool in = p < e1;
            if (in) {
                const uint32_t r = A.srank[(size_t)node * A.Sp + p];
                const uint64_t mask = A.pst[r];
                key = A.keys[(size_t)node * A.Sp + r];
#pragma unroll
                for (int b = 0; b < SUM_OB; ++b) ok |= (uint32_t)((mask & npc[b]) == 0ull) << b;
            }
            if (!__any_sync(0xffffffffu, ok != 0)) continue;
            const int last = (int)min((int64_t)31, e1 - 1 - (p - lane));
            const int64_t k0 = __shfl_sync(0xffffffffu, key, 0), kl = __shfl_sync(0xffffffffu, key, last);
            // one binade and at most a decade between k0 and kl: key differences are
            // differences of the scores in units of their last place, 2^(exp - 1075)
            const uint64_t bits0 = bits_from_key(k0), bitsl = bits_from_key(kl);
            const int ex = (int)(bits0 >> 52) & 0x7ff;
            const bool one = (bits0 >> 52) == (bitsl >> 52) && ex > 1015 && ex < 1075;
            const uint64_t decade = 1ull << (1075 - min(max(ex, 1015), 1075));
            if (one && (uint64_t)(k0 - kl) <= decade) {
                const int se = (int)(bits0 >> 52);                           // sign and exponent
                if (held && (held == 32 || se != ref_exp || (uint64_t)(ref - kl) > decade)) flush();
                if (!held) {
                    ref = k0;
                    ref_exp = se;
                }
                ++held;
                const uint64_t E = in ? exp10_fx((uint64_t)(ref - key) << (ex - 1015), s_T) : 0ull;
#pragma unroll
                for (int b = 0; b < SUM_OB; ++b)
                    if ((ok >> b) & 1u) sum[b] += E;
            } else {
                if (!slow_used) {
#pragma unroll
                    for (int b = 0; b < SUM_OB; ++b) s_slow[warp][b][lane] = 0.0;
                    slow_used = true;
                }
                // each lane its remaining orders in turn, those whose window holds the entry
#pragma unroll
                for (int b = 0; b < SUM_OB; ++b)
                    if (key < s_thr[b]) ok &= ~(1u << b);
                while (__any_sync(0xffffffffu, ok != 0)) {
                    if (ok) {
                        const int b = __ffs((int)ok) - 1;
                        ok &= ok - 1;
                        s_slow[warp][b][lane] += exp10(key_to_double(key) - s_m[b]);
                    }
                }
            }
        }
        if (held) flush();
        if (slow_used) {
            __syncwarp();
            if (lane < nb)
                for (int l = 0; l < 32; ++l) acc += s_slow[warp][lane][l];
        }
    }
    if (lane < SUM_OB) s_s[warp][lane] = acc;
    __syncthreads();
    if (tid < nb) {
        double s = 0.0;
        for (int w = 0; w < SUM_WARPS; ++w) s += s_s[w][tid];
        A.part[((size_t)node * (A.b1 - A.b0) + (b0 - A.b0) + tid) * A.nchunk + chunk] = s;
    }
}

// One block an order: a warp per node sums the chunks (lane-strided, then a fixed tree), a
// thread per node takes the logarithm, one adds the node terms in ascending node id.
__global__ void __launch_bounds__(SUM_THREADS) k_sum_finish(SumScanArgs A, double* __restrict__ node_score,
                                                            double* __restrict__ order_score)
{
    __shared__ double s_v[MAXN];
    const int b = A.b0 + blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double top = 0.0;
    if (tid < A.n) {
        uint32_t best = A.list_best[(size_t)tid * A.B + b];
        if ((int64_t)best >= A.S) best = 0;                            // only after a timed-out scan
        top = key_to_double(sorted_key(A, tid, best));
    }
    for (int i = warp; i < A.n; i += SUM_WARPS) {
        const double* p = A.part + ((size_t)i * (A.b1 - A.b0) + blockIdx.x) * A.nchunk;
        double s = 0.0;
        for (int c = lane; c < A.nchunk; c += 32) s += p[c];
#pragma unroll
        for (int off = 16; off; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (lane == 0) s_v[i] = s;
    }
    __syncthreads();
    if (tid < A.n) {
        const double v = top + log10(s_v[tid]);
        s_v[tid] = v;
        if (node_score) node_score[(size_t)b * A.n + tid] = v;
    }
    __syncthreads();
    if (tid == 0 && order_score) {
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
    // short runs where there are few: a warp's steps are its latency
    const int run = t->S >= 65536 ? 1024 : 256;
    const int nchunk = (int)((t->S + SUM_WARPS * run - 1) / (SUM_WARPS * run));
    const int batch = std::min(B, SUM_BATCH), slice = std::min(B, SUM_SLICE);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = (size_t)round_up((int64_t)(off + bytes), 256);
        return o;
    };
    const size_t o_orders = take(mem == BN_MEM_HOST ? (size_t)B * n : 0);
    const size_t o_pc = take(sizeof(uint64_t) * (size_t)n * slice);
    const size_t o_best = take(sizeof(uint32_t) * (size_t)n * slice);
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
    const double reach = std::log10((double)t->S) + 60.0 * 0.30102999566398120;
    for (int64_t s0 = 0; s0 < B; s0 += slice) {
        const int Bs = (int)std::min<int64_t>(slice, B - s0);
        int rc = launch_pred_lists(d_orders + (size_t)s0 * n, Bs, n, d_pc, d_best, d_cnt, d_st, s);
        if (rc) return rc;
        // the best consistent entries, by the fastest scan the table has (all give the same)
        if (t->amask) rc = launch_scan_pruned(t, d_cnt, d_pc, d_best, Bs, s);
        else if (t->sset) rc = launch_scan_sliced(t, d_cnt, d_pc, d_best, Bs, true, d_st, s);
        else rc = launch_scan(t, plan_scan(t, Bs), d_cnt, d_pc, d_best, Bs, d_st, s);
        if (rc) return rc;
        for (int b0 = 0; b0 < Bs; b0 += batch) {
            SumScanArgs A{t->keys, t->pst, t->srank, t->S, t->Sp, n, Bs, b0, std::min(Bs, b0 + batch), run, nchunk, reach,
                          d_pc, d_best, d_part};
            const int groups = (A.b1 - b0 + SUM_OB - 1) / SUM_OB;
            k_sum_window<<<dim3((unsigned)nchunk, (unsigned)n, (unsigned)groups), SUM_THREADS, 0, s>>>(A);
            BN_LAUNCH_CHECK("k_sum_window");
            k_sum_finish<<<(unsigned)(A.b1 - b0), SUM_THREADS, 0, s>>>(A, d_ns ? d_ns + (size_t)s0 * n : nullptr,
                                                                      d_os ? d_os + s0 : nullptr);
            BN_LAUNCH_CHECK("k_sum_finish");
        }
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
