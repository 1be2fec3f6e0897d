// bn_joint_tc.cu -- joint count tables of five and four nodes on the tensor cores.
//
// The count of a cell of the joint table of U = {a < b < c < d < e} is the number of rows in
// which (a, b, c) are in one given state and (d, e) in another: one entry of a product of
// two 0/1 matrices over the rows, features of pairs by features of low sets.  All tables of
// one size (4 or 5 nodes; low sets of 2 or 3) are blocks of that product: a 128 x 256 tile
// holds up to twelve ternary pairs against nine ternary triples.  The indicators are 8-bit floats
// of 2.0 (one logic op, one add, one logic op make four of them from a row of states), the
// products 4.0, and the FP32 sums 4 x count are exact up to 2^22 rows.
//
// A persistent CTA per SM walks (pair tile, low-set tile) items: twelve warps write the
// indicators of 128 rows at a time into shared memory (a thread per four tile rows and 32
// rows of the data, three stages), one thread issues tcgen05.mma kind::f8f6f4 into one of two 256-column TMEM
// accumulators, eight warps turn the other accumulator's counts into lgamma terms (96-bit
// fixed point, an eight-byte and a four-byte lookup whose small indices are free of bank
// conflicts), add them over each table and store G -- and, for sets that are parent sets
// too, the configuration sums H of every variant from the same counts.  Sets whose pair does not lie above
// the low set are computed and dropped; pairs come in order of falling d, so those are few.
//
// What bounds it is the shared-memory port: the indicators written (165 M wavefronts at
// n = 60) and read by the products (the tensor pipe is 27 % busy), three wavefronts of lookups
// a warp and cell (204 M); the LSU alone keeps it 64 % busy.  Against the histogram kernel
// (k_joint: 628 warp instructions a set, 4.1 ms for the 5.46 M 5-node sets of n = 60,
// m = 1000) it takes 2.69 ms, the build 6.1 ms instead of 7.08.  (With lookups behind a branch
// per cell, which serialises their latency, it took 5.5 ms; through generic addresses and
// with spills 3.9; with a thread per tile row, which loads the states of a set once for each
// of its cells, 2.81.)  The 487,635 sets of four nodes: 0.20 ms against 0.59, the build 4.87
// ms against 5.14 with the histograms for those.
#include <algorithm>
#include <vector>

#include "bn_joint_tc.cuh"
#include "bn_tc.cuh"

namespace bn {

static constexpr int TJ_M = 128, TJ_N = 256;
static constexpr int TJ_KC = 128;                       // rows of the data per stage
static constexpr int TJ_STAGES = 3;
static constexpr int TJ_GEN = TJ_M + TJ_N;              // generator threads
static constexpr int TJ_GEN_WARPS = TJ_GEN / 32;
static constexpr int TJ_EPI_WARPS = 8;                 // two for every quarter of the TMEM lanes
static constexpr int TJ_THREADS = TJ_GEN + 32 + 32 * TJ_EPI_WARPS;
static constexpr int TJ_A_BYTES = TJ_M * TJ_KC, TJ_B_BYTES = TJ_N * TJ_KC;
static constexpr int TJ_LUT_ROWS = 6300;                // entries of the lgamma tables in shared memory
static constexpr uint32_t TJ_NO_ROW = 0xffffffffu;
static constexpr int TJ_PAD_STATE = 0x3f;               // a state no feature has

struct TcJointArgs {
    const uint8_t* tlow;           // [NL][mp] states of the low sets' nodes as one number
    const uint8_t* thigh;          // [NH][mp] of the pairs; rows at or past m: TJ_PAD_STATE
    const uint32_t* low;           // [NL] states (cells) of each low set
    const uint32_t* nt_start;      // [NT + 1] first low set of every column tile
    const uint32_t* mt_first;      // [MT + 1] first item of every row tile
    const uint32_t* rowinfo;       // [MT][128] pair << 8 | state, or TJ_NO_ROW
    const uint32_t* pairs;         // [NH] d | e << 8 | r_d r_e << 16
    int mp;                        // rows padded to whole stages
    int m1;                        // m + 1
    uint32_t items, MT;
    int lowk;                      // nodes of a low set (2 or 3)
    int64_t base;                  // first rank of the sets' size
    const fx128* lut[4];           // lgamma terms of a cell count; configuration counts' variants
    fx128* G;
    fx128* H;                      // [variant][H_stride] by rank
    int64_t H_stride;
    uint32_t* status;
};

// cells of every low set; states of low sets (t < NL) and pairs, 16 rows a thread
__global__ void __launch_bounds__(128) k_tc_rows(const uint32_t* __restrict__ packed, int m, int mw, int mp,
                                                 const uint8_t* __restrict__ arity, int lowk, uint32_t NL,
                                                 const uint32_t* __restrict__ pairs, uint32_t* __restrict__ low,
                                                 uint8_t* __restrict__ tlow, uint8_t* __restrict__ thigh)
{
    __shared__ int s_v[3], s_st[3];
    const uint32_t t = blockIdx.x;
    const bool high = t >= NL;
    if (threadIdx.x == 0) {
        int v[3] = {0, 0, 0};
        const int cnt = high ? 2 : lowk;
        if (high) {
            v[0] = (int)(pairs[t - NL] & 0xffu);
            v[1] = (int)((pairs[t - NL] >> 8) & 0xffu);
        } else {
            uint64_t r = t;                              // colex: largest element first
            for (int q = lowk; q >= 1; --q) {
                int a = q - 1;
                while (a + 1 < 64 && g_binom.v[a + 1][q] <= r) ++a;
                v[q - 1] = a;
                r -= g_binom.v[a][q];
            }
        }
        int st = 1;
        for (int q = 0; q < 3; ++q) {
            s_v[q] = v[q];
            s_st[q] = q < cnt ? st : 0;
            if (q < cnt) st *= arity[v[q]];
        }
        if (!high) low[t] = (uint32_t)st;
    }
    __syncthreads();
    uint8_t* out = high ? thigh + (size_t)(t - NL) * mp : tlow + (size_t)t * mp;
    const uint32_t pad = high ? TJ_PAD_STATE * 0x01010101u : 0u;
    for (int w = threadIdx.x; w < mp / 16; w += 128) {
        uint32_t o[4] = {pad, pad, pad, pad};
        if (w < mw) {
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                uint32_t x = 0;
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    x += ((packed[(size_t)s_v[q] * mw + w] >> (2 * s)) & 0x03030303u) * (uint32_t)s_st[q];
                o[s] = x;
            }
            const int rows = m - 16 * w;                 // rows past m in the last word
            if (rows < 16)
                for (int b = max(rows, 0); b < 16; ++b)
                    o[b >> 2] = (o[b >> 2] & ~(0xffu << (8 * (b & 3)))) | (pad & (0xffu << (8 * (b & 3))));
        }
        *(uint4*)(out + 16 * w) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// 2.0 (0x40) where a byte of t equals the state s4 (repeated), else 0; bytes below 64;
// `on` is 0x40404040, or 0 for a row of zeros
__device__ __forceinline__ uint32_t indicator(uint32_t t, uint32_t s4, uint32_t on)
{
    return ~((t ^ s4) + 0x3f3f3f3fu) & on;
}
__device__ __forceinline__ void st_shared_v4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
// s += the 96-bit table entry at (lo, hi)
__device__ __forceinline__ void add_term(uint32_t (&s)[3], const uint32_t (&x)[3])
{
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(s[0]), "+r"(s[1]), "+r"(s[2])
        : "r"(x[0]), "r"(x[1]), "r"(x[2]));
}

// D[tmem] (+)= A[smem] B[smem]^T of 8-bit floats, issued by one thread
__device__ __forceinline__ void tc_mma_f8(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, bool accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate)
        : "memory");
}
// kind::f8f6f4: f32 accumulator, e4m3 operands (format code 0), both K-major
__host__ __device__ constexpr uint32_t tc_idesc_e4m3_f32(int M, int N)
{
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// core-matrix layout of a tile: row r, 16-byte chunk kc of its TJ_KC bytes
__device__ __forceinline__ uint32_t tj_off(int r, int kc) { return (uint32_t)((r >> 3) * (TJ_KC * 8) + kc * 128 + (r & 7) * 16); }

struct TjBars {
    uint64_t full[TJ_STAGES], empty[TJ_STAGES], acc_full[2], acc_empty[2], drain;
    uint32_t tmem;
    int abort;
};

// NH: variants of the configuration sums (sets that are parent sets too), or 0
template <int NH>
__global__ void __launch_bounds__(TJ_THREADS, 1) k_joint_tc(TcJointArgs A)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ TjBars S;
    uint8_t* sA = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sB = sA + TJ_STAGES * TJ_A_BYTES;
    uint64_t* lut_lo = (uint64_t*)(sB + TJ_STAGES * TJ_B_BYTES);       // [1 + NH][m1] low 64 bits
    uint32_t* lut_hi = (uint32_t*)(lut_lo + (1 + NH) * A.m1);          // [1 + NH][m1] next 32 bits
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nst = A.mp / TJ_KC;

#pragma unroll
    for (int l = 0; l <= NH; ++l)
        for (int i = tid; i < A.m1; i += TJ_THREADS) {
            lut_lo[l * A.m1 + i] = (uint64_t)A.lut[l][i];
            lut_hi[l * A.m1 + i] = (uint32_t)(A.lut[l][i] >> 64);
        }
    if (warp == TJ_GEN_WARPS) {
        tc_alloc(&S.tmem, 512);
        tc_relinquish();
    }
    if (tid == 0) {
        S.abort = 0;
        for (int s = 0; s < TJ_STAGES; ++s) {
            mbar_init(&S.full[s], TJ_GEN_WARPS);
            mbar_init(&S.empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&S.acc_full[s], 1);
            mbar_init(&S.acc_empty[s], TJ_EPI_WARPS);
        }
        mbar_init(&S.drain, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem;
    // a bounded wait, one decision a warp; a wait that runs out ends every role at its next
    auto wait = [&](uint64_t* bar, uint32_t parity) {
        if (__shfl_sync(0xffffffffu, *(volatile int*)&S.abort, 0)) return false;
        if (__all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, WAIT_TIMEOUT_NS))) return true;
        if (lane == 0) {
            *(volatile int*)&S.abort = 1;
            atomicOr(A.status, STATUS_TIMEOUT);
        }
        return false;
    };
    uint32_t mt = 0;                                    // row tile of the current item (items ascend)
    auto locate = [&](uint32_t item, uint32_t& t0, uint32_t& t1) {
        while (mt + 1 < A.MT && item >= __ldg(A.mt_first + mt + 1)) ++mt;
        const uint32_t nt = item - __ldg(A.mt_first + mt);
        t0 = __ldg(A.nt_start + nt);
        t1 = __ldg(A.nt_start + nt + 1);
    };

    if (warp < TJ_GEN_WARPS) {
        // ---- indicators: a thread writes four consecutive rows of 32 (two pieces of 16) rows of
        // the data; they belong to two sets at most (a set has four states or more), so it
        // loads two pieces a stage, seldom four, for the eight it stores.  Its rows come in an
        // order turned by its piece: eight lanes of a store phase then meet eight banks.
        const int quad = (warp >> 1) * 16 + (warp & 1) * 8 + (lane >> 2);   // (96 quads, A's first)
        const int piece = lane & 3;                     // and piece + 4
        const bool isA = quad < TJ_M / 4;
        const int row = 4 * (isA ? quad : quad - TJ_M / 4);
        const uint32_t dst0 = smem_u32(isA ? sA : sB) + tj_off(row, piece);
        const uint32_t stage_bytes = isA ? TJ_A_BYTES : TJ_B_BYTES;
        uint32_t st = 0, ph = 0;                        // stage and its phase
        bool go = true;
        for (uint32_t item = blockIdx.x; go && item < A.items; item += gridDim.x) {
            uint32_t t0, t1;
            locate(item, t0, t1);
            const uint8_t* src[2] = {isA ? A.thigh : A.tlow, nullptr};      // first and last row's set
            int split = 4;                              // rows of the first
            uint32_t s4[4], on = 0;                     // state of row (i + piece) % 4; bit i: it has one
            if (isA) {
                const uint4 x = __ldg((const uint4*)(A.rowinfo + (size_t)mt * TJ_M + row));
                const uint32_t info[4] = {x.x, x.y, x.z, x.w};
                if (info[0] != TJ_NO_ROW) src[0] += (size_t)(info[0] >> 8) * A.mp;
#pragma unroll
                for (int i = 3; i >= 1; --i)
                    if (info[i] != TJ_NO_ROW && info[i] >> 8 != info[0] >> 8) {
                        split = i;
                        src[1] = A.thigh + (size_t)(info[i] >> 8) * A.mp;
                    }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int q = (i + piece) & 3;
                    const uint32_t f = q == 0 ? info[0] : q == 1 ? info[1] : q == 2 ? info[2] : info[3];
                    s4[i] = (f & 0xffu) * 0x01010101u;
                    if (f != TJ_NO_ROW) on |= 1u << i;
                }
            } else {
                int o = 0, first = 0;                   // columns before the set; states of row 0
                uint32_t t = t0;
                int w = (int)__ldg(A.low + t);
                while (t < t1 && row >= o + w) {
                    o += w;
                    w = ++t < t1 ? (int)__ldg(A.low + t) : 0;
                }
                int n1 = 0;                             // rows with a set
                if (t < t1) {
                    src[0] += (size_t)t * A.mp;
                    first = row - o;
                    n1 = 4;
                    if (first + 4 > w) {
                        split = w - first;
                        if (t + 1 < t1) src[1] = A.tlow + (size_t)(t + 1) * A.mp;
                        else n1 = split;
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int q = (i + piece) & 3;
                    s4[i] = (uint32_t)(q < split ? first + q : q - split) * 0x01010101u;
                    if (q < n1) on |= 1u << i;
                }
            }
            const bool two = src[1] != nullptr;
            const uint4* p0 = (const uint4*)src[0] + piece;
            const uint4* p1 = (const uint4*)src[1] + piece;
            // the states of a stage are loaded while the one before is multiplied
            uint4 v[2], u[2];
            auto fetch = [&](int k) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    v[h] = __ldg(p0 + k * (TJ_KC / 16) + 4 * h);
                    u[h] = two ? __ldg(p1 + k * (TJ_KC / 16) + 4 * h) : v[h];
                }
            };
            fetch(0);
            for (int k = 0; k < nst; ++k) {
                if (!wait(&S.empty[st], ph ^ 1u)) {     // (the first pass over the stages is free)
                    go = false;
                    break;
                }
                const uint32_t dst = dst0 + st * stage_bytes;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int q = (i + piece) & 3;
                    const uint32_t bits = on >> i & 1u ? 0x40404040u : 0u;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint4 x = q < split ? v[h] : u[h];
                        st_shared_v4(dst + q * 16 + h * 512, indicator(x.x, s4[i], bits), indicator(x.y, s4[i], bits),
                                     indicator(x.z, s4[i], bits), indicator(x.w, s4[i], bits));
                    }
                }
                if (k + 1 < nst) fetch(k + 1);
                fence_proxy_async_smem();               // visible to the tensor core's async proxy
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.full[st]);
                if (++st == TJ_STAGES) {
                    st = 0;
                    ph ^= 1u;
                }
            }
        }
    } else if (warp == TJ_GEN_WARPS) {
        // ---- products
        constexpr uint32_t idesc = tc_idesc_e4m3_f32(TJ_M, TJ_N);
        uint32_t st = 0, ph = 0, done = 0;
        bool go = true;
        for (uint32_t item = blockIdx.x; go && item < A.items; item += gridDim.x, ++done) {
            const uint32_t buf = done & 1u;
            // this accumulator was read by the item before last
            if (!wait(&S.acc_empty[buf], ((done >> 1) & 1u) ^ 1u)) break;
            tc_fence_after();
            for (int k = 0; k < nst; ++k) {
                if (!wait(&S.full[st], ph)) {
                    go = false;
                    break;
                }
                if (lane == 0) {
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < TJ_KC / 32; ++kk) {
                        const uint64_t ad = tc_smem_desc(sA + st * TJ_A_BYTES + kk * 256, 128, TJ_KC * 8);
                        const uint64_t bd = tc_smem_desc(sB + st * TJ_B_BYTES + kk * 256, 128, TJ_KC * 8);
                        tc_mma_f8(tmem + buf * TJ_N, ad, bd, idesc, (k > 0) || (kk > 0));
                    }
                    tc_commit(&S.empty[st]);
                    if (k + 1 == nst) tc_commit(&S.acc_full[buf]);
                }
                __syncwarp();
                if (++st == TJ_STAGES) {
                    st = 0;
                    ph ^= 1u;
                }
            }
        }
        // every product issued must have completed before its memory goes away
        if (lane == 0) {
            tc_commit(&S.drain);
            mbar_wait_bounded(&S.drain, 0, WAIT_TIMEOUT_NS);
        }
        __syncwarp();
    } else {
        // ---- lgamma terms: warp w of the CTA reads TMEM lanes 32 (w % 4) .. + 31; two warps
        // share a quarter, one the even, one the odd sets
        const int quarter = warp & 3, row = quarter * 32 + lane;
        const uint32_t half = (uint32_t)(warp - TJ_GEN_WARPS - 1) >> 2;
        // where the entry of count 0 lies, less the bits of the float 2^23
        const uint32_t at_lo = smem_u32(lut_lo) - 2u * 0x4b000000u, at_hi = smem_u32(lut_hi) - 0x4b000000u;
        const uint32_t step = 4u * (uint32_t)A.m1;      // bytes of one table's high words
        uint32_t done = 0;
        for (uint32_t item = blockIdx.x; item < A.items; item += gridDim.x, ++done) {
            uint32_t t0, t1;
            locate(item, t0, t1);
            const uint32_t info = __ldg(A.rowinfo + (size_t)mt * TJ_M + row);
            int pos = 0, g = 1;
            uint32_t limit = 0;                         // low sets below it lie below the pair
            int64_t at = 0;
            if (info != TJ_NO_ROW) {
                const uint32_t pr = __ldg(A.pairs + (info >> 8));
                const int d = (int)(pr & 0xffu), e = (int)((pr >> 8) & 0xffu);
                pos = (int)(info & 0xffu);
                g = (int)(pr >> 16);
                limit = (uint32_t)g_binom.v[d][A.lowk];
                at = A.base + (int64_t)g_binom.v[d][A.lowk + 1] + (int64_t)g_binom.v[e][A.lowk + 2];
            }
            const uint32_t buf = done & 1u;
            if (!wait(&S.acc_full[buf], (done >> 1) & 1u)) break;
            tc_fence_after();
            const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + buf * TJ_N;
            int o = 0;                                  // the set's first column
            for (uint32_t t = t0; t < t1; ++t) {
                const int w = (int)__ldg(A.low + t);
                const int o0 = o;
                o += w;
                if (((t - t0) & 1u) != half) continue;  // the quarter's other warp takes it
                uint32_t sum[1 + NH][3] = {};
                for (int c0 = 0; c0 < w; c0 += 32) {
                    // 32 columns, moved back where they would leave this accumulator; those
                    // of other sets count as 0, whose term is 0
                    uint32_t r[32];
                    const int back = max(0, o0 + c0 + 32 - TJ_N);
                    tc_ld_32x32b_x32(acc + (uint32_t)(o0 + c0 - back), r);
                    tc_wait_ld();
                    const int j1 = min(32, w - c0 + back);
#pragma unroll
                    for (int j4 = 0; j4 < 32; j4 += 4) {
                        if (j4 + 4 <= back || j4 >= j1) continue;           // warp-uniform
                        if (j4 < back || j4 + 4 > j1) {
#pragma unroll
                            for (int j = j4; j < j4 + 4; ++j)
                                if (j < back || j >= j1) r[j] = 0u;
                        }
                        uint32_t x[1 + NH][4][3];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            // 4 x count as the low bits of the float 2^23 + 4 x count
                            const uint32_t i4 = __float_as_uint(__uint_as_float(r[j4 + q]) + 8388608.0f);
#pragma unroll
                            for (int l = 0; l <= NH; ++l) {
                                asm("ld.shared.v2.u32 {%0, %1}, [%2];"
                                    : "=r"(x[l][q][0]), "=r"(x[l][q][1]) : "r"(2 * i4 + at_lo + 2 * l * step));
                                asm("ld.shared.u32 %0, [%1];" : "=r"(x[l][q][2]) : "r"(i4 + at_hi + l * step));
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q)
#pragma unroll
                            for (int l = 0; l <= NH; ++l) add_term(sum[l], x[l][q]);
                    }
                }
                // the pair's rows (lanes pos = 0 .. g - 1 of one group), to the first
#pragma unroll
                for (int l = 0; l <= NH; ++l) {
#pragma unroll
                    for (int off = 8; off; off >>= 1) {
                        const uint32_t x[3] = {__shfl_down_sync(0xffffffffu, sum[l][0], off),
                                               __shfl_down_sync(0xffffffffu, sum[l][1], off),
                                               __shfl_down_sync(0xffffffffu, sum[l][2], off)};
                        if (pos < off && pos + off < g) add_term(sum[l], x);
                    }
                    fx128* out = l ? A.H + (size_t)(l - 1) * A.H_stride : A.G;
                    if (pos == 0 && t < limit)
                        out[at + t] = ((fx128)(uint64_t)(int64_t)(int32_t)sum[l][2] << 64) |
                                      (fx128)((uint64_t)sum[l][1] << 32 | sum[l][0]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.acc_empty[buf]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == TJ_GEN_WARPS) tc_dealloc(tmem, 512);
}

bool joint_tc_plan(int n, int m, int size, int luts, const uint8_t* ar, TcPlan* P)
{
    // Few sets: the set-up costs what the products save (k = 4, m = 1000: 26 nodes, 65,780 sets,
    // build 347 us against 365; 28 nodes with nearly constant columns 423 against 397; k = 3:
    // 30 nodes, 27,405 sets, m = 64, 240 against 211; 40 nodes, 91,390 sets, m = 1000, 336
    // against 400).  The lgamma tables have to fit beside the stages.
    const int lowk = size - 2;
    if ((size != 4 && size != 5) || n <= size || n > MAXN || m < 64 || luts * (m + 1) > TJ_LUT_ROWS) return false;
    const int64_t sets = (int64_t)h_binom.v[n][size];
    if (sets < 60000) return false;
    std::vector<uint32_t>&pairs = P->pairs, &rowinfo = P->rowinfo, &mt_first = P->mt_first, &nt_start = P->nt_start;
    // pairs d < e with room for a low set below d, d falling; 32-row blocks, no pair astride
    std::vector<int> tile_d;
    int used = 0;
    for (int d = n - 2; d >= lowk; --d)
        for (int e = d + 1; e < n; ++e) {
            const int g = ar[d] * ar[e];
            if (used + g > 32 || rowinfo.empty()) {
                rowinfo.resize((rowinfo.size() + 31) / 32 * 32, TJ_NO_ROW);
                if (rowinfo.size() % TJ_M == 0) tile_d.push_back(d);
                used = 0;
            }
            for (int q = 0; q < g; ++q) rowinfo.push_back((uint32_t)(pairs.size() << 8) | (uint32_t)q);
            used += g;
            pairs.push_back((uint32_t)d | (uint32_t)e << 8 | (uint32_t)g << 16);
        }
    rowinfo.resize((rowinfo.size() + TJ_M - 1) / TJ_M * TJ_M, TJ_NO_ROW);
    const uint32_t MT = (uint32_t)(rowinfo.size() / TJ_M);
    // low sets in colex order, packed into column tiles
    const uint32_t NL = (uint32_t)h_binom.v[n - 2][lowk];
    {
        int cols = 0;
        uint32_t t = 0;
        nt_start.push_back(0);
        auto add = [&](int w) {
            if (cols + w > TJ_N) {
                nt_start.push_back(t);
                cols = 0;
            }
            cols += w;
            ++t;
        };
        if (lowk == 2) {
            for (int b = 1; b < n - 2; ++b)
                for (int a = 0; a < b; ++a) add(ar[a] * ar[b]);
        } else {
            for (int c = 2; c < n - 2; ++c)
                for (int b = 1; b < c; ++b)
                    for (int a = 0; a < b; ++a) add(ar[a] * ar[b] * ar[c]);
        }
        nt_start.push_back(NL);
    }
    // items: a row tile with every column tile that starts below its largest d
    uint32_t items = 0;
    for (uint32_t i = 0; i < MT; ++i) {
        mt_first.push_back(items);
        const uint32_t limit = (uint32_t)h_binom.v[tile_d[i]][lowk];
        items += (uint32_t)(std::lower_bound(nt_start.begin(), nt_start.end() - 1, limit) - nt_start.begin());
    }
    mt_first.push_back(items);
    P->items = items;
    // An item costs the same however many sets it holds, a set of the histogram kernel the
    // same however few cells it has: at 99 sets an item (37 ternary nodes) the build takes
    // 773 us against 934, at 783 (binary) 591 against 966, at 30 (four states) 1,176 against
    // 1,031.  (Rows in which every node is nearly always in one state make the histograms
    // cheaper still: equal at 85 % of the rows.)
    return sets >= 48 * (int64_t)items;
}

template <int NH>
static int launch(const TcJointArgs& A, cudaStream_t s)
{
    static ContextOnce once;
    constexpr size_t fixed = (size_t)TJ_STAGES * (TJ_A_BYTES + TJ_B_BYTES) + 1024 + 16;
    const int rc = once_in_context(once, [&]() -> int {
        BN_CUDA(cudaFuncSetAttribute(k_joint_tc<NH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(fixed + 12 * (size_t)TJ_LUT_ROWS)));
        return BN_OK;
    });
    if (rc) return rc;
    const size_t smem = fixed + 12 * (size_t)(1 + NH) * A.m1;
    k_joint_tc<NH><<<std::min<uint32_t>((uint32_t)sm_count(), A.items), TJ_THREADS, smem, s>>>(A);
    BN_LAUNCH_CHECK("k_joint_tc");
    return BN_OK;
}

// the scratch block: lists | cells | states
struct TcScratch {
    size_t lists = 0, low, tlow, thigh, bytes;
    TcScratch(const TcPlan& P, int mp)
    {
        const size_t NL = P.nt_start.back(), NH = P.pairs.size();
        auto after = [](size_t at, size_t b) { return (size_t)round_up((int64_t)(at + b), 256); };
        low = after(0, 4 * (P.rowinfo.size() + P.nt_start.size() + P.mt_first.size() + NH));
        tlow = after(low, 4 * NL);
        thigh = after(tlow, NL * mp);
        bytes = after(thigh, NH * mp);
    }
};

size_t joint_tc_scratch(const TcPlan& P, int m) { return TcScratch(P, (int)round_up(m, TJ_KC)).bytes; }

int joint_tc_upload(const TcPlan& P, uint8_t* scratch, cudaStream_t s)
{
    std::vector<uint32_t> lists;
    lists.reserve(P.rowinfo.size() + P.nt_start.size() + P.mt_first.size() + P.pairs.size());
    for (const auto* v : {&P.rowinfo, &P.nt_start, &P.mt_first, &P.pairs}) lists.insert(lists.end(), v->begin(), v->end());
    BN_CUDA(cudaMemcpyAsync(scratch, lists.data(), 4 * lists.size(), cudaMemcpyHostToDevice, s));
    return BN_OK;
}

int launch_joint_tc(const TcJoint& J, const TcPlan& P, cudaStream_t s)
{
    const int n = J.n, lowk = J.size - 2, mp = (int)round_up(J.m, TJ_KC);
    const uint32_t NL = P.nt_start.back(), NH = (uint32_t)P.pairs.size();
    const TcScratch at(P, mp);
    uint8_t* base = J.scratch;
    TcJointArgs A;
    A.rowinfo = (const uint32_t*)base;                  // (first: read in pieces of 16 bytes)
    A.nt_start = A.rowinfo + P.rowinfo.size();
    A.mt_first = A.nt_start + P.nt_start.size();
    A.pairs = A.mt_first + P.mt_first.size();
    A.low = (const uint32_t*)(base + at.low);
    A.tlow = base + at.tlow;
    A.thigh = base + at.thigh;
    A.mp = mp;
    A.m1 = J.m + 1;
    A.items = P.items;
    A.MT = (uint32_t)P.mt_first.size() - 1;
    A.lowk = lowk;
    A.base = num_sets_host(n, J.size - 1);
    for (int l = 0; l < 4; ++l) A.lut[l] = J.lut[l];
    A.G = J.G;
    A.H = J.H;
    A.H_stride = J.H_stride;
    A.status = J.status;
    k_tc_rows<<<NL + NH, 128, 0, s>>>(J.packed, J.m, J.mw, mp, J.arity, lowk, NL, A.pairs, (uint32_t*)(base + at.low),
                                     base + at.tlow, base + at.thigh);
    BN_LAUNCH_CHECK("k_tc_rows");
    switch (J.nh) {
    case 0: return launch<0>(A, s);
    case 1: return launch<1>(A, s);
    case 2: return launch<2>(A, s);
    default: return launch<3>(A, s);
    }
}

}  // namespace bn
