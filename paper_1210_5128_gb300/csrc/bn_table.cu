// bn_table.cu -- the preprocessing step of Sec. III.A on the GPU: data staging, joint
// counting (N_ijk of Eq. (3)), the FP64 local score of Eq. (4) with the structure
// penalty, and the pairwise prior of Eq. (9)-(10), for every (node, parent set of size
// <= k).  The paper keeps these in a host hash table keyed by (node, parent set); here
// they are a dense device array indexed by (node, rank), plus the parent-set table
// (Sec. V.B) of candidate-space masks shared by all nodes.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <set>
#include <string>
#include <vector>

#include "bn_fx.cuh"
#include "bn_joint_tc.cuh"
#include "bn_table.cuh"

namespace bn {

static constexpr int BUILD_THREADS = 256;

// ---------------------------------------------------------------------------------
// rank <-> set on the device (sizes ascending, combinatorial number system)
// ---------------------------------------------------------------------------------
__device__ __forceinline__ void unrank_dev(int N, int64_t rank, int& j, uint64_t& mask)
{
    j = 0;
    while (rank >= (int64_t)c_binom.v[N][j]) { rank -= (int64_t)c_binom.v[N][j]; ++j; }
    mask = 0;
    for (int t = j; t >= 1; --t) {
        int a = N - 1;
        while ((int64_t)c_binom.v[a][t] > rank) --a;
        mask |= 1ull << a;
        rank -= (int64_t)c_binom.v[a][t];
    }
}

// next set in rank order: colex successor within a size (Gosper's hack), then the
// first set {0..j} of the next size
__device__ __forceinline__ void next_set(int N, int& j, uint64_t& mask)
{
    if (j == 0) { j = 1; mask = 1; return; }
    if (mask == (~0ull >> (64 - j)) << (N - j)) {       // {N - j .. N - 1}, the last of its size
        ++j;
        mask = (j >= 64) ? ~0ull : ((1ull << j) - 1);
        return;
    }
    uint64_t c = mask & (~mask + 1);
    uint64_t r = mask + c;
    mask = (((r ^ mask) >> 2) >> (__ffsll((long long)mask) - 1)) | r;
}

// ---------------------------------------------------------------------------------
// a1: data staging.  m x n row-major uint8 -> [n][mw] words of 16 two-bit values.  Row
// 16w + b sits at bits 8(b & 3) + 2(b >> 2), so one shift by 2s and a mask 0x03030303
// yields rows 16w + 4s .. 16w + 4s + 3 as four bytes.  Rows past m are 0 (every variable
// in state 0); the counting kernel takes their number back out of cell 0.
// ---------------------------------------------------------------------------------
__global__ void k_pack(const uint8_t* __restrict__ data, int m, int n, int mw,
                       const uint8_t* __restrict__ arity, uint32_t* __restrict__ packed,
                       uint32_t* status)
{
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * mw) return;
    int v = idx / mw, w = idx - v * mw;
    int av = arity[v];
    uint32_t word = 0;
    bool bad = false;
    for (int b = 0; b < 16; ++b) {
        int row = 16 * w + b;
        if (row < m) {
            uint32_t x = data[(size_t)row * n + v];
            if (x >= (uint32_t)av) { bad = true; x = 0; }   // never let a bad value index a count table
            word |= x << (8 * (b & 3) + 2 * (b >> 2));
        }
    }
    if (bad) atomicOr(status, STATUS_BADINPUT);
    packed[idx] = word;
}

// Per variable the rows that are not in its most frequent state, ascending, as row * 4 +
// (the state's index among the others): one block a variable, states from the packed words.
static constexpr int LIST_ROWS = 1 << 14;          // rows a 16-bit list entry can name
__global__ void __launch_bounds__(256) k_minor_rows(const uint32_t* __restrict__ packed, int m, int mw,
                                                    uint16_t* __restrict__ rows, uint32_t* __restrict__ len)
{
    __shared__ uint32_t s_cnt[4], s_w[8];
    const int v = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t* D = packed + (size_t)v * mw;
    auto state = [&](int r) { return (D[r >> 4] >> (8 * (r & 3) + 2 * ((r & 15) >> 2))) & 3u; };
    if (tid < 4) s_cnt[tid] = 0;
    __syncthreads();
    uint32_t c[4] = {0, 0, 0, 0};
    for (int r = tid; r < m; r += 256) {
        const uint32_t x = state(r);
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) c[q] += x == q;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t t = __reduce_add_sync(0xffffffffu, c[q]);
        if (lane == 0 && t) atomicAdd(&s_cnt[q], t);
    }
    __syncthreads();
    uint32_t mode = 0;
    for (uint32_t q = 1; q < 4; ++q)
        if (s_cnt[q] > s_cnt[mode]) mode = q;
    uint32_t at = 0;
    for (int r0 = 0; r0 < m; r0 += 256) {
        const int r = r0 + tid;
        const uint32_t x = r < m ? state(r) : mode;
        const unsigned bal = __ballot_sync(0xffffffffu, x != mode);
        if (lane == 0) s_w[warp] = __popc(bal);
        __syncthreads();
        uint32_t before = 0, all = 0;
        for (int w = 0; w < 8; ++w) {
            before += w < warp ? s_w[w] : 0u;
            all += s_w[w];
        }
        if (x != mode)
            rows[(size_t)v * m + at + before + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(r * 4 + x - (x > mode));
        at += all;
        __syncthreads();
    }
    if (tid == 0) len[v] = at;
}

// PPF of Eq. (10): ppf[i][m] = 100 (R[i][m] - 0.5)^3, evaluated left to right.
__global__ void k_ppf(const double* __restrict__ R, int n, double* __restrict__ ppf)
{
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * n) return;
    double d = __dsub_rn(R[idx], 0.5);
    ppf[idx] = __dmul_rn(__dmul_rn(__dmul_rn(100.0, d), d), d);
}

// lgamma lookup: lut[l][N] = lgamma(N + alpha_l) - lgamma(alpha_l) in 64.64 fixed point
__global__ void k_lut(const double* __restrict__ alpha, int nlut, int m1, fx128* __restrict__ lut)
{
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)nlut * m1) return;
    int l = (int)(idx / m1), N = (int)(idx - (int64_t)l * m1);
    double a = alpha[l];
    double g = (N == 0) ? 0.0 : __dsub_rn(lgamma((double)N + a), lgamma(a));
    lut[idx] = fx_from_double(g);
}

// a4: parent-set table, candidate-space mask of every rank; padding ranks get ~0 (they
// can never be consistent with an order).  A thread unranks the first of PST_RUN
// consecutive ranks (binomials in shared memory, binary searches) and steps to the others:
// 55 -> 8 us at n = 60, k = 4 against one unranking from the constant bank per rank.
static constexpr int PST_RUN = 4;
__global__ void __launch_bounds__(256) k_pst(int N, int k, int64_t S, int64_t Sp, uint64_t* __restrict__ pst)
{
    extern __shared__ uint64_t s_bin[];                 // C(a, t), a <= 63, t <= k
    const int T = k + 1;
    for (int q = threadIdx.x; q < 64 * T; q += blockDim.x) s_bin[q] = g_binom.v[q / T][q % T];
    __syncthreads();
    const int64_t r0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * PST_RUN;
    if (r0 >= Sp) return;                               // Sp is a multiple of PST_RUN
    int j = 0;
    uint64_t mask = 0;
    if (r0 < S) {
        uint64_t r = (uint64_t)r0;
        while (r >= s_bin[N * T + j]) r -= s_bin[N * T + j++];
        int hi = N - 1;
        for (int t = j; t >= 1; --t) {                  // largest a with C(a, t) <= r
            int lo = t - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_bin[mid * T + t] <= r) lo = mid;
                else hi = mid - 1;
            }
            mask |= 1ull << lo;
            r -= s_bin[lo * T + t];
            hi = lo - 1;
        }
    }
#pragma unroll
    for (int u = 0; u < PST_RUN; ++u) {
        pst[r0 + u] = r0 + u < S ? mask : ~0ull;
        next_set(N, j, mask);
    }
}

__global__ void k_pad_keys(int64_t* __restrict__ keys, int n, int64_t S, int64_t Sp)
{
    int64_t pad = Sp - S;
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)n * pad) return;
    int64_t i = idx / pad, e = idx - i * pad;
    keys[i * Sp + S + e] = KEY_NONE;
}

// ---------------------------------------------------------------------------------
// a2 + a3 by joint tables.  An entry's lgamma terms split into a sum over the cells of the
// joint count table of U = pi + {i} and a sum over the configurations of pi:
//     sum_c sum_x L_cell[N_cx] - sum_c L_cfg[N_c] = G(U) - H(pi).
// G depends on U alone (its lgamma table is the one of alpha = 1 for K2 and of ess over
// the number of cells for BDeu, whichever member of U is the child) and H on pi and, for
// K2, the child's arity.  Both are exact 128-bit fixed-point integers, so their difference
// is the exact sum and the entry's one rounding is unchanged.  So the rows are counted
// once per set U of at most k + 1 nodes (k_joint) instead of once per (node, parent set):
// C(60, 5) = 5.5 M tables instead of 29.4 M at n = 60, k = 4; k_assemble forms the entries.
// Measured at n = 60, k = 4, m = 1000, ternary: 20.0 ms with one count table per entry,
// 4.51 ms for k_joint over all of them; with the sets of four and five nodes on the tensor
// cores (bn_joint_tc.cu) 2.90 ms for those, 0.08 for k_joint and 0.34 for k_assemble.
// ---------------------------------------------------------------------------------
struct JointArgs {
    const uint32_t* packed;
    const uint16_t* minor;    // [n][m] rows not in the variable's most frequent state
    const uint32_t* minor_len;
    int n, m, mw;
    uint32_t pad;             // zero rows of the last word, all in cell 0
    int k;                    // largest parent set
    int64_t S0, S1;           // sets of at most k and of at most k + 1 of the n nodes
    int range;                // consecutive sets per warp work unit
    int cells_cap;
    const uint8_t* arity;
    const fx128* lut;
    int lut_stride;           // m + 1
    const int16_t* cell_lut;  // [cells] lgamma table of a joint table of that many cells
    const int16_t* cfg_lut;   // [q * nv + v] of variant v's configuration counts
    int nv;                   // variants of H: the distinct child arities (K2), 1 (BDeu)
    fx128* G;                 // [S1]
    fx128* H;                 // [nv][S0]
};

// warp sum, exact mod 2^128: five limbs (26, 26, 26, 26, 24 bits) of every lane's value
// summed by one 32-bit reduction instruction each (32 lanes x 2^26 < 2^32)
__device__ __forceinline__ fx128 warp_sum_fx(fx128 acc)
{
    const uint64_t lo = (uint64_t)acc, hi = (uint64_t)(acc >> 64);
    constexpr uint64_t M26 = (1ull << 26) - 1;
    const uint32_t s0 = __reduce_add_sync(0xffffffffu, (uint32_t)(lo & M26));
    const uint32_t s1 = __reduce_add_sync(0xffffffffu, (uint32_t)((lo >> 26) & M26));
    const uint32_t s2 = __reduce_add_sync(0xffffffffu, (uint32_t)(((lo >> 52) | (hi << 12)) & M26));
    const uint32_t s3 = __reduce_add_sync(0xffffffffu, (uint32_t)((hi >> 14) & M26));
    const uint32_t s4 = __reduce_add_sync(0xffffffffu, (uint32_t)(hi >> 40));
    return (fx128)s0 + ((fx128)s1 << 26) + ((fx128)s2 << 52) + ((fx128)s3 << 78) + ((fx128)s4 << 104);
}

// the lgamma terms of one cell count for the joint sum and, if the set is a parent set too,
// for every variant of its configuration sum
struct JointLuts {
    const fx128* x;
    const fx128* c[3];
};
template <bool PARENT>
__device__ __forceinline__ void add_cell(uint32_t v, const JointLuts& L, int nv, fx128& g, fx128 (&h)[3])
{
    g += L.x[v];
    if (PARENT) {
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (q < nv) h[q] += L.c[q][v];
    }
}

// The counts of the cells hist[q * Qp + c] (q-th of the lowest node's RI - 1 minor states,
// configuration c of the nodes above) and, as what is left of pre[c], of its most frequent
// state.  Every cell read is set back to 0 for the next set.
template <int RI, bool PARENT>
__device__ __forceinline__ void minor_cells(uint32_t* hist, const uint32_t* pre, int Qp, const JointLuts& L, int nv,
                                            int lane, fx128& g, fx128 (&h)[3])
{
    for (int c = lane; c < Qp; c += 32) {
        uint32_t v[RI > 1 ? RI - 1 : 1], rest = pre[c];
#pragma unroll
        for (int q = 0; q < RI - 1; ++q) {
            v[q] = hist[q * Qp + c];
            rest -= v[q];
        }
#pragma unroll
        for (int q = 0; q < RI - 1; ++q) {
            hist[q * Qp + c] = 0u;
            add_cell<PARENT>(v[q], L, nv, g, h);
        }
        add_cell<PARENT>(rest, L, nv, g, h);
    }
}

// One warp per unit of `range` consecutive sets U (colex order: the lowest node varies
// fastest).  MINOR keeps, while the nodes above the lowest stay the same (about 12 sets on
// average at n = 60, k = 4), every row's configuration of them (16 bits a row, as a byte
// offset) and the configurations' counts; a set then visits only the rows in which its
// lowest node is not in its most frequent state -- about half -- and the frequent state's
// cells are what is left of the configurations' counts.  A visit is two 16-bit loads (the
// list ascends, so the second is nearly consecutive over the lanes), a multiply-add and a
// shared atomic; the hottest cells take no atomics at all.  Without MINOR (few sets, or many
// rows: the rule is in build_enqueue) every row's cell is formed from all nodes.  Shared memory
// holds the warps' histograms, the rows' offsets (MINOR), then (SMEM_DATA) the packed data.
// n = 60, k = 4, m = 1000: 4.51 ms against 5.05 with every row visited; 628 warp
// instructions a set at two thirds of the issue slots, and the shared-memory pipe 72 % busy
// with atomics (a third of it) and the lgamma lookups.
template <int KT, bool SMEM_DATA, bool MINOR>
__global__ void __launch_bounds__(BUILD_THREADS) k_joint(JointArgs A)
{
    extern __shared__ __align__(16) uint32_t sm[];
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int items = A.mw * 4;                 // of four rows
    uint32_t* hist = sm + warp * A.cells_cap;
    uint2* base = (uint2*)(sm + nw * A.cells_cap) + (MINOR ? warp * items : 0);
    const uint32_t* D = A.packed;
    for (int c = lane; c < A.cells_cap; c += 32) hist[c] = 0u;
    if (SMEM_DATA) {
        uint32_t* sd = sm + nw * A.cells_cap + (MINOR ? nw * items * 2 : 0);
        for (int t = threadIdx.x; t < A.n * A.mw; t += blockDim.x) sd[t] = A.packed[t];
        D = sd;
    }
    __syncthreads();
    uint8_t* hb = (uint8_t*)hist;
    const int64_t units = (A.S1 + A.range - 1) / A.range;
    for (int64_t u = (int64_t)blockIdx.x * nw + warp; u < units; u += (int64_t)gridDim.x * nw) {
        const int64_t r0 = u * A.range;
        const int64_t r1 = min(r0 + (int64_t)A.range, A.S1);
        int j;
        uint64_t mask;
        unrank_dev(A.n, r0, j, mask);
        uint64_t above = ~0ull;                 // the nodes above the lowest that `base` is for
        int poff[KT];
        uint32_t cs[KT];
        int Qp = 1;
        uint32_t* pre = hist;                   // (MINOR) configuration counts, the histogram's last Qp words
        fx128 my_acc = 0;
        for (int64_t rho = r0; rho < r1; ++rho) {
            const uint64_t up = mask & (mask - 1);
            if (up != above) {                  // (warp-uniform)
                above = up;
                if (MINOR) {
                    for (int c = lane; c < Qp; c += 32) pre[c] = 0u;
                }
                Qp = 1;
                uint64_t mm = up;
#pragma unroll
                for (int t = 0; t < KT; ++t) {
                    poff[t] = 0;
                    cs[t] = 0u;
                    if (mm) {
                        const int p = __ffsll((long long)mm) - 1;
                        mm &= mm - 1;
                        poff[t] = p * A.mw;
                        cs[t] = (uint32_t)(4 * Qp);
                        Qp *= __ldg(&A.arity[p]);
                    }
                }
                if (MINOR) {
                    pre = hist + A.cells_cap - Qp;
                    uint8_t* pb = (uint8_t*)pre;
                    __syncwarp();
                    for (int c = lane; c < items; c += 32) {
                        const int w = c >> 2, sft = 2 * (c & 3);
                        uint32_t e = 0u, o = 0u;             // rows 4 c, 4 c + 2 and 4 c + 1, 4 c + 3
#pragma unroll
                        for (int t = 0; t < KT; ++t) {
                            const uint32_t x = D[poff[t] + w] >> sft;
                            e += (x & 0x00030003u) * cs[t];
                            o += ((x >> 8) & 0x00030003u) * cs[t];
                        }
                        base[c] = make_uint2(__byte_perm(e, o, 0x5410), __byte_perm(e, o, 0x7632));
                        atomicAdd((uint32_t*)(pb + (e & 0xffffu)), 1u);
                        atomicAdd((uint32_t*)(pb + (e >> 16)), 1u);
                        atomicAdd((uint32_t*)(pb + (o & 0xffffu)), 1u);
                        atomicAdd((uint32_t*)(pb + (o >> 16)), 1u);
                    }
                    __syncwarp();
                    if (lane == 0) pre[0] -= A.pad;
                    __syncwarp();
                }
            }
            const int low = mask ? __ffsll((long long)mask) - 1 : 0;
            const int ri = mask ? (int)__ldg(&A.arity[low]) : 1;
            const int Q = Qp * ri;
            const uint32_t scale = mask ? (uint32_t)(4 * Qp) : 0u;
            if (MINOR) {
                const uint16_t* L = A.minor + (size_t)low * A.m;
                const int len = mask ? (int)__ldg(&A.minor_len[low]) : 0;
                const uint16_t* rowoff = (const uint16_t*)base;
#pragma unroll 4
                for (int i = lane; i < len; i += 32) {
                    const uint32_t e = __ldg(L + i);
                    const uint32_t off = rowoff[e >> 2] + (e & 3u) * scale;
                    atomicAdd((uint32_t*)(hb + off), 1u);
                }
            } else {
                const uint32_t* Dl = D + (size_t)low * A.mw;
                for (int c = lane; c < items; c += 32) {
                    const int w = c >> 2, sft = 2 * (c & 3);
                    const uint32_t x = Dl[w] >> sft;
                    uint32_t e = (x & 0x00030003u) * scale, o = ((x >> 8) & 0x00030003u) * scale;
#pragma unroll
                    for (int t = 0; t < KT; ++t) {
                        const uint32_t y = D[poff[t] + w] >> sft;
                        e += (y & 0x00030003u) * cs[t];
                        o += ((y >> 8) & 0x00030003u) * cs[t];
                    }
                    atomicAdd((uint32_t*)(hb + (e & 0xffffu)), 1u);
                    atomicAdd((uint32_t*)(hb + (e >> 16)), 1u);
                    atomicAdd((uint32_t*)(hb + (o & 0xffffu)), 1u);
                    atomicAdd((uint32_t*)(hb + (o >> 16)), 1u);
                }
                __syncwarp();
                if (lane == 0 && A.pad) hist[0] -= A.pad;
            }
            __syncwarp();
            JointLuts L;
            L.x = A.lut + (size_t)A.cell_lut[Q] * A.lut_stride;
            fx128 acc = 0, h[3] = {0, 0, 0};
            const bool parent = j <= A.k;       // a parent set too
            if (parent) {
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (q < A.nv) L.c[q] = A.lut + (size_t)A.cfg_lut[Q * A.nv + q] * A.lut_stride;
            }
            if (MINOR) {
                if (parent) {
                    if (ri == 1) minor_cells<1, true>(hist, pre, Qp, L, A.nv, lane, acc, h);
                    else if (ri == 2) minor_cells<2, true>(hist, pre, Qp, L, A.nv, lane, acc, h);
                    else if (ri == 3) minor_cells<3, true>(hist, pre, Qp, L, A.nv, lane, acc, h);
                    else minor_cells<4, true>(hist, pre, Qp, L, A.nv, lane, acc, h);
                } else {
                    if (ri == 2) minor_cells<2, false>(hist, pre, Qp, L, A.nv, lane, acc, h);
                    else if (ri == 3) minor_cells<3, false>(hist, pre, Qp, L, A.nv, lane, acc, h);
                    else minor_cells<4, false>(hist, pre, Qp, L, A.nv, lane, acc, h);
                }
            } else {
                for (int c = lane; c < Q; c += 32) {
                    const uint32_t v = hist[c];
                    hist[c] = 0u;
                    if (parent) add_cell<true>(v, L, A.nv, acc, h);
                    else add_cell<false>(v, L, A.nv, acc, h);
                }
            }
            if (parent) {
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (q < A.nv) {
                        h[q] = warp_sum_fx(h[q]);
                        if (lane == 0) A.H[(size_t)q * A.S0 + rho] = h[q];
                    }
            }
            acc = warp_sum_fx(acc);
            // lane (rho - r0) % 32 keeps the set's sum; 32 of them go out at once
            const int slot = (int)((rho - r0) & 31);
            if (lane == slot) my_acc = acc;
            if (slot == 31 || rho + 1 == r1) {
                if (lane <= slot) A.G[rho - slot + lane] = my_acc;
                __syncwarp();
            }
            __syncwarp();
            next_set(A.n, j, mask);
        }
        if (MINOR) {
            for (int c = lane; c < Qp; c += 32) pre[c] = 0u;
            __syncwarp();
        }
    }
}

struct AssembleArgs {
    const uint64_t* pst;
    int n, k;
    int64_t S, Sp, S0;
    const fx128* G;
    const fx128* H;
    const uint8_t* arity;
    uint32_t vmap;            // byte r - 1: variant of a child of arity r
    const double* ppf;        // n*n or null
    double log10g;
    int64_t* keys;
};

static constexpr int ASM_BLOCK = 2048;     // entries of a block (its binomial table is paid once)

// One entry a thread at a time: the node-space ranks of pi and pi + {i}, their sums, one
// rounding, / ln 10, the size penalty, the prior of every parent (ascending node ids).
// Consecutive ranks differ in their lowest parents, so both gathers are mostly coalesced.
// Bound by integer instructions and the 16-byte gathers: 0.34 ms at n = 60, k = 4 (0.51 ms
// with the rounding and the division on the FP64 pipe, 0.89 ms with 256 entries a block too).
__global__ void __launch_bounds__(256) k_assemble(AssembleArgs A)
{
    __shared__ int64_t s_bin[65 * (MAXK + 2)];          // C(a, t), t <= k + 1
    __shared__ int64_t s_base[MAXK + 3];                // first rank of every set size
    __shared__ double s_pen[MAXK + 1];                  // its structure penalty
    const int T = A.k + 2;
    for (int q = threadIdx.x; q < 65 * T; q += blockDim.x) s_bin[q] = (int64_t)g_binom.v[q / T][q % T];
    if ((int)threadIdx.x <= A.k) s_pen[threadIdx.x] = __dmul_rn((double)threadIdx.x, A.log10g);
    if (threadIdx.x == 0) {
        int64_t b = 0;
        for (int t = 0; t <= A.k + 1; ++t) {
            s_base[t] = b;
            b += (int64_t)c_binom.v[A.n][t];
        }
    }
    __syncthreads();
    const int i = blockIdx.y;
    const int v = (int)((A.vmap >> (8 * (A.arity[i] - 1))) & 0xffu);
    const fx128* H = A.H + (size_t)v * A.S0;
    const bool penalty = A.log10g != 0.0;
    const int64_t r1 = min((int64_t)(blockIdx.x + 1) * ASM_BLOCK, A.Sp);
#pragma unroll 2
    for (int64_t rho = (int64_t)blockIdx.x * ASM_BLOCK + threadIdx.x; rho < r1; rho += 256) {
        int64_t* out = A.keys + (size_t)i * A.Sp + rho;
        if (rho >= A.S) {
            *out = KEY_NONE;                            // padding
            continue;
        }
        const uint64_t mask = A.pst[rho];
        const int j = __popcll(mask);
        int64_t rp = s_base[j], ru = s_base[j + 1];
        int t = 0, below = 0;
        uint64_t mm = mask;
        while (mm) {
            const int c = __ffsll((long long)mm) - 1;
            mm &= mm - 1;
            const int gt = c >= i;
            const int64_t* row = s_bin + (c + gt) * T + ++t;
            rp += row[0];
            ru += row[gt];
            below += !gt;
        }
        ru += s_bin[i * T + below + 1];
        const fx128 acc = A.G[ru] - H[rp];
        uint64_t bits = fx_div_ln10(acc);
        if (!penalty && !A.ppf) {                       // (adding a zero changes no entry's value)
            *out = key_from_bits(bits);
            continue;
        }
        double ls = __longlong_as_double((long long)bits);
        if (penalty) ls = __dadd_rn(ls, s_pen[j]);
        if (A.ppf) {
            mm = mask;
            while (mm) {
                const int c = __ffsll((long long)mm) - 1;
                mm &= mm - 1;
                ls = __dadd_rn(ls, A.ppf[(size_t)i * A.n + c + (c >= i ? 1 : 0)]);
            }
        }
        *out = double_to_key(ls);
    }
}

// score table upload / readout
__global__ void k_keys_from_scores(const double* __restrict__ sc, int n, int64_t S, int64_t Sp,
                                   int64_t* __restrict__ keys, uint32_t* status)
{
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)n * S) return;
    int64_t i = idx / S, r = idx - i * S;
    double v = sc[idx];
    if (isnan(v) || v == INFINITY) atomicOr(status, STATUS_BADINPUT);
    keys[i * Sp + r] = double_to_key(v);
}

__global__ void k_scores_from_keys(const int64_t* __restrict__ keys, int n0, int nn, int64_t S,
                                   int64_t Sp, double* __restrict__ out)
{
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)nn * S) return;
    int64_t i = idx / S, r = idx - i * S;
    out[idx] = key_to_double(keys[(n0 + i) * Sp + r]);
}

// ---------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------
static int table_alloc(int n, int k, bn_table** out)
{
    bn_table* t = new bn_table();
    t->n = n;
    t->k = k;
    t->dev = device_id();
    t->S = num_sets_host(n - 1, k);
    t->Sp = round_up(t->S, SUBQ);
    cudaError_t e = obj_alloc(&t->keys, sizeof(int64_t) * (size_t)n * (size_t)t->Sp);
    if (e == cudaSuccess) e = obj_alloc(&t->pst, sizeof(uint64_t) * (size_t)t->Sp);
    if (e == cudaSuccess) e = obj_alloc(&t->spos, sizeof(uint32_t) * (size_t)n * (size_t)t->Sp);
    if (e == cudaSuccess) e = obj_alloc(&t->srank, sizeof(uint32_t) * (size_t)n * (size_t)t->Sp);
    if (e == cudaSuccess) e = obj_alloc(&t->spos_t, sizeof(uint32_t) * (size_t)n * (size_t)t->Sp);
    if (e != cudaSuccess) {
        obj_free({t->keys, t->pst, t->spos, t->srank, t->spos_t});
        delete t;
        cudaGetLastError();
        return set_error(BN_ENOMEM, "table allocation of %lld entries failed: %s",
                         (long long)((int64_t)n * num_sets_host(n - 1, k)), cudaGetErrorString(e));
    }
    t->bytes = (sizeof(int64_t) + 3 * sizeof(uint32_t)) * (size_t)n * (size_t)t->Sp + sizeof(uint64_t) * (size_t)t->Sp;
    *out = t;
    return BN_OK;
}

static int build_pst(bn_table* t, cudaStream_t s, bool pad_keys)
{
    int thr = 256;
    const int64_t blocks = (t->Sp / PST_RUN + thr - 1) / thr;
    k_pst<<<(unsigned)blocks, thr, sizeof(uint64_t) * 64 * (t->k + 1), s>>>(t->n - 1, t->k, t->S, t->Sp, t->pst);
    BN_LAUNCH_CHECK("k_pst");
    if (pad_keys && t->Sp > t->S) {
        int64_t tot = (int64_t)t->n * (t->Sp - t->S);
        k_pad_keys<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(t->keys, t->n, t->S, t->Sp);
        BN_LAUNCH_CHECK("k_pad_keys");
    }
    return BN_OK;
}

// RAII list of stream-ordered temporaries
struct Temps {
    cudaStream_t s;
    std::vector<void*> p;
    explicit Temps(cudaStream_t st) : s(st) {}
    template <class T>
    int get(T** out, size_t count)
    {
        void* q = nullptr;
        cudaError_t e = dev_alloc(&q, std::max<size_t>(count, 1) * sizeof(T), s);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return set_error(BN_ENOMEM, "device memory (%zu bytes) failed: %s", count * sizeof(T),
                             cudaGetErrorString(e));
        }
        p.push_back(q);
        *out = (T*)q;
        return BN_OK;
    }
    void release()
    {
        for (void* q : p) dev_free(q, s);
        p.clear();
    }
    ~Temps() { release(); }
};

static constexpr size_t JOINT_SMEM = 220 * 1024;       // of a block of k_joint, at most

template <int KT, bool SMEM_DATA, bool MINOR>
static int launch_joint(const JointArgs& A, size_t smem, int grid, int threads, cudaStream_t s)
{
    // (the limit of every build: one thread's smaller build must not lower another's)
    static ContextOnce once;
    const int rc = once_in_context(once, [&]() -> int {
        BN_CUDA(cudaFuncSetAttribute(k_joint<KT, SMEM_DATA, MINOR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)JOINT_SMEM));
        return BN_OK;
    });
    if (rc) return rc;
    k_joint<KT, SMEM_DATA, MINOR><<<grid, threads, smem, s>>>(A);
    BN_LAUNCH_CHECK("k_joint");
    return BN_OK;
}

template <int KT>
static int launch_joint_kt(const JointArgs& A, bool smem_data, bool base, size_t smem, int grid, int threads,
                           cudaStream_t s)
{
    if (smem_data) return base ? launch_joint<KT, true, true>(A, smem, grid, threads, s)
                               : launch_joint<KT, true, false>(A, smem, grid, threads, s);
    return base ? launch_joint<KT, false, true>(A, smem, grid, threads, s)
                : launch_joint<KT, false, false>(A, smem, grid, threads, s);
}

static int copy_in(void* dst, const void* src, size_t bytes, int mem, cudaStream_t s)
{
    if (bytes == 0) return BN_OK;
    BN_CUDA(cudaMemcpyAsync(dst, src, bytes, mem == BN_MEM_DEVICE ? cudaMemcpyDeviceToDevice
                                                                 : cudaMemcpyHostToDevice, s));
    return BN_OK;
}


}  // namespace bn

using namespace bn;

// Host half of a table build: argument checks and the plan of the lgamma tables.
struct BuildPlan {
    const uint8_t* data = nullptr;
    int m = 0, n = 0, k = 0, mem = BN_MEM_HOST, kind = 0;
    double log10g = 0.0;
    const double* R = nullptr;
    std::vector<uint8_t> ar;
    std::vector<double> Rh;
    int64_t S = 0;
    int cells_max = 1;
    bool one_arity = true;
    int nv = 1;                       // variants of the configuration sums
    uint32_t vmap = 0;                // byte r - 1: variant of a child of arity r
    std::vector<int16_t> cell_lut, cfg_lut;
    std::vector<double> alpha;
};

static int build_plan(const uint8_t* data, int m, int n, const uint8_t* arity, int k, const double* R,
                      const bn_score_params* params, int mem, cudaStream_t s, BuildPlan* P)
{
    if (n < 2 || n > MAXN) return set_error(BN_EINVAL, "bn_build_scores: n=%d outside [2, 64]", n);
    if (m < 0 || (m > 0 && !data)) return set_error(BN_EINVAL, "bn_build_scores: bad data/m");
    if (k < 0 || k > n - 1) return set_error(BN_EINVAL, "bn_build_scores: k=%d outside [0, n-1]", k);
    if (!arity) return set_error(BN_EINVAL, "bn_build_scores: arity is NULL");
    if (mem != BN_MEM_HOST && mem != BN_MEM_DEVICE) return set_error(BN_EINVAL, "bn_build_scores: bad mem");
    if (k > MAXK) return set_error(BN_EUNSUPPORTED, "bn_build_scores: k=%d above %d", k, MAXK);
    int kind = params ? params->score_kind : 0;
    double ess = params ? params->ess : 1.0;
    double log10g = params ? params->log10_gamma : 0.0;
    if (kind != 0 && kind != 1) return set_error(BN_EINVAL, "bn_build_scores: score_kind %d", kind);
    if (kind == 1 && !(ess > 0.0 && std::isfinite(ess))) return set_error(BN_EINVAL, "bn_build_scores: ess must be > 0");
    if (!std::isfinite(log10g)) return set_error(BN_EINVAL, "bn_build_scores: log10_gamma not finite");
    P->data = data;
    P->m = m;
    P->n = n;
    P->k = k;
    P->mem = mem;
    P->kind = kind;
    P->log10g = log10g;
    P->R = R;
    // small arrays are checked on the host
    std::vector<uint8_t>& ar = P->ar;
    std::vector<double>& Rh = P->Rh;
    ar.resize(n);
    if (mem == BN_MEM_DEVICE) {
        BN_CUDA(cudaMemcpyAsync(ar.data(), arity, n, cudaMemcpyDeviceToHost, s));
        if (R) {
            Rh.resize((size_t)n * n);
            BN_CUDA(cudaMemcpyAsync(Rh.data(), R, sizeof(double) * n * n, cudaMemcpyDeviceToHost, s));
        }
        BN_CUDA(cudaStreamSynchronize(s));
    } else {
        memcpy(ar.data(), arity, n);
        if (R) Rh.assign(R, R + (size_t)n * n);
    }
    for (int i = 0; i < n; ++i)
        if (ar[i] < 2 || ar[i] > 4) return set_error(BN_EINVAL, "bn_build_scores: arity[%d]=%d outside [2,4]", i, ar[i]);
    for (size_t t = 0; t < Rh.size(); ++t) {
        if ((int)(t / n) == (int)(t % n)) continue;
        if (!(Rh[t] >= 0.0 && Rh[t] <= 1.0)) return set_error(BN_EINVAL, "bn_build_scores: R[%zu] outside [0,1]", t);
    }
    if (mem == BN_MEM_HOST && m > 0) {
        for (int64_t r = 0; r < (int64_t)m; ++r)
            for (int i = 0; i < n; ++i)
                if (data[r * n + i] >= ar[i])
                    return set_error(BN_EINVAL, "bn_build_scores: data[%lld][%d]=%d >= arity %d", (long long)r, i,
                                     data[r * n + i], ar[i]);
    }
    const int64_t S = num_sets_host(n - 1, k);
    if (S >= (int64_t)1 << 31) return set_error(BN_EUNSUPPORTED, "bn_build_scores: %lld sets per node", (long long)S);
    P->S = S;
    // count-table size bound: r_i times the product of the k largest other arities
    int cells_max = 1;
    for (int i = 0; i < n; ++i) {
        std::vector<int> o;
        for (int p = 0; p < n; ++p)
            if (p != i) o.push_back(ar[p]);
        std::sort(o.rbegin(), o.rend());
        int64_t c = ar[i];
        for (int t = 0; t < k && t < (int)o.size(); ++t) c *= o[t];
        if (c > MAX_CELLS) return set_error(BN_EUNSUPPORTED, "bn_build_scores: count tables up to %lld cells (max %d)",
                                            (long long)c, MAX_CELLS);
        cells_max = std::max<int>(cells_max, (int)c);
    }
    P->cells_max = cells_max;
    P->one_arity = std::count(ar.begin(), ar.end(), ar[0]) == n;

    // LUT plan: K2 uses alpha = 1 for cells and alpha = r for configurations; BDeu uses
    // ess/(q r) and ess/q for every reachable q (products of <= k arities)
    std::set<int> qs = {1};
    for (int t = 0; t < k; ++t) {
        std::set<int> nq = qs;
        for (int q : qs)
            for (int a = 2; a <= 4; ++a)
                if ((int64_t)q * a <= MAX_CELLS / 2) nq.insert(q * a);
        qs.swap(nq);
    }
    // cell_lut[cells of a joint table], cfg_lut[configurations * nv + variant]: a joint
    // table of Q cells is q * r of some reachable q and child arity r, and its alpha is
    // ess / Q whichever; K2's configuration alpha is the child's arity (a variant per
    // arity present), BDeu's is ess / q
    const int qmax = *qs.rbegin();
    std::vector<int16_t>& cell_lut = P->cell_lut;
    std::vector<int16_t>& cfg_lut = P->cfg_lut;
    std::vector<double>& alpha = P->alpha;
    P->vmap = 0;
    P->nv = 1;
    if (kind == 0) {
        P->nv = 0;
        for (int r = 2; r <= 4; ++r)
            if (std::find(ar.begin(), ar.end(), (uint8_t)r) != ar.end()) {
                P->vmap |= (uint32_t)P->nv << (8 * (r - 1));
                ++P->nv;
                alpha.push_back((double)r);
            }
        alpha.push_back(1.0);
        cell_lut.assign((size_t)4 * qmax + 1, (int16_t)(alpha.size() - 1));
        cfg_lut.assign((size_t)(qmax + 1) * P->nv, 0);
        for (size_t q = 0; q < cfg_lut.size(); ++q) cfg_lut[q] = (int16_t)(q % P->nv);
    } else {
        cell_lut.assign((size_t)4 * qmax + 1, 0);
        cfg_lut.assign((size_t)qmax + 1, 0);
        auto table = [&](int v) {
            const double a = ess / (double)v;
            for (size_t x = 0; x < alpha.size(); ++x)
                if (alpha[x] == a) return (int16_t)x;
            alpha.push_back(a);
            return (int16_t)(alpha.size() - 1);
        };
        for (int q : qs) {
            cfg_lut[q] = table(q);
            for (int r = 2; r <= 4; ++r) cell_lut[(size_t)q * r] = table(q * r);
        }
        cell_lut[1] = table(1);
    }
    if (alpha.size() > 32000) return set_error(BN_EUNSUPPORTED, "bn_build_scores: too many lgamma tables");
    return BN_OK;
}

// Device half: every kernel of the build on stream s, writing t (allocated), OR-ing
// STATUS_BADINPUT into d_meta[0] for a data value at or above its arity and leaving the
// nodes' empty-set positions + 1 in d_meta[1..n] (META_WORDS words).  Temporaries are
// stream-ordered; the host waits for the device only where rank_entries takes memory.
static constexpr int META_WORDS = 1 + MAXN;
static int build_enqueue(const BuildPlan& P, bn_table* t, uint32_t* d_meta, cudaStream_t s,
                         cudaEvent_t ev0 = nullptr, cudaEvent_t ev1 = nullptr)
{
    const int n = P.n, m = P.m, k = P.k;
    const std::vector<double>& alpha = P.alpha;
    int rc = BN_OK;
    Temps tmp(s);
    const int mw = (m + 15) / 16;
    uint8_t *d_data = nullptr, *d_ar = nullptr;
    uint32_t* d_packed = nullptr;
    double *d_ppf = nullptr, *d_R = nullptr, *d_alpha = nullptr;
    fx128* d_lut = nullptr;
    int16_t *d_cell = nullptr, *d_cfg = nullptr;
    if ((rc = tmp.get(&d_ar, n)) || (rc = tmp.get(&d_packed, (size_t)n * mw)) ||
        (rc = tmp.get(&d_alpha, alpha.size())) || (rc = tmp.get(&d_lut, alpha.size() * (size_t)(m + 1))) ||
        (rc = tmp.get(&d_cell, P.cell_lut.size())) || (rc = tmp.get(&d_cfg, P.cfg_lut.size())))
        return rc;
    BN_CUDA(cudaMemcpyAsync(d_ar, P.ar.data(), n, cudaMemcpyHostToDevice, s));
    BN_CUDA(cudaMemcpyAsync(d_alpha, alpha.data(), sizeof(double) * alpha.size(), cudaMemcpyHostToDevice, s));
    BN_CUDA(cudaMemcpyAsync(d_cell, P.cell_lut.data(), sizeof(int16_t) * P.cell_lut.size(), cudaMemcpyHostToDevice, s));
    BN_CUDA(cudaMemcpyAsync(d_cfg, P.cfg_lut.data(), sizeof(int16_t) * P.cfg_lut.size(), cudaMemcpyHostToDevice, s));
    if (m > 0) {
        if (P.mem == BN_MEM_DEVICE) d_data = (uint8_t*)P.data;
        else {
            if ((rc = tmp.get(&d_data, (size_t)m * n))) return rc;
            if ((rc = copy_in(d_data, P.data, (size_t)m * n, BN_MEM_HOST, s))) return rc;
        }
        k_pack<<<(n * mw + 255) / 256, 256, 0, s>>>(d_data, m, n, mw, d_ar, d_packed, d_meta);
        BN_LAUNCH_CHECK("k_pack");
    }
    if (P.R) {
        if ((rc = tmp.get(&d_ppf, (size_t)n * n)) || (rc = tmp.get(&d_R, (size_t)n * n))) return rc;
        BN_CUDA(cudaMemcpyAsync(d_R, P.Rh.data(), sizeof(double) * n * n, cudaMemcpyHostToDevice, s));
        k_ppf<<<(n * n + 255) / 256, 256, 0, s>>>(d_R, n, d_ppf);
        BN_LAUNCH_CHECK("k_ppf");
    }
    {
        int64_t tot = (int64_t)alpha.size() * (m + 1);
        k_lut<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(d_alpha, (int)alpha.size(), m + 1, d_lut);
        BN_LAUNCH_CHECK("k_lut");
    }
    if ((rc = build_pst(t, s, false))) return rc;

    // joint sets over all n nodes; the LUT index of every table size
    JointArgs A;
    A.packed = d_packed;
    A.n = n;
    A.mw = mw;
    A.pad = (uint32_t)(16 * mw - m);
    A.k = k;
    A.S0 = num_sets_host(n, k);
    A.S1 = num_sets_host(n, k + 1);
    A.cells_cap = (int)round_up(P.cells_max, 32);
    A.arity = d_ar;
    A.lut = d_lut;
    A.lut_stride = m + 1;
    A.cell_lut = d_cell;
    A.cfg_lut = d_cfg;
    A.nv = P.nv;
    A.m = m;
    uint16_t* d_minor = nullptr;
    uint32_t* d_len = nullptr;
    Temps sums(s);
    if ((rc = sums.get(&A.G, (size_t)A.S1)) || (rc = sums.get(&A.H, (size_t)A.S0 * P.nv))) return rc;
    // the largest sets -- nearly all of them -- and those of four nodes on the tensor cores
    // where they are many and one set of lgamma tables serves them all (K2; BDeu with one arity)
    TcPlan tcp[2];                    // k + 1 nodes; four nodes where they are parent sets too
    bool tc[2] = {false, false};
    uint8_t* d_tc[2] = {nullptr, nullptr};
    if (P.kind == 0 || P.one_arity) {
        tc[0] = joint_tc_plan(n, m, k + 1, 1, P.ar.data(), &tcp[0]);
        tc[1] = tc[0] && k == 4 && joint_tc_plan(n, m, k, 1 + P.nv, P.ar.data(), &tcp[1]);
    }
    for (int q = 0; q < 2; ++q) {
        if (!tc[q]) continue;
        if (sums.get(&d_tc[q], joint_tc_scratch(tcp[q], m))) {      // no room: count them as the others
            set_error(BN_OK, "");
            tc[q] = false;
            if (!q) tc[1] = false;
        } else if ((rc = joint_tc_upload(tcp[q], d_tc[q], s)))
            return rc;
    }
    if (tc[0]) A.S1 = tc[1] ? num_sets_host(n, k - 1) : A.S0;
    // Shared memory of a block: the histograms, with `base` the rows' offsets, and the packed
    // data as long as two blocks fit an SM with them
    const int nwarps = BUILD_THREADS / 32;
    const size_t data_bytes = sizeof(uint32_t) * (size_t)n * mw;
    const size_t per_hist = sizeof(uint32_t) * (size_t)A.cells_cap, per_base = (size_t)mw * 32;
    static_assert(sizeof(uint32_t) * MAX_CELLS * (BUILD_THREADS / 32) <= JOINT_SMEM, "the histograms of a block fit");
    size_t smem = 0;
    bool smem_data = false;
    int per_sm = 1;
    auto shape = [&](bool base) {
        smem = nwarps * (per_hist + (base ? per_base : 0));
        smem_data = smem + data_bytes <= JOINT_SMEM / 2;
        if (smem_data) smem += data_bytes;
        per_sm = std::max(1, std::min(2048 / (32 * nwarps), (int)((224 * 1024) / std::max<size_t>(smem + 1024, 1))));
        return (int64_t)sm_count() * per_sm * nwarps;               // resident warps
    };
    // The rows' offsets pay while two blocks an SM hold them and, up to k = 4, a warp keeps
    // them for a few sets (five a unit) and there are not many rows: beyond, fewer warps are
    // resident, with 16,000 rows a quarter of those without.  us of k_joint with and without,
    // two to four states, BDeu: 37 nodes, k = 4, m = 1,000 480 / 593, 2,500 920 / 960, 4,000
    // 1,742 / 1,390, 8,000 5,262 / 2,532; 30 nodes, m = 900 (4 sets a unit) 312 / 268, 1,000
    // (5) 233 / 271; k = 3, ternary, m = 1,000 67 / 63, 16,000 1,088 / 360.  k = 5, binary, 24
    // nodes: m = 1,000 277 / 302, 5,000 614 / 896.
    bool base = m > 0 && m <= LIST_ROWS && nwarps * (per_hist + per_base) <= JOINT_SMEM / 2;
    if (base && k <= 4) base = m <= 2500 && A.S1 >= 5 * 8 * shape(true);
    const int64_t warps = shape(base);
    // 8 to 64 sets a unit: about eight units a resident warp where there are enough sets
    A.range = (int)std::max<int64_t>(4, std::min<int64_t>(64, A.S1 / (8 * warps)));
    const int64_t units = (A.S1 + A.range - 1) / A.range;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sm_count() * per_sm, (units + nwarps - 1) / nwarps));
    if (ev0) BN_CUDA(cudaEventRecord(ev0, s));
    if (base) {
        if ((rc = sums.get(&d_minor, (size_t)n * m)) || (rc = sums.get(&d_len, (size_t)n))) return rc;
        k_minor_rows<<<n, 256, 0, s>>>(d_packed, m, mw, d_minor, d_len);
        BN_LAUNCH_CHECK("k_minor_rows");
    }
    A.minor = d_minor;
    A.minor_len = d_len;
    const int thr = 32 * nwarps;
    if (k <= 2) rc = launch_joint_kt<2>(A, smem_data, base, smem, grid, thr, s);
    else if (k <= 4) rc = launch_joint_kt<4>(A, smem_data, base, smem, grid, thr, s);
    else if (k <= 8) rc = launch_joint_kt<8>(A, smem_data, base, smem, grid, thr, s);
    else rc = launch_joint_kt<12>(A, smem_data, base, smem, grid, thr, s);
    if (rc) return rc;
    for (int q = 0; q < 2; ++q) {
        if (!tc[q]) continue;
        int Q = 1;                    // cells of a set (K2's tables serve any number)
        for (int j = 0; j < k + 1 - q; ++j) Q *= P.ar[0];
        TcJoint J{n, m, mw, k + 1 - q, q ? P.nv : 0, d_ar, d_packed, {}, A.G, A.H, A.S0, d_meta, d_tc[q]};
        J.lut[0] = d_lut + (size_t)P.cell_lut[P.kind == 0 ? 1 : Q] * (m + 1);
        for (int v = 0; v < J.nh; ++v)
            J.lut[1 + v] = d_lut + (size_t)P.cfg_lut[(P.kind == 0 ? 1 : Q) * P.nv + v] * (m + 1);
        if ((rc = launch_joint_tc(J, tcp[q], s))) return rc;
    }
    AssembleArgs B{t->pst, n, k, P.S, t->Sp, A.S0, A.G, A.H, d_ar, P.vmap, d_ppf, P.log10g, t->keys};
    k_assemble<<<dim3((unsigned)((t->Sp + ASM_BLOCK - 1) / ASM_BLOCK), (unsigned)n), 256, 0, s>>>(B);
    BN_LAUNCH_CHECK("k_assemble");
    if (ev1) BN_CUDA(cudaEventRecord(ev1, s));
    sums.release();
    return rank_entries(t, d_meta + 1, s);
}

// the status word and the table's empty-set positions, once the work on s is done
static int read_meta(const uint32_t* d_meta, bn_table* t, uint32_t* status, cudaStream_t s)
{
    uint32_t h[META_WORDS];
    BN_CUDA(cudaMemcpyAsync(h, d_meta, sizeof(uint32_t) * (1 + t->n), cudaMemcpyDeviceToHost, s));
    BN_CUDA(cudaStreamSynchronize(s));
    *status = h[0];
    memcpy(t->cut, h + 1, sizeof(uint32_t) * t->n);
    return BN_OK;
}

static int build_scores_impl(const uint8_t* data, int m, int n, const uint8_t* arity, int k, const double* R,
                             const bn_score_params* params, int mem, void* stream, bn_table** out,
                             cudaEvent_t ev0, cudaEvent_t ev1)
{
    set_error(BN_OK, "");
    if (!out) return set_error(BN_EINVAL, "bn_build_scores: out is NULL");
    *out = nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    BuildPlan P;
    int rc = build_plan(data, m, n, arity, k, R, params, mem, s, &P);
    if (rc) return rc;
    bn_table* t = nullptr;
    if ((rc = table_alloc(n, k, &t))) return rc;
    struct Guard {
        bn_table*& t;
        bool ok = false;
        ~Guard()
        {
            if (!ok && t) bn_table_free(t);
        }
    } guard{t};
    uint32_t* d_meta = nullptr;
    {
        Temps tmp(s);
        if ((rc = tmp.get(&d_meta, META_WORDS))) return rc;
        BN_CUDA(cudaMemsetAsync(d_meta, 0, sizeof(uint32_t), s));
        if ((rc = build_enqueue(P, t, d_meta, s, ev0, ev1))) return rc;
        uint32_t st = 0;
        if ((rc = read_meta(d_meta, t, &st, s))) return rc;
        if (st & STATUS_BADINPUT) return set_error(BN_EINVAL, "bn_build_scores: a data value is >= its arity");
        if (st & STATUS_TIMEOUT) return set_error(BN_ETIMEOUT, "bn_build_scores: a bounded device wait expired");
    }
    guard.ok = true;
    *out = t;
    return BN_OK;
}

extern "C" int bn_build_scores(const uint8_t* data, int m, int n, const uint8_t* arity, int k,
                               const double* R, const bn_score_params* params, int mem,
                               void* stream, bn_table** out)
{
    return build_scores_impl(data, m, n, arity, k, R, params, mem, stream, out, nullptr, nullptr);
}

extern "C" int bn_build_scores_profiled(const uint8_t* data, int m, int n, const uint8_t* arity, int k,
                                        const double* R, const bn_score_params* params, int mem,
                                        void* stream, bn_table** out, double* build_ms)
{
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        return cuda_fail(cudaGetLastError(), "cudaEventCreate", __FILE__, __LINE__);
    }
    int rc = build_scores_impl(data, m, n, arity, k, R, params, mem, stream, out, e0, e1);
    float ms = 0.f;
    if (rc == BN_OK && cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess)
        rc = cuda_fail(cudaGetLastError(), "cudaEventElapsedTime", __FILE__, __LINE__);
    if (build_ms) *build_ms = (double)ms;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}

extern "C" int bn_build_scores_batch(int count, const uint8_t* const* data, const int* m, const int* n,
                                     const uint8_t* const* arity, const int* k, const double* const* R,
                                     const bn_score_params* params, int mem, void* stream, bn_table** out)
{
    set_error(BN_OK, "");
    if (count < 1 || !data || !m || !n || !arity || !k || !out)
        return set_error(BN_EINVAL, "bn_build_scores_batch: bad arguments");
    for (int i = 0; i < count; ++i) out[i] = nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<BuildPlan> plans(count);
    for (int i = 0; i < count; ++i) {
        int rc = build_plan(data[i], m[i], n[i], arity[i], k[i], R ? R[i] : nullptr, params ? &params[i] : nullptr,
                            mem, s, &plans[i]);
        if (rc) {
            std::string msg = bn_last_error();
            return set_error(rc, "bn_build_scores_batch: network %d: %s", i, msg.c_str());
        }
    }
    std::vector<bn_table*> tabs(count, nullptr);
    struct Guard {
        std::vector<bn_table*>& t;
        bool ok = false;
        ~Guard()
        {
            if (!ok)
                for (bn_table* x : t) bn_table_free(x);
        }
    } guard{tabs};
    for (int i = 0; i < count; ++i) {
        int rc = table_alloc(n[i], k[i], &tabs[i]);
        if (rc) return rc;
    }
    // the builds run on a few side streams that fork from and join into `stream`; the
    // largest networks are spread over the streams first
    std::vector<int> order(count);
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return (double)n[a] * (double)plans[a].S * (double)(m[a] + 1) > (double)n[b] * (double)plans[b].S * (double)(m[b] + 1);
    });
    const int ns = std::min(count, 4);
    std::vector<cudaStream_t> side(ns, nullptr);
    std::vector<cudaEvent_t> ev(ns + 1, nullptr);
    struct Streams {
        std::vector<cudaStream_t>& s;
        std::vector<cudaEvent_t>& e;
        ~Streams()
        {
            for (cudaStream_t x : s)
                if (x) cudaStreamDestroy(x);
            for (cudaEvent_t x : e)
                if (x) cudaEventDestroy(x);
        }
    } sg{side, ev};
    uint32_t* d_meta = nullptr;
    BN_CUDA(dev_alloc((void**)&d_meta, sizeof(uint32_t) * META_WORDS * count, s));
    struct Free {
        uint32_t* p;
        cudaStream_t s;
        ~Free() { dev_free(p, s); }
    } fr{d_meta, s};
    BN_CUDA(cudaMemsetAsync(d_meta, 0, sizeof(uint32_t) * META_WORDS * count, s));
    for (int j = 0; j <= ns; ++j) BN_CUDA(cudaEventCreateWithFlags(&ev[j], cudaEventDisableTiming));
    BN_CUDA(cudaEventRecord(ev[ns], s));
    for (int j = 0; j < ns; ++j) {
        BN_CUDA(cudaStreamCreateWithFlags(&side[j], cudaStreamNonBlocking));
        BN_CUDA(cudaStreamWaitEvent(side[j], ev[ns], 0));
    }
    int rc = BN_OK;
    for (int q = 0; q < count && !rc; ++q) {
        const int i = order[q];
        rc = build_enqueue(plans[i], tabs[i], d_meta + (size_t)META_WORDS * i, side[q % ns]);
    }
    for (int j = 0; j < ns; ++j) {
        cudaEventRecord(ev[j], side[j]);
        cudaStreamWaitEvent(s, ev[j], 0);
    }
    if (rc) {
        cudaStreamSynchronize(s);
        return rc;
    }
    std::vector<uint32_t> st((size_t)META_WORDS * count, 0);
    BN_CUDA(cudaMemcpyAsync(st.data(), d_meta, sizeof(uint32_t) * st.size(), cudaMemcpyDeviceToHost, s));
    BN_CUDA(cudaStreamSynchronize(s));
    for (int i = 0; i < count; ++i) memcpy(tabs[i]->cut, &st[(size_t)META_WORDS * i + 1], sizeof(uint32_t) * n[i]);
    for (int i = 0; i < count; ++i)
        if (st[(size_t)META_WORDS * i] & STATUS_BADINPUT)
            return set_error(BN_EINVAL, "bn_build_scores_batch: network %d: a data value is >= its arity", i);
    for (int i = 0; i < count; ++i)
        if (st[(size_t)META_WORDS * i] & STATUS_TIMEOUT)
            return set_error(BN_ETIMEOUT, "bn_build_scores_batch: network %d: a bounded device wait expired", i);
    guard.ok = true;
    for (int i = 0; i < count; ++i) out[i] = tabs[i];
    return BN_OK;
}

extern "C" int bn_table_from_scores(const double* scores, int n, int k, int mem, void* stream, bn_table** out)
{
    set_error(BN_OK, "");
    if (!out) return set_error(BN_EINVAL, "bn_table_from_scores: out is NULL");
    *out = nullptr;
    if (n < 2 || n > MAXN || k < 0 || k > n - 1 || !scores)
        return set_error(BN_EINVAL, "bn_table_from_scores: bad n/k/scores");
    if (mem != BN_MEM_HOST && mem != BN_MEM_DEVICE) return set_error(BN_EINVAL, "bn_table_from_scores: bad mem");
    const int64_t S = num_sets_host(n - 1, k);
    if (S >= (int64_t)1 << 31) return set_error(BN_EUNSUPPORTED, "bn_table_from_scores: too many sets");
    cudaStream_t s = (cudaStream_t)stream;
    bn_table* t = nullptr;
    int rc = table_alloc(n, k, &t);
    if (rc) return rc;
    Temps tmp(s);
    double* d_sc = nullptr;
    uint32_t* d_meta = nullptr;
    if ((rc = tmp.get(&d_meta, META_WORDS))) { bn_table_free(t); return rc; }
    if (mem == BN_MEM_DEVICE) d_sc = (double*)scores;
    else {
        if ((rc = tmp.get(&d_sc, (size_t)n * S))) { bn_table_free(t); return rc; }
        if ((rc = copy_in(d_sc, scores, sizeof(double) * (size_t)n * S, BN_MEM_HOST, s))) { bn_table_free(t); return rc; }
    }
    if (cudaMemsetAsync(d_meta, 0, 4, s) != cudaSuccess) { bn_table_free(t); return cuda_fail(cudaGetLastError(), "memset", __FILE__, __LINE__); }
    int64_t tot = (int64_t)n * S;
    k_keys_from_scores<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(d_sc, n, S, t->Sp, t->keys, d_meta);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { bn_table_free(t); return cuda_fail(e, "k_keys_from_scores", __FILE__, __LINE__); }
    count_launches(1);
    if ((rc = build_pst(t, s, true))) { bn_table_free(t); return rc; }
    if ((rc = rank_entries(t, d_meta + 1, s))) { bn_table_free(t); return rc; }
    uint32_t st = 0;
    if ((rc = read_meta(d_meta, t, &st, s))) { bn_table_free(t); return rc; }
    if (st) { bn_table_free(t); return set_error(BN_EINVAL, "bn_table_from_scores: NaN or +inf score"); }
    *out = t;
    return BN_OK;
}

extern "C" int bn_table_info(const bn_table* t, int* n, int* k, int64_t* sets_per_node, int64_t* device_bytes)
{
    if (!t) return set_error(BN_EINVAL, "bn_table_info: NULL table");
    if (n) *n = t->n;
    if (k) *k = t->k;
    if (sets_per_node) *sets_per_node = t->S;
    if (device_bytes) *device_bytes = (int64_t)t->bytes;
    return BN_OK;
}

extern "C" int bn_table_scores(const bn_table* t, int node, double* out, int mem, void* stream)
{
    set_error(BN_OK, "");
    if (!t || !out) return set_error(BN_EINVAL, "bn_table_scores: NULL argument");
    if (node < -1 || node >= t->n) return set_error(BN_EINVAL, "bn_table_scores: node %d", node);
    if (mem != BN_MEM_HOST && mem != BN_MEM_DEVICE) return set_error(BN_EINVAL, "bn_table_scores: bad mem");
    cudaStream_t s = (cudaStream_t)stream;
    int n0 = node < 0 ? 0 : node, nn = node < 0 ? t->n : 1;
    int64_t tot = (int64_t)nn * t->S;
    Temps tmp(s);
    double* d = nullptr;
    int rc;
    if (mem == BN_MEM_DEVICE) d = out;
    else if ((rc = tmp.get(&d, (size_t)tot))) return rc;
    k_scores_from_keys<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(t->keys, n0, nn, t->S, t->Sp, d);
    BN_LAUNCH_CHECK("k_scores_from_keys");
    if (mem == BN_MEM_HOST) BN_CUDA(cudaMemcpyAsync(out, d, sizeof(double) * tot, cudaMemcpyDeviceToHost, s));
    BN_CUDA(cudaStreamSynchronize(s));
    return BN_OK;
}

extern "C" void bn_table_free(bn_table* t)
{
    if (!t) return;
    obj_free({t->keys, t->pst, t->spos, t->srank, t->spos_t, t->sset, t->alive_block, t->gcache});
    delete t;
}
