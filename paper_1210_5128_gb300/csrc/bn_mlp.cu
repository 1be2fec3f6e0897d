// bn_mlp.cu -- the learned swap proposal: a small MLP over the current order whose
// output is a distribution over the n(n-1)/2 swap pairs, used inside an exact MH ratio.
// The paper proposes uniform swaps (Sec. III.C); this network and its training target
// are the build's own specification (see include/bn.h).
//
// Dense layers run on the 5th-generation tensor cores: k_gemm_tc is a bf16 x bf16 -> f32
// GEMM, C = A B^T with both operands K-major, 128 x 128 tiles, a 3-stage cp.async
// pipeline into no-swizzle core-matrix shared-memory layouts, tcgen05.mma issued by one
// thread into a TMEM accumulator, completion through tcgen05.commit on an mbarrier, and
// a tcgen05.ld epilogue.  Bias, ReLU, bf16 rounding, transposed copies, the loss
// gradient, the scatter of the embedding gradient and Adam are small elementwise kernels.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "bn_tc.cuh"
#include "bn_mlp.cuh"

namespace bn {

typedef __nv_bfloat16 bf16;

static constexpr int TC_BM = 128, TC_BN = 128, TC_BK = 64, TC_STAGES = 3;
static constexpr int TC_TILE = TC_BM * TC_BK * 2;                       // bytes of one operand tile
static constexpr size_t TC_SMEM = 2 * TC_STAGES * TC_TILE + 256 + 1024;  // tiles + barriers + align slack
static constexpr uint32_t TC_IDESC = tc_idesc_bf16_f32(TC_BM, TC_BN);

struct GemmArgs {
    const bf16* A;   // M x K, row stride lda (elements)
    const bf16* B;   // N x K, row stride ldb
    float* C;        // M x N, row stride ldc; with split-K: partials [split][M][N]
    int M, N, K, lda, ldb, ldc;
    int ksplit;      // K / ksplit per CTA along grid z (1 = no split)
    uint32_t* status;
};

// core-matrix layout of a 128 x 64 bf16 tile: row r, 16-byte chunk kc of the row
__device__ __forceinline__ uint32_t tc_tile_off(int r, int kc) { return (r >> 3) * 1024 + kc * 128 + (r & 7) * 16; }

// Up to two independent products in one launch (the weight and the input gradient of a
// layer): blocks below `blocks0` belong to the first.
struct GemmPair {
    GemmArgs g[2];
    int blocks0;
};

__global__ void __launch_bounds__(128) k_gemm_tc(GemmPair gp)
{
    const bool second = (int)blockIdx.x >= gp.blocks0;
    const GemmArgs& g = gp.g[second];
    int tile = blockIdx.x - (second ? gp.blocks0 : 0);
    const int tn = g.N / TC_BN, tm = g.M / TC_BM;
    const int bx = tile % tn;
    tile /= tn;
    const int by = tile % tm, bz = tile / tm;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sB = smem + TC_STAGES * TC_TILE;
    uint64_t* bar = (uint64_t*)(smem + 2 * TC_STAGES * TC_TILE);
    uint32_t* tslot = (uint32_t*)(bar + TC_STAGES);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = by * TC_BM, n0 = bx * TC_BN;
    const int kpart = g.K / g.ksplit;               // this CTA's K range (multiple of 64)
    const int kbase = bz * kpart;
    const int nk = kpart / TC_BK;
    float* Cz = g.C + (size_t)bz * g.M * g.ldc;

    if (warp == 0) {
        tc_alloc(tslot, 128);
        tc_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < TC_STAGES; ++s) mbar_init(&bar[s], 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    auto load_stage = [&](int kt, int s) {
        uint8_t* a = sA + s * TC_TILE;
        uint8_t* b = sB + s * TC_TILE;
        for (int c = tid; c < TC_BM * 8; c += 128) {
            const int r = c >> 3, kc = c & 7;
            cp_async16(a + tc_tile_off(r, kc), g.A + (size_t)(m0 + r) * g.lda + kbase + kt * TC_BK + kc * 8);
            cp_async16(b + tc_tile_off(r, kc), g.B + (size_t)(n0 + r) * g.ldb + kbase + kt * TC_BK + kc * 8);
        }
        cp_async_commit();
    };

    for (int s = 0; s < TC_STAGES - 1; ++s) {
        if (s < nk) load_stage(s, s);
        else cp_async_commit();
    }
    bool ok = true;
    for (int kt = 0; kt < nk; ++kt) {
        const int s = kt % TC_STAGES;
        const int kp = kt + TC_STAGES - 1;
        if (kp < nk) {
            const int sp = kp % TC_STAGES;        // last read by the MMAs of step kt-1
            if (kt >= 1) ok &= mbar_wait_bounded(&bar[sp], (uint32_t)(((kt - 1) / TC_STAGES) & 1), WAIT_TIMEOUT_NS);
            load_stage(kp, sp);
        } else {
            cp_async_commit();
        }
        cp_async_wait<TC_STAGES - 1>();            // step kt's tiles have landed
        fence_proxy_async_smem();                  // visible to the tensor core's async proxy
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < TC_BK / 16; ++kk) {
                const uint64_t ad = tc_smem_desc(sA + s * TC_TILE + kk * 256, 128, 1024);
                const uint64_t bd = tc_smem_desc(sB + s * TC_TILE + kk * 256, 128, 1024);
                tc_mma_bf16(tmem, ad, bd, TC_IDESC, (kt > 0) || (kk > 0));
            }
            tc_commit(&bar[s]);
        }
    }
    if (nk > 0) ok &= mbar_wait_bounded(&bar[(nk - 1) % TC_STAGES], (uint32_t)(((nk - 1) / TC_STAGES) & 1),
                                        WAIT_TIMEOUT_NS);
    tc_fence_after();
    const bool all_ok = __syncthreads_and(ok);
    if (all_ok) {
        const int row = m0 + warp * 32 + lane;
        for (int c0 = 0; c0 < TC_BN; c0 += 32) {
            uint32_t r[32];
            tc_ld_32x32b_x32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
            tc_wait_ld();
            float* dst = Cz + (size_t)row * g.ldc + n0 + c0;
            if (nk > 0) {
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    *(float4*)(dst + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                      __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
            } else {
#pragma unroll
                for (int j = 0; j < 32; j += 4) *(float4*)(dst + j) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    } else if (tid == 0) {
        atomicOr(g.status, STATUS_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tc_dealloc(tmem, 128);
}

// C = sum over the split partials, in split order (deterministic)
__global__ void k_splitk_reduce(const float* __restrict__ ws, int ksplit, int M, int N, float* __restrict__ C,
                                int ldc)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)M * N) return;
    const int r = (int)(idx / N), c = (int)(idx - (int64_t)r * N);
    float s = 0.f;
    for (int z = 0; z < ksplit; ++z) s += ws[(size_t)z * M * N + idx];
    C[(size_t)r * ldc + c] = s;
}

// Few output tiles and a long K split K (each part at least four 64-wide stages) into
// partials that the consumer adds in split order
static int gemm_split(int M, int N, int K, size_t ws_elems)
{
    const int tiles = (M / TC_BM) * (N / TC_BN), stages = K / TC_BK;
    const int lim = std::min(sm_count() / std::max(tiles, 1), stages / 4);
    for (int dv = lim; dv >= 2; --dv)
        if (stages % dv == 0 && (size_t)dv * M * N <= ws_elems) return dv;
    return 1;
}

static int gemm_launch(const GemmArgs& a, const GemmArgs* b, cudaStream_t s)
{
    static ContextOnce once;
    const int rc = once_in_context(once, [&]() -> int {
        BN_CUDA(cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM));
        return BN_OK;
    });
    if (rc) return rc;
    auto blocks = [](const GemmArgs& g) { return (g.M / TC_BM) * (g.N / TC_BN) * g.ksplit; };
    GemmPair gp{{a, b ? *b : a}, blocks(a)};
    k_gemm_tc<<<(unsigned)(gp.blocks0 + (b ? blocks(*b) : 0)), 128, TC_SMEM, s>>>(gp);
    BN_LAUNCH_CHECK("k_gemm_tc");
    return BN_OK;
}

// C = A B^T, whole
static int gemm_tc(const bf16* A, int lda, const bf16* B, int ldb, float* C, int ldc, int M, int N, int K,
                   uint32_t* status, cudaStream_t s, float* ws, size_t ws_elems)
{
    if (M % TC_BM || N % TC_BN || K % TC_BK)
        return set_error(BN_EINVAL, "gemm: M=%d N=%d K=%d must be multiples of 128, 128, 64", M, N, K);
    const int split = ws ? gemm_split(M, N, K, ws_elems) : 1;
    GemmArgs g{A, B, split > 1 ? ws : C, M, N, K, lda, ldb, split > 1 ? N : ldc, split, status};
    const int rc = gemm_launch(g, nullptr, s);
    if (rc) return rc;
    if (split > 1) {
        const int64_t tot = (int64_t)M * N;
        k_splitk_reduce<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(ws, split, M, N, C, ldc);
        BN_LAUNCH_CHECK("k_splitk_reduce");
    }
    return BN_OK;
}

// An M x N product as the GEMM left it: C, or the split partials the reader has to add
struct Product {
    const float* p;
    int split;
    int64_t stride;              // elements between partials
    __device__ __forceinline__ float at(int64_t idx) const
    {
        if (split == 1) return p[idx];
        float s = 0.f;
        for (int z0 = 0; z0 < split; z0 += 8) {
            float a[8];                                             // eight loads in flight
#pragma unroll
            for (int z = 0; z < 8; ++z) a[z] = z0 + z < split ? p[(size_t)(z0 + z) * stride + idx] : 0.f;
#pragma unroll
            for (int z = 0; z < 8; ++z)
                if (z0 + z < split) s += a[z];
        }
        return s;
    }
};

// ---------------------------------------------------------------------------------
// elementwise kernels
// ---------------------------------------------------------------------------------

// The elementwise kernels of the dense layers work on 32 x 32 tiles, 32 x 8 threads, so that
// the transposed copies the weight gradients read go out coalesced through shared memory.
// dst [.., ld] natural, dstT [.., ldt] transposed (may be null).
__device__ __forceinline__ void store_tile(bf16 (&tile)[32][33], const bf16 (&v)[4], int r0, int c0, bf16* dst, int ld,
                                           bf16* dstT, int ldt)
{
    const int x = threadIdx.x, y = threadIdx.y;
#pragma unroll
    for (int k = 0; k < 4; ++k) dst[(size_t)(r0 + y + 8 * k) * ld + c0 + x] = v[k];
    if (!dstT) return;                                              // block-uniform
#pragma unroll
    for (int k = 0; k < 4; ++k) tile[y + 8 * k][x] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) dstT[(size_t)(c0 + y + 8 * k) * ldt + r0 + x] = tile[x][y + 8 * k];
}

// x rows: X[r][p*d + j] = E[order_r(p)][j] (bf16), zero padding; XT and inv (the inverse
// orders: inv[r * 64 + v] = position of node v in order r) for training.  An entry that is no
// node counts as zero and sets STATUS_BADINPUT.
__global__ void __launch_bounds__(256) k_embed(const uint8_t* __restrict__ orders, int B, int n, int d, int ndp, int Mp,
                                               const bf16* __restrict__ Eb, bf16* __restrict__ X, bf16* __restrict__ XT,
                                               uint8_t* __restrict__ inv, uint32_t* status)
{
    __shared__ bf16 tile[32][33];
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32, col = c0 + threadIdx.x;
    const int p = col / d, j = col - p * d;
    bf16 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int r = r0 + threadIdx.y + 8 * k;
        v[k] = __float2bfloat16_rn(0.f);
        if (r < B && p < n) {
            const int o = orders[(size_t)r * n + p];
            if (o < n) {
                v[k] = Eb[(size_t)o * d + j];
                if (inv && j == 0) inv[(size_t)r * 64 + o] = (uint8_t)p;
            } else {
                atomicOr(status, STATUS_BADINPUT);
            }
        }
    }
    store_tile(tile, v, r0, c0, X, ndp, XT, Mp);
}

// Z = the product + bias; H = bf16(relu(Z)) (rows >= B -> 0); HT optional
__global__ void __launch_bounds__(256) k_bias_relu(Product in, float* __restrict__ Z, const float* __restrict__ bias,
                                                   int Mp, int N, int B, bf16* __restrict__ H, bf16* __restrict__ HT)
{
    __shared__ bf16 tile[32][33];
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32, c = c0 + threadIdx.x;
    bf16 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int r = r0 + threadIdx.y + 8 * k;
        const int64_t idx = (int64_t)r * N + c;
        const float z = in.at(idx) + bias[c];
        Z[idx] = z;
        v[k] = __float2bfloat16_rn(r < B ? fmaxf(z, 0.f) : 0.f);
    }
    store_tile(tile, v, r0, c0, H, N, HT, Mp);
}

// Z = the product + bias; for training the rest of the grid clears the output layer's
// gradients (only the rows of the batch's pairs are written later)
__global__ void __launch_bounds__(256) k_bias(Product in, float* __restrict__ Z, const float* __restrict__ bias, int Mp,
                                              int N, float4* __restrict__ zero, int64_t zeros)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t tot = (int64_t)Mp * N;
    if (idx < tot) Z[idx] = in.at(idx) + bias[idx % N];
    else if (idx - tot < zeros) zero[idx - tot] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// output layer gradient of the BCE loss (one logit per row): block per row.  The row's
// d loss / d logit and loss term go to grow[r] and lrow[r]; k_out_grad_w and k_loss_sum
// sum them in row order, so the gradients and the loss do not depend on scheduling.  A pair
// that does not exist counts as pair 0 here and nowhere in gW3, and sets STATUS_BADINPUT.
__global__ void k_out_grad(const float* __restrict__ L, int ldl, const uint32_t* __restrict__ pairs,
                           const float* __restrict__ alpha, int B, int P, int Mp, int H, const float* __restrict__ Z2,
                           const bf16* __restrict__ W3b, bf16* __restrict__ dZ2, bf16* __restrict__ dZ2T,
                           float* __restrict__ grow, float* __restrict__ lrow, uint32_t* status)
{
    const int r = blockIdx.x;
    float g = 0.f;
    int p = 0;
    if (r < B) {
        p = pairs[r] < (uint32_t)P ? (int)pairs[r] : 0;
        if (threadIdx.x == 0 && pairs[r] >= (uint32_t)P) atomicOr(status, STATUS_BADINPUT);
        const float l = L[(size_t)r * ldl + p];
        const float s = 1.f / (1.f + expf(-l));
        const float a = alpha[r];
        g = (s - a) / (float)B;
        if (threadIdx.x == 0) {
            lrow[r] = -(a * logf(s + 1e-30f) + (1.f - a) * logf(1.f - s + 1e-30f)) / (float)B;
            grow[r] = g;
        }
    }
    for (int c = threadIdx.x; c < H; c += blockDim.x) {
        bf16 dz = __float2bfloat16_rn(0.f);
        if (r < B) {
            const float dh = g * __bfloat162float(W3b[(size_t)p * H + c]);
            dz = __float2bfloat16_rn(Z2[(size_t)r * H + c] > 0.f ? dh : 0.f);
        }
        dZ2[(size_t)r * H + c] = dz;
        dZ2T[(size_t)c * Mp + r] = dz;
    }
}

// Column sums over the first B rows of a bf16 matrix (a bias gradient), 32 columns a block:
// the rows come in side by side through shared memory, each column adds them in row order.
static constexpr int CS_ROWS = 128;
__device__ __forceinline__ void colsum_block(float (&s_t)[CS_ROWS][33], const bf16* __restrict__ M, int N, int B, int c0,
                                             float* __restrict__ out)
{
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    float s = 0.f;
    for (int r0 = 0; r0 < B; r0 += CS_ROWS) {
        const int rows = min(CS_ROWS, B - r0);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < CS_ROWS / 8; ++k) {
            const int r = y + 8 * k;
            if (r < rows) s_t[r][x] = __bfloat162float(M[(size_t)(r0 + r) * N + c0 + x]);
        }
        __syncthreads();
        if (y == 0) {
#pragma unroll 8
            for (int r = 0; r < rows; ++r) s += s_t[r][x];
        }
    }
    if (y == 0) out[c0 + x] = s;
}

// What follows from the output layer's row gradients, one launch: blocks below B the gW3 and
// gb3 rows of the pairs the batch touches (the block of the first row holding a pair sums
// that pair's rows in row order, the others of the pair leave it), then H / 32 blocks the
// column sums of dZ2 (gb2), the last block the batch loss (per thread a strided run, then a
// fixed shared-memory tree).
__global__ void __launch_bounds__(256) k_out_sums(const uint32_t* __restrict__ pairs, const float* __restrict__ grow,
                                                  const float* __restrict__ lrow, int B, int P, int H,
                                                  const bf16* __restrict__ H2, const bf16* __restrict__ dZ2,
                                                  float* __restrict__ gW3, float* __restrict__ gb3,
                                                  float* __restrict__ gb2, float* __restrict__ loss)
{
    __shared__ float s_t[CS_ROWS][33];
    __shared__ int s_list[256];
    __shared__ int s_w[8];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if ((int)blockIdx.x >= B + H / 32) {
        float* red = &s_t[0][0];
        float s = 0.f;
        for (int r = tid; r < B; r += 256) s += lrow[r];
        red[tid] = s;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if (tid < w) red[tid] += red[tid + w];
            __syncthreads();
        }
        if (tid == 0) *loss = red[0];
        return;
    }
    if ((int)blockIdx.x >= B) {
        colsum_block(s_t, dZ2, H, B, ((int)blockIdx.x - B) * 32, gb2);
        return;
    }
    const int r = blockIdx.x;
    const uint32_t p = pairs[r];
    bool dup = false;
    for (int q = tid; q < r; q += 256) dup |= pairs[q] == p;
    if (__syncthreads_or(dup) || p >= (uint32_t)P) return;              // block-uniform
    float sb = 0.f;
    for (int c0 = 0; c0 < H; c0 += 256) {
        const int c = c0 + tid;
        float s = 0.f;
        for (int q0 = r; q0 < B; q0 += 256) {
            // this chunk's rows of the pair, in row order
            const bool hit = q0 + tid < B && pairs[q0 + tid] == p;
            const unsigned bal = __ballot_sync(0xffffffffu, hit);
            if (lane == 0) s_w[warp] = __popc(bal);
            __syncthreads();
            int before = 0, cnt = 0;
            for (int w = 0; w < 8; ++w) {
                before += w < warp ? s_w[w] : 0;
                cnt += s_w[w];
            }
            if (hit) s_list[before + __popc(bal & ((1u << lane) - 1u))] = q0 + tid;
            __syncthreads();
            for (int k = 0; k < cnt; ++k) {
                const int q = s_list[k];
                if (c < H) s += grow[q] * __bfloat162float(H2[(size_t)q * H + c]);
                if (c0 == 0 && tid == 0) sb += grow[q];
            }
            __syncthreads();
        }
        if (c < H) gW3[(size_t)p * H + c] = s;
    }
    if (tid == 0) gb3[p] = sb;
}

// dZ = bf16(dH * (Z > 0)), rows >= B -> 0, with the transposed copy
__global__ void __launch_bounds__(256) k_relu_grad(Product dH, const float* __restrict__ Z, int Mp, int N, int B,
                                                   bf16* __restrict__ dZ, bf16* __restrict__ dZT)
{
    __shared__ bf16 tile[32][33];
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
    bf16 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int r = r0 + threadIdx.y + 8 * k;
        const int64_t idx = (int64_t)r * N + c0 + threadIdx.x;
        v[k] = __float2bfloat16_rn((r < B && Z[idx] > 0.f) ? dH.at(idx) : 0.f);
    }
    store_tile(tile, v, r0, c0, dZ, N, dZT, Mp);
}

// Blocks below n * ceil(d / 32): dE[v][j] = sum over the rows r, in row order, of
// dX[r][inv_r(v) d + j], 32 columns j of one node a block, the rows side by side through
// shared memory as in colsum_block.  The rest: the column sums of dZ1 (gb1).
__global__ void __launch_bounds__(256) k_embed_grad(const uint8_t* __restrict__ inv, Product dX, int B, int n, int d,
                                                    int ndp, float* __restrict__ gE, const bf16* __restrict__ dZ1, int H,
                                                    float* __restrict__ gb1)
{
    __shared__ float s_t[CS_ROWS][33];
    const int jb = (d + 31) / 32;
    if ((int)blockIdx.x >= n * jb) {
        colsum_block(s_t, dZ1, H, B, ((int)blockIdx.x - n * jb) * 32, gb1);
        return;
    }
    const int v = blockIdx.x / jb, j = (blockIdx.x - v * jb) * 32 + (threadIdx.x & 31), x = threadIdx.x & 31,
              y = threadIdx.x >> 5;
    float s = 0.f;
    for (int r0 = 0; r0 < B; r0 += CS_ROWS) {
        const int rows = min(CS_ROWS, B - r0);
        __syncthreads();
        int at[CS_ROWS / 8];
#pragma unroll
        for (int k = 0; k < CS_ROWS / 8; ++k) {
            const int r = y + 8 * k;
            at[k] = r < rows ? inv[(size_t)(r0 + r) * 64 + v] : 0;
        }
#pragma unroll
        for (int k = 0; k < CS_ROWS / 8; ++k) {
            const int r = y + 8 * k;
            if (r < rows && j < d) s_t[r][x] = dX.at((int64_t)(r0 + r) * ndp + (int64_t)at[k] * d + j);
        }
        __syncthreads();
        if (y == 0) {
#pragma unroll 8
            for (int r = 0; r < rows; ++r) s += s_t[r][x];
        }
    }
    if (y == 0 && j < d) gE[(size_t)v * d + j] = s;
}

// Adam (Kingma & Ba): moments and the FP32 master weight.  The bias corrections of the next
// step live on the device (bn_adam) and every step advances them itself, so that a
// captured step replays with the corrections of its own place in the run.
struct AdamRates {
    float lr, b1, b2, eps, c1, c2;
};
__device__ __forceinline__ float adam_at(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                                         float* __restrict__ v, int64_t i, const AdamRates& R)
{
    // (the fused multiply-adds written out, so that inlining cannot change which is fused)
    const float gi = g[i];
    const float mi = __fmaf_rn(1.f - R.b1, gi, __fmul_rn(R.b1, m[i]));
    const float vi = __fmaf_rn(__fmul_rn(1.f - R.b2, gi), gi, __fmul_rn(R.b2, v[i]));
    m[i] = mi;
    v[i] = vi;
    const float x = w[i] - R.lr * (mi / R.c1) / (sqrtf(vi / R.c2) + R.eps);
    w[i] = x;
    return x;
}
struct AdamTensor {
    float *w, *g, *m, *v;
    bf16 *b, *bT;               // bf16 copy and its transpose, or null
    int rows, cols;             // tiled (bT): multiples of 32; else rows = 1, cols = elements
    int blocks;                 // of this tensor, after those of the tensors before it
};
struct AdamArgs {
    AdamTensor t[7];
    AdamRates R;                // c1 and c2 filled in by the kernel
    bn_adam* next;
};
// powers of the moments' rates: exact products rounded once to FP64 each step, far inside the
// FP32 that the corrections are rounded to
__host__ __device__ __forceinline__ void adam_set(bn_adam* a, double p1, double p2)
{
    a->p1 = p1;
    a->p2 = p2;
    a->c1 = 1.f - (float)p1;
    a->c2 = 1.f - (float)p2;
}

// Every parameter in one launch, with the bf16 copies the GEMMs read: 1,024 elements a block,
// W1 and W2 by 32 x 32 tiles for their transposes.  Bound by the weights' and moments'
// traffic, 24 bytes a parameter and step; seven launches for the step and four for the
// copies took 61 us of kernels at n = 60, H = 512, this one 19.
__global__ void __launch_bounds__(256) k_adam(AdamArgs A)
{
    __shared__ bf16 tile[32][33];
    AdamRates R = A.R;
    R.c1 = A.next->c1;
    R.c2 = A.next->c2;
    int blk = blockIdx.x, k = 0;
    while (blk >= A.t[k].blocks) blk -= A.t[k++].blocks;
    const AdamTensor& T = A.t[k];
    const int x = threadIdx.x, y = threadIdx.y;
    if (T.bT) {
        const int tc = T.cols / 32, r0 = blk / tc * 32, c0 = blk % tc * 32;
        bf16 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = __float2bfloat16_rn(adam_at(T.w, T.g, T.m, T.v, (int64_t)(r0 + y + 8 * q) * T.cols + c0 + x, R));
        store_tile(tile, v, r0, c0, T.b, T.cols, T.bT, T.rows);
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = (int64_t)blk * 1024 + q * 256 + y * 32 + x;
            if (i < T.cols) {
                const float w = adam_at(T.w, T.g, T.m, T.v, i, R);
                if (T.b) T.b[i] = __float2bfloat16_rn(w);
            }
        }
    }
    // the last block to come here -- every block has used the corrections -- sets the next step's
    __syncthreads();
    if (x == 0 && y == 0) {
        __threadfence();
        if (atomicAdd(&A.next->done, 1u) == gridDim.x - 1) {
            adam_set(A.next, A.next->p1 * (double)R.b1, A.next->p2 * (double)R.b2);
            A.next->done = 0;
        }
    }
}

// bf16 copy of a rows x cols FP32 matrix (row stride ld), zero-padded to prow x pcol,
// and optionally its transpose (pcol x prow)
__global__ void k_to_bf16(const float* __restrict__ src, int ld, int rows, int cols, int prow, int pcol,
                          bf16* __restrict__ dst, bf16* __restrict__ dstT)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)prow * pcol) return;
    const int r = (int)(idx / pcol), c = (int)(idx - (int64_t)r * pcol);
    const bf16 v = __float2bfloat16_rn((r < rows && c < cols) ? src[(size_t)r * ld + c] : 0.f);
    if (dst) dst[idx] = v;
    if (dstT) dstT[(size_t)c * prow + r] = v;
}

static inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace bn

using namespace bn;

// ---------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------
// A B^T of the network's buffers, left in partials where K is split
static int gemm_part(bn_mlp* m, const bf16* A, int lda, const bf16* B, int ldb, float* C, int ldc, int M, int N, int K,
                     cudaStream_t s, Product* out)
{
    const int split = gemm_split(M, N, K, m->ws_elems);
    const GemmArgs g{A, B, split > 1 ? m->ws : C, M, N, K, lda, ldb, split > 1 ? N : ldc, split, m->status};
    *out = Product{g.C, split, (int64_t)M * N};
    return gemm_launch(g, nullptr, s);
}

static int mlp_refresh_bf16(bn_mlp* m, cudaStream_t s)
{
    k_to_bf16<<<nblk((int64_t)m->n * m->d), 256, 0, s>>>(m->E, m->d, m->n, m->d, m->n, m->d, m->Eb, nullptr);
    BN_LAUNCH_CHECK("k_to_bf16");
    k_to_bf16<<<nblk((int64_t)m->H * m->ndp), 256, 0, s>>>(m->W1, m->ndp, m->H, m->nd, m->H, m->ndp, m->W1b,
                                                          m->W1T);
    BN_LAUNCH_CHECK("k_to_bf16");
    k_to_bf16<<<nblk((int64_t)m->H * m->H), 256, 0, s>>>(m->W2, m->H, m->H, m->H, m->H, m->H, m->W2b, m->W2T);
    BN_LAUNCH_CHECK("k_to_bf16");
    k_to_bf16<<<nblk((int64_t)m->Pp * m->H), 256, 0, s>>>(m->W3, m->H, m->P, m->H, m->Pp, m->H, m->W3b, nullptr);
    BN_LAUNCH_CHECK("k_to_bf16");
    return BN_OK;
}

static dim3 tiles_of(int rows, int cols) { return dim3((unsigned)(cols / 32), (unsigned)(rows / 32)); }
static const dim3 TILE(32, 8);

// forward of B <= cap orders; `train` also leaves the transposed operands and the inverse
// orders, and clears the output layer's gradients
static int mlp_forward(bn_mlp* m, const uint8_t* d_orders, int B, bool train, cudaStream_t s)
{
    const int Mp = (int)round_up(std::max(B, 1), 128), H = m->H;
    if (Mp > m->cap) return set_error(BN_EINVAL, "mlp: batch %d above capacity %d", B, m->cap);
    m->Mp = Mp;
    k_embed<<<tiles_of(Mp, m->ndp), TILE, 0, s>>>(d_orders, B, m->n, m->d, m->ndp, Mp, m->Eb, m->X, train ? m->XT : nullptr,
                                                 train ? m->inv : nullptr, m->status);
    BN_LAUNCH_CHECK("k_embed");
    int rc;
    Product z;
    if ((rc = gemm_part(m, m->X, m->ndp, m->W1b, m->ndp, m->Z1, H, Mp, H, m->ndp, s, &z))) return rc;
    k_bias_relu<<<tiles_of(Mp, H), TILE, 0, s>>>(z, m->Z1, m->b1, Mp, H, B, m->H1, train ? m->H1T : nullptr);
    BN_LAUNCH_CHECK("k_bias_relu");
    if ((rc = gemm_part(m, m->H1, H, m->W2b, H, m->Z2, H, Mp, H, H, s, &z))) return rc;
    k_bias_relu<<<tiles_of(Mp, H), TILE, 0, s>>>(z, m->Z2, m->b2, Mp, H, B, m->H2, nullptr);
    BN_LAUNCH_CHECK("k_bias_relu");
    if ((rc = gemm_part(m, m->H2, H, m->W3b, H, m->L, m->Pp, Mp, m->Pp, H, s, &z))) return rc;
    // gW3 and gb3 lie side by side, in multiples of 256 bytes
    const int64_t zeros = train ? ((m->gb3 + m->Pp) - m->gW3) / 4 : 0;
    k_bias<<<nblk((int64_t)Mp * m->Pp + zeros), 256, 0, s>>>(z, m->L, m->b3, Mp, m->Pp, (float4*)m->gW3, zeros);
    BN_LAUNCH_CHECK("k_bias");
    return BN_OK;
}

int bn::mlp_forward_dev(bn_mlp* m, const uint8_t* d_orders, int B, cudaStream_t s)
{
    return mlp_forward(m, d_orders, B, false, s);
}

// A layer's weight gradient gW = dZT actT^T and input gradient dA = dZ WT^T, in one launch
// unless the weight gradient's K is split (large batches)
static int grad_pair(bn_mlp* m, const bf16* dZT, const bf16* actT, float* gW, int ldg, int cols, const bf16* dZ,
                     const bf16* WT, float* dA, cudaStream_t s, Product* out)
{
    const int Mp = m->Mp, H = m->H;
    if (gemm_split(H, cols, Mp, m->ws_elems) > 1) {
        int rc = gemm_tc(dZT, Mp, actT, Mp, gW, ldg, H, cols, Mp, m->status, s, m->ws, m->ws_elems);
        if (rc) return rc;
        return gemm_part(m, dZ, H, WT, H, dA, cols, Mp, cols, H, s, out);
    }
    const GemmArgs a{dZT, actT, gW, H, cols, Mp, Mp, Mp, ldg, 1, m->status};
    const int split = gemm_split(Mp, cols, H, m->ws_elems);
    const GemmArgs b{dZ, WT, split > 1 ? m->ws : dA, Mp, cols, H, H, H, cols, split, m->status};
    *out = Product{b.C, split, (int64_t)Mp * cols};
    return gemm_launch(a, &b, s);
}

int bn::mlp_loss_grad_dev(bn_mlp* m, const uint8_t* d_orders, const uint32_t* d_pairs, const float* d_alpha, int B,
                          cudaStream_t s)
{
    int rc = mlp_forward(m, d_orders, B, true, s);
    if (rc) return rc;
    const int Mp = m->Mp, H = m->H;
    k_out_grad<<<Mp, 256, 0, s>>>(m->L, m->Pp, d_pairs, d_alpha, B, m->P, Mp, H, m->Z2, m->W3b, m->dZ2, m->dZ2T,
                                  m->grow, m->lrow, m->status);
    BN_LAUNCH_CHECK("k_out_grad");
    k_out_sums<<<(unsigned)(B + H / 32 + 1), 256, 0, s>>>(d_pairs, m->grow, m->lrow, B, m->P, H, m->H2, m->dZ2, m->gW3, m->gb3,
                                                        m->gb2, m->loss);
    BN_LAUNCH_CHECK("k_out_sums");
    Product dH, dX;
    // dW2 = dZ2^T H1 ; dH1 = dZ2 W2
    if ((rc = grad_pair(m, m->dZ2T, m->H1T, m->gW2, H, H, m->dZ2, m->W2T, m->dH1, s, &dH))) return rc;
    k_relu_grad<<<tiles_of(Mp, H), TILE, 0, s>>>(dH, m->Z1, Mp, H, B, m->dZ1, m->dZ1T);
    BN_LAUNCH_CHECK("k_relu_grad");
    // dW1 = dZ1^T X ; dX = dZ1 W1
    if ((rc = grad_pair(m, m->dZ1T, m->XT, m->gW1, m->ndp, m->ndp, m->dZ1, m->W1T, m->dX, s, &dX))) return rc;
    k_embed_grad<<<(unsigned)(m->n * ((m->d + 31) / 32) + H / 32), 256, 0, s>>>(m->inv, dX, B, m->n, m->d, m->ndp, m->gE,
                                                                              m->dZ1, H, m->gb1);
    BN_LAUNCH_CHECK("k_embed_grad");
    return BN_OK;
}

int bn::mlp_adam_dev(bn_mlp* m, cudaStream_t s)
{
    auto flat = [](float* w, float* g, float* mm, float* v, bf16* b, int64_t cnt) {
        return AdamTensor{w, g, mm, v, b, nullptr, 1, (int)cnt, (int)((cnt + 1023) / 1024)};
    };
    auto tiled = [](float* w, float* g, float* mm, float* v, bf16* b, bf16* bT, int rows, int cols) {
        return AdamTensor{w, g, mm, v, b, bT, rows, cols, rows / 32 * (cols / 32)};
    };
    AdamArgs A{{tiled(m->W1, m->gW1, m->mW1, m->vW1, m->W1b, m->W1T, m->H, m->ndp),
                tiled(m->W2, m->gW2, m->mW2, m->vW2, m->W2b, m->W2T, m->H, m->H),
                flat(m->W3, m->gW3, m->mW3, m->vW3, m->W3b, (int64_t)m->P * m->H),
                flat(m->E, m->gE, m->mE, m->vE, m->Eb, (int64_t)m->n * m->d),
                flat(m->b1, m->gb1, m->mb1, m->vb1, nullptr, m->H), flat(m->b2, m->gb2, m->mb2, m->vb2, nullptr, m->H),
                flat(m->b3, m->gb3, m->mb3, m->vb3, nullptr, m->P)},
               {m->lr, m->beta1, m->beta2, m->adam_eps, 0.f, 0.f},
               m->adam};
    int blocks = 0;
    for (const AdamTensor& t : A.t) blocks += t.blocks;
    k_adam<<<(unsigned)blocks, TILE, 0, s>>>(A);
    BN_LAUNCH_CHECK("k_adam");
    return BN_OK;
}

extern "C" int bn_mlp_create(int n, const bn_mlp_params* p, const float* E, const float* W1, const float* b1,
                             const float* W2, const float* b2, const float* W3, const float* b3, int mem, void* stream,
                             bn_mlp** out)
{
    set_error(BN_OK, "");
    if (!out || !p) return set_error(BN_EINVAL, "bn_mlp_create: NULL argument");
    *out = nullptr;
    if (n < 2 || n > MAXN || p->d < 1 || p->hidden < 128 || p->hidden % 128 || p->batch_cap < 1 ||
        !(p->lr >= 0.f))
        return set_error(BN_EINVAL, "bn_mlp_create: bad sizes (hidden must be a positive multiple of 128)");
    if (!E || !W1 || !b1 || !W2 || !b2 || !W3 || !b3) return set_error(BN_EINVAL, "bn_mlp_create: NULL weights");
    if (mem != BN_MEM_HOST && mem != BN_MEM_DEVICE) return set_error(BN_EINVAL, "bn_mlp_create: bad mem");
    cudaStream_t s = (cudaStream_t)stream;
    bn_mlp* m = new bn_mlp();
    m->n = n;
    m->d = p->d;
    m->H = p->hidden;
    m->P = n * (n - 1) / 2;
    m->Pp = (int)round_up(m->P, 128);
    m->nd = n * p->d;
    m->ndp = (int)round_up(m->nd, 128);
    m->cap = (int)round_up(p->batch_cap, 128);
    m->lr = p->lr;
    m->beta1 = p->beta1 > 0 ? p->beta1 : 0.9f;
    m->beta2 = p->beta2 > 0 ? p->beta2 : 0.999f;
    m->adam_eps = p->adam_eps > 0 ? p->adam_eps : 1e-8f;
    const int H = m->H, ndp = m->ndp, Pp = m->Pp, cap = m->cap;
    const size_t nE = (size_t)n * m->d, nW1 = (size_t)H * ndp, nW2 = (size_t)H * H, nW3 = (size_t)Pp * H;
    // one FP32 block: master (E W1 b1 W2 b2 W3 b3) x {w, grad, m, v}, activations
    size_t off = 0;
    std::vector<std::pair<float**, size_t>> f32 = {
        {&m->E, nE}, {&m->W1, nW1}, {&m->b1, (size_t)H}, {&m->W2, nW2}, {&m->b2, (size_t)H}, {&m->W3, nW3},
        {&m->b3, (size_t)Pp}, {&m->gE, nE}, {&m->gW1, nW1}, {&m->gb1, (size_t)H}, {&m->gW2, nW2},
        {&m->gb2, (size_t)H}, {&m->gW3, nW3}, {&m->gb3, (size_t)Pp}, {&m->mE, nE}, {&m->mW1, nW1},
        {&m->mb1, (size_t)H}, {&m->mW2, nW2}, {&m->mb2, (size_t)H}, {&m->mW3, nW3}, {&m->mb3, (size_t)Pp},
        {&m->vE, nE}, {&m->vW1, nW1}, {&m->vb1, (size_t)H}, {&m->vW2, nW2}, {&m->vb2, (size_t)H},
        {&m->vW3, nW3}, {&m->vb3, (size_t)Pp}, {&m->Z1, (size_t)cap * H}, {&m->Z2, (size_t)cap * H},
        {&m->L, (size_t)cap * Pp}, {&m->dH1, (size_t)cap * H}, {&m->dX, (size_t)cap * ndp}, {&m->loss, 4},
        {&m->grow, (size_t)cap}, {&m->lrow, (size_t)cap},
        {&m->ws, (size_t)8 * cap * std::max(std::max(Pp, ndp), H)}};
    std::vector<std::pair<bf16**, size_t>> b16 = {
        {&m->Eb, nE}, {&m->W1b, nW1}, {&m->W1T, nW1}, {&m->W2b, nW2}, {&m->W2T, nW2}, {&m->W3b, nW3},
        {&m->X, (size_t)cap * ndp}, {&m->XT, (size_t)cap * ndp}, {&m->H1, (size_t)cap * H},
        {&m->H1T, (size_t)cap * H}, {&m->H2, (size_t)cap * H}, {&m->dZ2, (size_t)cap * H},
        {&m->dZ2T, (size_t)cap * H}, {&m->dZ1, (size_t)cap * H}, {&m->dZ1T, (size_t)cap * H}};
    std::vector<size_t> offs;
    for (auto& e : f32) { offs.push_back(off); off = (size_t)round_up((int64_t)(off + 4 * e.second), 256); }
    for (auto& e : b16) { offs.push_back(off); off = (size_t)round_up((int64_t)(off + 2 * e.second), 256); }
    const size_t o_status = off;
    off += 256;
    const size_t o_stage = off;                      // staging for host inputs: orders, pairs, alpha
    off += (size_t)round_up((int64_t)cap * n, 256) + (size_t)round_up((int64_t)cap * 4, 256) * 2;
    const size_t o_inv = off;                        // inverse orders of a training batch
    off += (size_t)round_up((int64_t)cap * 64, 256);
    cudaError_t e = obj_alloc(&m->block, off);
    if (e != cudaSuccess) {
        cudaGetLastError();
        delete m;
        return set_error(BN_ENOMEM, "bn_mlp_create: %zu bytes: %s", off, cudaGetErrorString(e));
    }
    uint8_t* base = (uint8_t*)m->block;
    size_t k = 0;
    for (auto& e2 : f32) *e2.first = (float*)(base + offs[k++]);
    for (auto& e2 : b16) *e2.first = (bf16*)(base + offs[k++]);
    m->status = (uint32_t*)(base + o_status);
    m->adam = (bn_adam*)(base + o_status + 64);
    bn_adam first = {};
    adam_set(&first, (double)m->beta1, (double)m->beta2);
    m->stage_orders = base + o_stage;
    m->stage_pairs = (uint32_t*)(base + o_stage + (size_t)round_up((int64_t)cap * n, 256));
    m->stage_alpha = (float*)((uint8_t*)m->stage_pairs + (size_t)round_up((int64_t)cap * 4, 256));
    m->inv = base + o_inv;
    m->bytes = off;
    m->ws_elems = (size_t)8 * cap * std::max(std::max(Pp, ndp), H);
    auto fail = [&](int rc) { bn_mlp_free(m); return rc; };
    if (cudaMemsetAsync(m->block, 0, off, s) != cudaSuccess) return fail(cuda_fail(cudaGetLastError(), "memset", __FILE__, __LINE__));
    const cudaMemcpyKind kind = mem == BN_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    // weights come row-major and unpadded: E n x d, W1 H x (n d), W2 H x H, W3 P x H
    if (cudaMemcpyAsync(m->adam, &first, sizeof(first), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(m->E, E, 4 * nE, kind, s) != cudaSuccess ||
        cudaMemcpy2DAsync(m->W1, 4 * (size_t)ndp, W1, 4 * (size_t)m->nd, 4 * (size_t)m->nd, H, kind, s) != cudaSuccess ||
        cudaMemcpyAsync(m->b1, b1, 4 * (size_t)H, kind, s) != cudaSuccess ||
        cudaMemcpyAsync(m->W2, W2, 4 * nW2, kind, s) != cudaSuccess ||
        cudaMemcpyAsync(m->b2, b2, 4 * (size_t)H, kind, s) != cudaSuccess ||
        cudaMemcpyAsync(m->W3, W3, 4 * (size_t)m->P * H, kind, s) != cudaSuccess ||
        cudaMemcpyAsync(m->b3, b3, 4 * (size_t)m->P, kind, s) != cudaSuccess)
        return fail(cuda_fail(cudaGetLastError(), "bn_mlp_create weights", __FILE__, __LINE__));
    int rc = mlp_refresh_bf16(m, s);
    if (rc) return fail(rc);
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail(cuda_fail(cudaGetLastError(), "sync", __FILE__, __LINE__));
    *out = m;
    return BN_OK;
}

static int stage_in(void* dst, const void* src, size_t bytes, int mem, cudaStream_t s, const void** out)
{
    if (mem == BN_MEM_DEVICE) { *out = src; return BN_OK; }
    BN_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, s));
    *out = dst;
    return BN_OK;
}

static int check_status(bn_mlp* m, cudaStream_t s, const char* who)
{
    uint32_t st = 0;
    BN_CUDA(cudaMemcpyAsync(&st, m->status, 4, cudaMemcpyDeviceToHost, s));
    BN_CUDA(cudaStreamSynchronize(s));
    if (st & STATUS_TIMEOUT) return set_error(BN_ETIMEOUT, "%s: a bounded device wait expired", who);
    if (st & STATUS_BADINPUT) {
        BN_CUDA(cudaMemsetAsync(m->status, 0, 4, s));       // the next call's inputs are its own
        BN_CUDA(cudaStreamSynchronize(s));
        return set_error(BN_EINVAL, "%s: an order names a node or a row a swap pair that does not exist", who);
    }
    return BN_OK;
}

extern "C" int bn_mlp_forward(bn_mlp* m, const uint8_t* orders, int B, float* logits, int mem, void* stream)
{
    set_error(BN_OK, "");
    if (!m || !orders || !logits || B < 1) return set_error(BN_EINVAL, "bn_mlp_forward: bad arguments");
    if (B > m->cap) return set_error(BN_EINVAL, "bn_mlp_forward: B=%d above batch capacity %d", B, m->cap);
    cudaStream_t s = (cudaStream_t)stream;
    const void* d_o = nullptr;
    int rc = stage_in(m->stage_orders, orders, (size_t)B * m->n, mem, s, &d_o);
    if (rc) return rc;
    if ((rc = mlp_forward_dev(m, (const uint8_t*)d_o, B, s))) return rc;
    BN_CUDA(cudaMemcpy2DAsync(logits, 4 * (size_t)m->P, m->L, 4 * (size_t)m->Pp, 4 * (size_t)m->P, B,
                              mem == BN_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    return check_status(m, s, "bn_mlp_forward");
}

extern "C" int bn_mlp_loss_grad(bn_mlp* m, const uint8_t* orders, const uint32_t* pairs, const float* alpha, int B,
                                float* loss, int mem, void* stream)
{
    set_error(BN_OK, "");
    if (!m || !orders || !pairs || !alpha || B < 1) return set_error(BN_EINVAL, "bn_mlp_loss_grad: bad arguments");
    if (B > m->cap) return set_error(BN_EINVAL, "bn_mlp_loss_grad: B=%d above batch capacity %d", B, m->cap);
    cudaStream_t s = (cudaStream_t)stream;
    const void *d_o = nullptr, *d_p = nullptr, *d_a = nullptr;
    int rc;
    if ((rc = stage_in(m->stage_orders, orders, (size_t)B * m->n, mem, s, &d_o)) ||
        (rc = stage_in(m->stage_pairs, pairs, 4 * (size_t)B, mem, s, &d_p)) ||
        (rc = stage_in(m->stage_alpha, alpha, 4 * (size_t)B, mem, s, &d_a)))
        return rc;
    if ((rc = mlp_loss_grad_dev(m, (const uint8_t*)d_o, (const uint32_t*)d_p, (const float*)d_a, B, s))) return rc;
    if (loss)
        BN_CUDA(cudaMemcpyAsync(loss, m->loss, 4, mem == BN_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    return check_status(m, s, "bn_mlp_loss_grad");
}

extern "C" int bn_mlp_adam_step(bn_mlp* m, void* stream)
{
    set_error(BN_OK, "");
    if (!m) return set_error(BN_EINVAL, "bn_mlp_adam_step: NULL");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = mlp_adam_dev(m, s);
    if (rc) return rc;
    BN_CUDA(cudaStreamSynchronize(s));
    return BN_OK;
}

extern "C" int bn_mlp_read(const bn_mlp* m, int what, float* out, int mem, void* stream)
{
    set_error(BN_OK, "");
    if (!m || !out) return set_error(BN_EINVAL, "bn_mlp_read: NULL");
    cudaStream_t s = (cudaStream_t)stream;
    const bool grad = what >= BN_MLP_GRAD_E;
    const int w = grad ? what - BN_MLP_GRAD_E : what;
    const float* src = nullptr;
    size_t rows = 1, cols = 0, spitch = 0;
    switch (w) {
        case BN_MLP_E: src = grad ? m->gE : m->E; rows = m->n; cols = m->d; spitch = m->d; break;
        case BN_MLP_W1: src = grad ? m->gW1 : m->W1; rows = m->H; cols = m->nd; spitch = m->ndp; break;
        case BN_MLP_B1: src = grad ? m->gb1 : m->b1; cols = m->H; spitch = cols; break;
        case BN_MLP_W2: src = grad ? m->gW2 : m->W2; rows = m->H; cols = m->H; spitch = m->H; break;
        case BN_MLP_B2: src = grad ? m->gb2 : m->b2; cols = m->H; spitch = cols; break;
        case BN_MLP_W3: src = grad ? m->gW3 : m->W3; rows = m->P; cols = m->H; spitch = m->H; break;
        case BN_MLP_B3: src = grad ? m->gb3 : m->b3; cols = m->P; spitch = cols; break;
        default: return set_error(BN_EINVAL, "bn_mlp_read: unknown tensor %d", what);
    }
    BN_CUDA(cudaMemcpy2DAsync(out, 4 * cols, src, 4 * spitch, 4 * cols, rows,
                              mem == BN_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    BN_CUDA(cudaStreamSynchronize(s));
    return BN_OK;
}

extern "C" void bn_mlp_free(bn_mlp* m)
{
    if (!m) return;
    obj_free({m->block});
    delete m;
}

extern "C" int bn_gemm_bf16(const uint16_t* A, const uint16_t* B, float* C, int M, int N, int K, void* stream)
{
    set_error(BN_OK, "");
    if (!A || !B || !C) return set_error(BN_EINVAL, "bn_gemm_bf16: NULL");
    cudaStream_t s = (cudaStream_t)stream;
    uint32_t* st = nullptr;
    BN_CUDA(dev_alloc((void**)&st, 4, s));
    BN_CUDA(cudaMemsetAsync(st, 0, 4, s));
    int rc = gemm_tc((const bf16*)A, K, (const bf16*)B, K, C, N, M, N, K, st, s, nullptr, 0);
    uint32_t h = 0;
    if (!rc) {
        BN_CUDA(cudaMemcpyAsync(&h, st, 4, cudaMemcpyDeviceToHost, s));
    }
    dev_free(st, s);
    BN_CUDA(cudaStreamSynchronize(s));
    if (rc) return rc;
    if (h & STATUS_TIMEOUT) return set_error(BN_ETIMEOUT, "bn_gemm_bf16: a bounded device wait expired");
    return BN_OK;
}
