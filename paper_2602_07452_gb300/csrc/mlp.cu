// Learned implicit guess: the MLP 14 -> 128 -> 128 -> 128 -> 9 (ReLU) on the
// fifth-generation tensor cores (tcgen05, BF16 operands, FP32 accumulators
// in tensor memory).
//
//   k_gemm_bf16  generic C (+)= A B^T, one 128-row block per CTA, K staged
//                through shared memory in 64-wide slices.
//   k_mlp_fwd    fused persistent forward: the four weight matrices stay in
//                shared memory, each 128-sample tile runs layer after layer
//                through one TMEM accumulator, the epilogue (bias, ReLU,
//                bf16 rounding) writes the next layer's A operand back to
//                shared memory.
// Parameter layout (FP32 master copy, as the oracle): W1 [128][14] b1 W2
// [128][128] b2 W3 [128][128] b3 W4 [9][128] b4.  Every wait on an mbarrier
// is bounded; a timeout sets an error word and the kernel frees its tensor
// memory and returns.
#include <math.h>

#include <vector>

#include "fpic_internal.h"
#include "mlp_dev.cuh"
#include "tc.cuh"

namespace fpic {

constexpr long long MLP_NPARAM = 128LL * 14 + 128 + 2 * (128LL * 128 + 128) + 9LL * 128 + 9;

// ---------------------------------------------------------------------------
// Generic GEMM
// ---------------------------------------------------------------------------
constexpr int GK = 64;   // K slice staged per round

__global__ void __launch_bounds__(128) k_gemm_bf16(const uint16_t* __restrict__ A, int lda,
                                                   const uint16_t* __restrict__ B, int ldb, float* __restrict__ C,
                                                   int ldc, int M, int N, int K, int accumulate, int* err)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sA = smem;                        // 128 x 64 bf16 = 16 KB
    uint8_t* sB = smem + 16384;                // N x 64 bf16 <= 32 KB
    uint64_t* mbar = (uint64_t*)(smem + 16384 + 32768);
    uint32_t* tslot = (uint32_t*)(mbar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * 128;
    const uint32_t ncols = N <= 32 ? 32u : (N <= 64 ? 64u : (N <= 128 ? 128u : 256u));
    if (warp == 0) tc::tmem_alloc(tslot, ncols);
    if (tid == 0) tc::mbar_init(mbar, 1);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    uint32_t phase = 0;
    int ok = 1;
    for (int k0 = 0; k0 < K && ok; k0 += GK) {
        const int kc = min(GK, K - k0);
        const int nv = kc / 8;
        for (int v = tid; v < 128 * nv; v += 128) {
            const int r = v / nv, g = v % nv;
            uint4 val = make_uint4(0, 0, 0, 0);
            if (m0 + r < M) val = *(const uint4*)(A + (size_t)(m0 + r) * lda + k0 + g * 8);
            *(uint4*)(sA + tc::kmajor_off(r, g * 8, 128)) = val;
        }
        for (int v = tid; v < N * nv; v += 128) {
            const int r = v / nv, g = v % nv;
            *(uint4*)(sB + tc::kmajor_off(r, g * 8, N)) = *(const uint4*)(B + (size_t)r * ldb + k0 + g * 8);
        }
        tc::fence_async_smem();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after();
            const uint32_t idesc = tc::idesc_bf16(128, N);
            const uint32_t a0 = tc::smem_addr(sA), b0 = tc::smem_addr(sB);
            for (int kk = 0; kk < kc / 16; ++kk) {
                const uint64_t ad = tc::smem_desc(a0 + kk * 2 * (128 * 16), 128 * 16, 128);
                const uint64_t bd = tc::smem_desc(b0 + kk * 2 * (N * 16), N * 16, 128);
                tc::mma_bf16(tbase, ad, bd, idesc, (k0 > 0 || kk > 0) ? 1u : 0u);
            }
            tc::mma_commit(mbar);
        }
        const int done = tc::mbar_wait(mbar, phase) ? 1 : 0;
        phase ^= 1u;
        ok = __syncthreads_and(done);
    }
    tc::fence_after();
    if (ok) {
        const int row = m0 + warp * 32 + lane;
        for (int c0 = 0; c0 < N; c0 += 32) {
            float v[32];
            const uint32_t ta = tbase + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
            int w = min(32, N - c0);
            if (w == 32) tc::tmem_ld32(ta, v);
            else tc::tmem_ld16(ta, v);
            if (row < M) {
                float* cr = C + (size_t)row * ldc + c0;
                for (int i = 0; i < w; ++i) cr[i] = accumulate ? cr[i] + v[i] : v[i];
            }
        }
    } else if (tid == 0) {
        atomicExch(err, 1);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, ncols);
}

// ---------------------------------------------------------------------------
// Parameter packing: FP32 master -> padded bf16 matrices (and transposes)
// ---------------------------------------------------------------------------

__global__ void k_mlp_pack(const float* __restrict__ P, MlpDev d)
{
    const long long oW1 = 0, ob1 = oW1 + 128 * 14, oW2 = ob1 + 128, ob2 = oW2 + 128 * 128, oW3 = ob2 + 128,
                    ob3 = oW3 + 128 * 128, oW4 = ob3 + 128, ob4 = oW4 + 9 * 128;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < 128 * 128; t += gridDim.x * blockDim.x) {
        const int o = t / 128, i = t % 128;
        const uint16_t w2 = tc::f2bf(P[oW2 + t]), w3 = tc::f2bf(P[oW3 + t]);
        d.W2[t] = w2;
        d.W3[t] = w3;
        d.W2t[i * 128 + o] = w2;
        d.W3t[i * 128 + o] = w3;
        if (i < 16) d.W1[o * 16 + i] = i < 14 ? tc::f2bf(P[oW1 + o * 14 + i]) : (uint16_t)0;
        if (o < 16) {
            const uint16_t w4 = o < 9 ? tc::f2bf(P[oW4 + o * 128 + i]) : (uint16_t)0;
            d.W4[o * 128 + i] = w4;
            d.W4t[i * 16 + o] = w4;
        }
        if (t < 128) {
            d.b1[t] = P[ob1 + t];
            d.b2[t] = P[ob2 + t];
            d.b3[t] = P[ob3 + t];
        }
        if (t < 16) d.b4[t] = t < 9 ? P[ob4 + t] : 0.0f;
    }
}

// ---------------------------------------------------------------------------
// Fused forward (building blocks in mlp_dev.cuh)
// ---------------------------------------------------------------------------
struct FwdK {
    MlpDev w;
    const float* X;      // B x 16 FP32 features (standardised, padded with zeros)
    float* Y;            // B x 16 FP32 outputs (9 used)
    long long B;         // rows (bound of the launch)
    const long long* count;   // nullable: rows = min(B, *count), read on the device
    int* err;
};

// Fused persistent forward, 256 threads: thread t owns row t % 128 of each
// 128-row tile and half t / 128 of its 16 inputs and of the hidden columns.
// The next tile's inputs are loaded into registers while the current tile
// runs through the four layers.
__global__ void __launch_bounds__(FW_THREADS) k_mlp_fwd(FwdK k)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    long long B = k.B;
    if (k.count) {
        const long long c = *k.count;
        B = c < 0 ? 0 : (c < B ? c : B);
    }
    const long long ntiles = (B + 127) / 128;
    if ((long long)blockIdx.x >= ntiles) return;     // whole block, before any allocation
    float* sb = (float*)(smem + FW_B);
    const int tid = threadIdx.x, warp = tid >> 5, r = tid & 127, half = tid >> 7;
    uint64_t* mbar;
    const uint32_t tbase = mlp_cta_setup(k.w, smem, &mbar);
    uint32_t phase = 0;
    int ok = 1;
    // this thread's 8 inputs of the first tile
    float4 xa = make_float4(0.f, 0.f, 0.f, 0.f), xb = xa;
    {
        const long long row = (long long)blockIdx.x * 128 + r;
        if (row < B) {
            xa = *(const float4*)(k.X + row * 16 + 8 * half);
            xb = *(const float4*)(k.X + row * 16 + 8 * half + 4);
        }
    }
    for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const long long row = tile * 128 + r;
        *(uint4*)(smem + FW_X + tc::kmajor_off(r, 8 * half, 128)) =
            make_uint4(tc::pack_bf2(xa.x, xa.y), tc::pack_bf2(xa.z, xa.w), tc::pack_bf2(xb.x, xb.y),
                       tc::pack_bf2(xb.z, xb.w));
        {
            const long long nrow = (tile + gridDim.x) * 128 + r;
            xa = make_float4(0.f, 0.f, 0.f, 0.f);
            xb = xa;
            if (nrow < B) {
                xa = *(const float4*)(k.X + nrow * 16 + 8 * half);
                xb = *(const float4*)(k.X + nrow * 16 + 8 * half + 4);
            }
        }
        ok = mlp_tile_layers(tbase, smem, mbar, phase);
        if (!ok) break;
        if (half == 0) {
            float v[16];
            tc::tmem_ld16(tbase + ((uint32_t)(warp * 32) << 16), v);
            if (row < B) {
                float4* y = (float4*)(k.Y + row * 16);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    y[q] = make_float4(v[4 * q] + sb[384 + 4 * q], v[4 * q + 1] + sb[385 + 4 * q],
                                       v[4 * q + 2] + sb[386 + 4 * q], v[4 * q + 3] + sb[387 + 4 * q]);
            }
        }
    }
    mlp_cta_teardown(tbase, ok, k.err);
}


// ---------------------------------------------------------------------------
// Training: three launches per step
//   k_train_tile   forward, loss gradient and the backward chain dZ of one
//                  128-row tile, everything between the layers in shared and
//                  tensor memory; writes the activations and dZ (bf16) that
//                  the weight gradients contract, and per-CTA bias gradients;
//   k_train_dw     the four weight gradients dW = dZ^T H, TRAIN_SPLITS
//                  batch slices each;
//   k_train_apply  slices and bias parts summed in a fixed order into the
//                  flat gradient and, for a step, Adam and the handle's bf16
//                  weights.
// What bounds it: at a minibatch of 8192 the work is 1.8 GFLOP and a few MB,
// so launches and per-tile latency.  One GEMM launch per slice (64 of them,
// each a single CTA of 54-98 us) plus separate transposes, masks and column
// sums took 3.27 ms per step of 8192 samples; these three launches 55 us.
// The MMAs keep their shapes and their K order, so the gradients are the
// same bits as those of separate GEMMs.
// ---------------------------------------------------------------------------
struct LossW {
    float m[16];     // regression weights per output (entry 6: the logit, unused)
};

constexpr int TRAIN_SPLITS = 16;                       // batch slices of each weight gradient
constexpr int TRAIN_NDB = 3 * 128 + 16;                // bias gradients b1 b2 b3 b4 (b4 padded)
constexpr int TRAIN_MAX_CTAS = 256;                    // CTAs of k_train_tile at most (their bias parts are kept apart)

// shared memory of k_train_tile: the forward's map, then the transposed
// weights, dY (bf16 operand), the column-sum staging of both halves
constexpr int TR_W4T = ((FW_SMEM + 127) / 128) * 128, TR_W3T = TR_W4T + 128 * 16 * 2, TR_W2T = TR_W3T + 128 * 128 * 2,
              TR_DY = TR_W2T + 128 * 128 * 2, TR_STG = TR_DY + 128 * 16 * 2, TR_SMEM = TR_STG + 2 * 128 * 33 * 4;

struct TrainK {
    MlpDev w;
    const float *X, *T, *S;
    LossW lw;
    long long B;         // a multiple of 128
    float invB;
    float* rowloss;
    uint16_t *H, *dZ;    // [3][B][128]
    uint16_t *Xb, *dY;   // [B][16]
    double* db;          // [gridDim.x][TRAIN_NDB]
    int* err;
};

// FP32 accumulation with its rounding errors carried along (Knuth's two-sum):
// s + e is the sum to about 2^-46, in place of FP64 additions.
__device__ __forceinline__ void add_carry(float& s, float& e, float x)
{
    const float t = __fadd_rn(s, x);
    const float v = __fsub_rn(t, s);
    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, v)), __fsub_rn(x, v)));
    s = t;
}

// Backward epilogue of a hidden layer: d = dH where the activation was
// positive, else 0 (FP32); its bf16 rounding to the next MMA's operand tile
// and to global memory, and the column sums of d (the bias gradient) of
// this thread's (column, quarter of the rows) added to cs[2].
__device__ __forceinline__ void train_bwd_epilogue(uint32_t tbase, const uint32_t* mask, uint8_t* sH,
                                                   uint16_t* dZrow, float* stg, double* cs)
{
    const int r = threadIdx.x & 127, warp = (threadIdx.x >> 5) & 3, half = threadIdx.x >> 7;
    float* st = stg + half * 128 * 33;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c0 = 64 * half + 32 * h;
        float v[32];
        tc::tmem_ld32(tbase + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            v[c] = (mask[h] >> c) & 1u ? v[c] : 0.f;
            st[r * 33 + c] = v[c];
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint4 u = make_uint4(tc::pack_bf2(v[8 * g], v[8 * g + 1]), tc::pack_bf2(v[8 * g + 2], v[8 * g + 3]),
                                       tc::pack_bf2(v[8 * g + 4], v[8 * g + 5]),
                                       tc::pack_bf2(v[8 * g + 6], v[8 * g + 7]));
            *(uint4*)(sH + tc::kmajor_off(r, c0 + g * 8, 128)) = u;
            *(uint4*)(dZrow + c0 + g * 8) = u;
        }
        __syncthreads();
        float s = 0.f, e = 0.f;
        const float* col = st + (r >> 5) * 32 * 33 + (r & 31);
#pragma unroll 8
        for (int q = 0; q < 32; ++q) add_carry(s, e, col[q * 33]);
        cs[h] += (double)s + (double)e;
        __syncthreads();
    }
}

// 256 threads, thread t owns row t % 128 and half t / 128 of the hidden
// columns, as in k_mlp_fwd; one CTA per SM (216 KB of shared memory), each
// over tiles blockIdx.x, + gridDim.x, ...  The activations' signs stay in six
// registers.  Latency-bound: seven dependent MMA + epilogue rounds per tile.
__global__ void __launch_bounds__(FW_THREADS) k_train_tile(const __grid_constant__ TrainK k)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const float* sb = (const float*)(smem + FW_B);
    float* stg = (float*)(smem + TR_STG);
    const int tid = threadIdx.x, warp = tid >> 5, r = tid & 127, half = tid >> 7;
    load_tile_kmajor(smem + TR_W4T, k.w.W4t, 128, 16);
    load_tile_kmajor(smem + TR_W3T, k.w.W3t, 128, 128);
    load_tile_kmajor(smem + TR_W2T, k.w.W2t, 128, 128);
    uint64_t* mbar;
    const uint32_t tbase = mlp_cta_setup(k.w, smem, &mbar);
    uint32_t phase = 0;
    int ok = 1;
    double cs[6] = {0, 0, 0, 0, 0, 0}, cy = 0.0;
    const size_t BH = (size_t)k.B * 128;
    for (long long row0 = blockIdx.x * 128LL; row0 < k.B; row0 += gridDim.x * 128LL) {
        const size_t row = (size_t)row0 + r;
        {
            const float4 xa = *(const float4*)(k.X + row * 16 + 8 * half);
            const float4 xb = *(const float4*)(k.X + row * 16 + 8 * half + 4);
            const uint4 u = make_uint4(tc::pack_bf2(xa.x, xa.y), tc::pack_bf2(xa.z, xa.w), tc::pack_bf2(xb.x, xb.y),
                                       tc::pack_bf2(xb.z, xb.w));
            *(uint4*)(smem + FW_X + tc::kmajor_off(r, 8 * half, 128)) = u;
            *(uint4*)(k.Xb + row * 16 + 8 * half) = u;
        }
        uint32_t mask[6];
        ok = mlp_tile_layers<true>(tbase, smem, mbar, phase, k.H + row * 128, BH, mask);
        if (!ok) break;
        // d loss / d y (scaled by 1/B): 2 m_k (y_k - t_k) and, for the logit,
        // sigmoid(y_6) - s
        if (half == 0) {
            float v[16], d[16];
            tc::tmem_ld16(tbase + ((uint32_t)(warp * 32) << 16), v);
            float L = 0.f;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                d[c] = 0.f;
                const float y = v[c] + sb[384 + c];
                if (c == 6) {
                    const float sv = k.S[row];
                    const float sp = y > 0.f ? y + log1pf(expf(-y)) : log1pf(expf(y));
                    L += sp - sv * y;
                    d[c] = 1.f / (1.f + expf(-y)) - sv;
                } else if (c < 9) {
                    const float e = y - k.T[row * 16 + c];
                    L += k.lw.m[c] * e * e;
                    d[c] = 2.f * k.lw.m[c] * e;
                }
                d[c] *= k.invB;
                stg[r * 17 + c] = d[c];
            }
            k.rowloss[row] = L;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const uint4 u = make_uint4(tc::pack_bf2(d[8 * g], d[8 * g + 1]),
                                           tc::pack_bf2(d[8 * g + 2], d[8 * g + 3]),
                                           tc::pack_bf2(d[8 * g + 4], d[8 * g + 5]),
                                           tc::pack_bf2(d[8 * g + 6], d[8 * g + 7]));
                *(uint4*)(smem + TR_DY + tc::kmajor_off(r, 8 * g, 128)) = u;
                *(uint4*)(k.dY + row * 16 + 8 * g) = u;
            }
        }
        ok = layer_mma(tbase, smem + TR_DY, smem + TR_W4T, 128, 16, mbar, phase);
        if (!ok) break;
        {   // column sums of dY: column tid % 16, rows 8 (tid / 16) .. + 7
            float s = 0.f, e = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) add_carry(s, e, stg[((tid >> 4) * 8 + q) * 17 + (tid & 15)]);
            cy += (double)s + (double)e;
            __syncthreads();
        }
        train_bwd_epilogue(tbase, mask + 4, smem + FW_H, k.dZ + 2 * BH + row * 128, stg, cs + 4);
        ok = layer_mma(tbase, smem + FW_H, smem + TR_W3T, 128, 128, mbar, phase);
        if (!ok) break;
        train_bwd_epilogue(tbase, mask + 2, smem + FW_H, k.dZ + BH + row * 128, stg, cs + 2);
        ok = layer_mma(tbase, smem + FW_H, smem + TR_W2T, 128, 128, mbar, phase);
        if (!ok) break;
        train_bwd_epilogue(tbase, mask, smem + FW_H, k.dZ + row * 128, stg, cs);
    }
    // this CTA's bias gradients: the quarters (hidden layers) and the row
    // groups (output layer) in a fixed order
    __syncthreads();
    double* part = (double*)stg;     // [6][256], then [256]
#pragma unroll
    for (int q = 0; q < 6; ++q) part[q * 256 + tid] = cs[q];
    part[6 * 256 + tid] = cy;
    __syncthreads();
    for (int o = tid; o < TRAIN_NDB; o += FW_THREADS) {
        double a = 0.0;
        if (o < 384) {
            const int l = o >> 7, c = o & 127, hf = c >> 6, h = (c >> 5) & 1;
            for (int q = 0; q < 4; ++q) a += part[(2 * l + h) * 256 + hf * 128 + q * 32 + (c & 31)];
        } else {
            for (int q = 0; q < 16; ++q) a += part[6 * 256 + q * 16 + (o - 384)];
        }
        k.db[(size_t)blockIdx.x * TRAIN_NDB + o] = a;
    }
    mlp_cta_teardown(tbase, ok, k.err);
}

// Weight gradients: CTA (slice s, gradient g) contracts rows [s ks, (s+1) ks)
// of the batch, ks = B / TRAIN_SPLITS:
//   g 0: dW4^T [128][16] = H3^T dY, 1: dW3 = dZ3^T H2, 2: dW2 = dZ2^T H1,
//   3: dW1 [128][16] = dZ1^T X.
// The operands are K-major in the batch while memory is row-major, so each
// chunk of up to 128 rows goes through shared memory as it is and its 8 x 8
// blocks are transposed by ldmatrix.trans, one 128-byte core matrix each;
// the next chunk's loads are in flight meanwhile, and the MMAs of a chunk
// run while the next one is transposed into the other operand buffer.  64
// CTAs of 512 rows each at a minibatch of 8192: latency-bound, like the tiles.
constexpr int DW_KC = 128, DW_LD = 272;     // chunk rows; padded row of the staging (bytes): conflict-free ldmatrix
constexpr int DW_RAW = DW_KC * DW_LD, DW_OP = DW_KC * 128 * 2;
constexpr int DW_BAR = 2 * DW_RAW + 4 * DW_OP, DW_SMEM = DW_BAR + 64;

struct DwK {
    const uint16_t *H, *dZ, *Xb, *dY;
    long long B;
    float* part;      // dW4t, dW3, dW2, dW1 slices: TRAIN_SPLITS x 128 x (16, 128, 128, 16)
    int* err;
};

__host__ __device__ constexpr size_t dw_part_off(int g)
{
    return (size_t)TRAIN_SPLITS * 128 * (g == 0 ? 0 : g == 1 ? 16 : g == 2 ? 144 : 272);
}

// The 8 x 8 blocks of a staged chunk (rows k, R columns) into the K-major
// operand layout of an R-row tile.
__device__ __forceinline__ void dw_transpose(const uint8_t* raw, uint8_t* op, int R, int kc)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nr = R >> 3, nb = (kc >> 3) * nr;          // a multiple of 4
    for (int b0 = 4 * warp; b0 < nb; b0 += 4 * (FW_THREADS / 32)) {
        const int bl = b0 + (lane >> 3), ko = bl / nr, ro = bl - ko * nr;
        const uint32_t src = tc::smem_addr(raw + (ko * 8 + (lane & 7)) * DW_LD + ro * 16);
        uint32_t m[4];
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                     : "=r"(m[0]), "=r"(m[1]), "=r"(m[2]), "=r"(m[3])
                     : "r"(src));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int bj = b0 + j, kj = bj / nr, rj = bj - kj * nr;
            *(uint32_t*)(op + kj * R * 16 + rj * 128 + lane * 4) = m[j];
        }
    }
}

template <int N>
__device__ __forceinline__ void dw_slice(const uint16_t* A, const uint16_t* Bm, long long ks, float* out, int* err,
                                         uint8_t* smem)
{
    uint64_t* mbar = (uint64_t*)(smem + DW_BAR);
    uint32_t* tslot = (uint32_t*)(smem + DW_BAR + 16);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t ncols = N < 32 ? 32u : (uint32_t)N;
    if (warp == 0) tc::tmem_alloc(tslot, ncols);
    if (tid < 2) tc::mbar_init(mbar + tid, 1);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    const int kc = (int)(ks < DW_KC ? ks : DW_KC);       // ks is a power of two >= 16: whole chunks
    const int na = kc * 16, nbv = kc * (N / 8);          // 16-byte pieces of a chunk
    constexpr int PA = DW_KC * 16 / FW_THREADS, PB = (DW_KC * (N / 8) + FW_THREADS - 1) / FW_THREADS;
    uint4 ra[PA], rb[PB];
    auto load = [&](long long k0) {
#pragma unroll
        for (int i = 0; i < PA; ++i) {
            const int v = tid + i * FW_THREADS;
            if (v < na) ra[i] = *(const uint4*)(A + (size_t)k0 * 128 + 8 * v);
        }
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            const int v = tid + i * FW_THREADS;
            if (v < nbv) rb[i] = *(const uint4*)(Bm + (size_t)k0 * N + 8 * v);
        }
    };
    load(0);
    uint32_t ph[2] = {0, 0};
    int ok = 1, it = 0;
    for (long long k0 = 0; k0 < ks && ok; k0 += kc, ++it) {
        const int buf = it & 1;
        __syncthreads();                 // the previous chunk's transposes have read the staging
#pragma unroll
        for (int i = 0; i < PA; ++i) {
            const int v = tid + i * FW_THREADS;
            if (v < na) *(uint4*)(smem + (v >> 4) * DW_LD + (v & 15) * 16) = ra[i];
        }
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            const int v = tid + i * FW_THREADS;
            if (v < nbv) *(uint4*)(smem + DW_RAW + (v / (N / 8)) * DW_LD + (v % (N / 8)) * 16) = rb[i];
        }
        if (k0 + kc < ks) load(k0 + kc);
        // the MMAs that read this operand buffer two chunks ago
        int done = 1;
        if (it >= 2) {
            done = tc::mbar_wait(mbar + buf, ph[buf]) ? 1 : 0;
            ph[buf] ^= 1u;
        }
        ok = __syncthreads_and(done);
        if (!ok) break;
        uint8_t* opA = smem + 2 * DW_RAW + buf * 2 * DW_OP;
        uint8_t* opB = opA + DW_OP;
        dw_transpose(smem, opA, 128, kc);
        dw_transpose(smem + DW_RAW, opB, N, kc);
        tc::fence_async_smem();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after();
            const uint32_t idesc = tc::idesc_bf16(128, N);
            const uint32_t a0 = tc::smem_addr(opA), b0 = tc::smem_addr(opB);
            for (int kk = 0; kk < kc / 16; ++kk) {
                const uint64_t ad = tc::smem_desc(a0 + kk * 2 * (128 * 16), 128 * 16, 128);
                const uint64_t bd = tc::smem_desc(b0 + kk * 2 * (N * 16), N * 16, 128);
                tc::mma_bf16(tbase, ad, bd, idesc, (k0 > 0 || kk > 0) ? 1u : 0u);
            }
            tc::mma_commit(mbar + buf);
        }
    }
    // the last one or two chunks' MMAs
    if (ok) {
        int done = 1;
        if (it >= 2) done = tc::mbar_wait(mbar + (it & 1), ph[it & 1]) ? 1 : 0;
        done = (tc::mbar_wait(mbar + ((it - 1) & 1), ph[(it - 1) & 1]) && done) ? 1 : 0;
        ok = __syncthreads_and(done);
    }
    tc::fence_after();
    if (ok) {
        const int rowi = (warp & 3) * 32 + lane;
        const uint32_t tl = tbase + ((uint32_t)((warp & 3) * 32) << 16);
        if (N == 16) {
            if (warp < 4) {
                float v[16];
                tc::tmem_ld16(tl, v);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    *(float4*)(out + rowi * 16 + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c0 = 64 * (warp >> 2) + 32 * h;
                float v[32];
                tc::tmem_ld32(tl + (uint32_t)c0, v);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    *(float4*)(out + rowi * N + c0 + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
        }
    } else if (tid == 0) {
        atomicExch(err, 1);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, ncols);
}

__global__ void __launch_bounds__(FW_THREADS) k_train_dw(const __grid_constant__ DwK k)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int sp = blockIdx.x, g = blockIdx.y;
    const long long ks = k.B / TRAIN_SPLITS;
    const size_t BH = (size_t)k.B * 128, r0 = (size_t)sp * ks;
    if (g == 0) dw_slice<16>(k.H + 2 * BH + r0 * 128, k.dY + r0 * 16, ks, k.part + dw_part_off(0) + sp * 128 * 16, k.err, smem);
    else if (g == 3) dw_slice<16>(k.dZ + r0 * 128, k.Xb + r0 * 16, ks, k.part + dw_part_off(3) + sp * 128 * 16, k.err, smem);
    else dw_slice<128>(k.dZ + (3 - g) * BH + r0 * 128, k.H + (2 - g) * BH + r0 * 128, ks,
                       k.part + dw_part_off(g) + (size_t)sp * 128 * 128, k.err, smem);
}

// One thread per parameter of the flat layout (W1 b1 W2 b2 W3 b3 W4 b4): its
// gradient (slices and CTAs in a fixed order, FP32 slices and FP64 bias
// parts), written to grad when given and, with P, the Adam step (Kingma &
// Ba 2015) on the FP32 master parameters and the handle's bf16 copies: one
// short launch in place of the slice sums, the assembly, Adam and the packing.
struct ApplyK {
    MlpDev w;
    const float* part;
    const double* db;
    int ncta;
    float *grad, *P, *mom, *vel;     // each nullable (P, mom, vel together)
    float lr, b1, b2, eps, c1, c2;
};

__global__ void __launch_bounds__(128) k_train_apply(const __grid_constant__ ApplyK k)
{
    const int t = blockIdx.x * 128 + threadIdx.x;
    if (t >= (int)MLP_NPARAM) return;
    constexpr int ob1 = 128 * 14, oW2 = ob1 + 128, ob2 = oW2 + 128 * 128, oW3 = ob2 + 128, ob3 = oW3 + 128 * 128,
                  oW4 = ob3 + 128, ob4 = oW4 + 9 * 128;
    // layer, output o, input i (-1: the bias)
    int l, o, i;
    if (t < oW2) { l = 0; o = t < ob1 ? t / 14 : t - ob1; i = t < ob1 ? t % 14 : -1; }
    else if (t < oW3) { l = 1; o = t < ob2 ? (t - oW2) >> 7 : t - ob2; i = t < ob2 ? (t - oW2) & 127 : -1; }
    else if (t < oW4) { l = 2; o = t < ob3 ? (t - oW3) >> 7 : t - ob3; i = t < ob3 ? (t - oW3) & 127 : -1; }
    else { l = 3; o = t < ob4 ? (t - oW4) >> 7 : t - ob4; i = t < ob4 ? (t - oW4) & 127 : -1; }
    float g;
    if (i >= 0) {
        const int N = (l == 1 || l == 2) ? 128 : 16;
        const float* p = k.part + dw_part_off(3 - l) + (l == 3 ? i * 16 + o : o * N + i);
        float acc = 0.f;
#pragma unroll
        for (int s = 0; s < TRAIN_SPLITS; ++s) acc += p[(size_t)s * 128 * N];
        g = acc;
    } else {
        double acc = 0.0;
        for (int c = 0; c < k.ncta; ++c) acc += k.db[(size_t)c * TRAIN_NDB + 128 * l + o];
        g = (float)acc;
    }
    if (k.grad) k.grad[t] = g;
    if (!k.P) return;
    const float m = k.b1 * k.mom[t] + (1.0f - k.b1) * g;
    const float v = k.b2 * k.vel[t] + (1.0f - k.b2) * g * g;
    k.mom[t] = m;
    k.vel[t] = v;
    float p = k.P[t];
    p -= k.lr * (m / k.c1) / (sqrtf(v / k.c2) + k.eps);
    k.P[t] = p;
    if (i < 0) {
        (l == 0 ? k.w.b1 : l == 1 ? k.w.b2 : l == 2 ? k.w.b3 : k.w.b4)[o] = p;
        return;
    }
    const uint16_t b = tc::f2bf(p);
    if (l == 0) {
        k.w.W1[o * 16 + i] = b;
    } else if (l == 3) {
        k.w.W4[o * 128 + i] = b;
        k.w.W4t[i * 16 + o] = b;
    } else {
        (l == 1 ? k.w.W2 : k.w.W3)[o * 128 + i] = b;
        (l == 1 ? k.w.W2t : k.w.W3t)[i * 128 + o] = b;
    }
}

}  // namespace fpic

using namespace fpic;

struct fpic_mlp {
    int device = 0, sm_count = 0;
    void* buf = nullptr;     // device: bf16 weights + biases + error word
    MlpDev d{};
    int* err = nullptr;
};

namespace fpic {
const MlpDev& mlp_weights(const fpic_mlp* m) { return m->d; }
int* mlp_err(const fpic_mlp* m) { return m->err; }
int mlp_sm_count(const fpic_mlp* m) { return m->sm_count; }
}  // namespace fpic

static bool g_fwd_attr_set = false;

extern "C" int fpic_mma_bf16(const uint16_t* A, int lda, const uint16_t* B, int ldb, float* C, int ldc, int M,
                             int N, int K, int accumulate, int* err, void* stream)
{
    if (!A || !B || !C || !err) return set_error(FPIC_EINVAL, "fpic_mma_bf16: NULL argument");
    if (M < 1 || N < 16 || N > 256 || N % 16 || K < 16 || K % 16 || lda % 8 || ldb % 8 || lda < K || ldb < K ||
        ldc < N)
        return set_error(FPIC_EINVAL, "fpic_mma_bf16: need N in [16, 256] and K multiples of 16, lda/ldb >= K "
                                      "and multiples of 8, ldc >= N");
    if (((uintptr_t)A | (uintptr_t)B) & 15) return set_error(FPIC_EINVAL, "fpic_mma_bf16: A, B must be 16-byte aligned");
    // 48 KB are used; asking for 100 KB keeps at most two CTAs per SM, so
    // their tensor-memory allocations (<= 256 columns each) always fit.
    const int smem = 100 * 1024;
    static bool attr = false;
    if (!attr) {
        FPIC_CUDA(cudaFuncSetAttribute(k_gemm_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        attr = true;
    }
    k_gemm_bf16<<<(M + 127) / 128, 128, smem, (cudaStream_t)stream>>>(A, lda, B, ldb, C, ldc, M, N, K, accumulate, err);
    FPIC_CUDA(cudaGetLastError());
    return FPIC_OK;
}

extern "C" int fpic_mlp_create(fpic_mlp** out)
{
    if (!out) return set_error(FPIC_EINVAL, "fpic_mlp_create: NULL");
    *out = nullptr;
    fpic_mlp* m = new fpic_mlp();
    int rc = check_cuda(cudaGetDevice(&m->device), "cudaGetDevice");
    if (!rc) rc = check_cuda(cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, m->device), "attr");
    const size_t w_elems = 128 * 16 + 2 * 128 * 128 + 16 * 128 + 2 * 128 * 128 + 128 * 16;
    const size_t bytes = w_elems * 2 + (3 * 128 + 16) * 4 + 256;
    if (!rc) rc = check_cuda(cudaMalloc(&m->buf, bytes), "cudaMalloc(mlp)");
    if (rc) {
        delete m;
        return rc;
    }
    uint16_t* p = (uint16_t*)m->buf;
    m->d.W1 = p; p += 128 * 16;
    m->d.W2 = p; p += 128 * 128;
    m->d.W3 = p; p += 128 * 128;
    m->d.W4 = p; p += 16 * 128;
    m->d.W2t = p; p += 128 * 128;
    m->d.W3t = p; p += 128 * 128;
    m->d.W4t = p; p += 128 * 16;
    float* f = (float*)p;
    m->d.b1 = f; f += 128;
    m->d.b2 = f; f += 128;
    m->d.b3 = f; f += 128;
    m->d.b4 = f; f += 16;
    m->err = (int*)f;
    cudaMemset(m->err, 0, sizeof(int));
    *out = m;
    return FPIC_OK;
}

extern "C" void fpic_mlp_destroy(fpic_mlp* m)
{
    if (!m) return;
    cudaSetDevice(m->device);
    cudaDeviceSynchronize();
    if (m->buf) cudaFree(m->buf);
    delete m;
}

extern "C" long long fpic_mlp_nparams(void) { return MLP_NPARAM; }

extern "C" int fpic_mlp_set_params(fpic_mlp* m, const float* P, void* stream)
{
    if (!m || !P) return set_error(FPIC_EINVAL, "fpic_mlp_set_params: NULL argument");
    k_mlp_pack<<<64, 256, 0, (cudaStream_t)stream>>>(P, m->d);
    FPIC_CUDA(cudaGetLastError());
    return FPIC_OK;
}

static int mlp_forward_impl(fpic_mlp* m, const float* X, float* Y, long long B, const long long* count,
                            cudaStream_t s)
{
    if (!g_fwd_attr_set) {
        FPIC_CUDA(cudaFuncSetAttribute(k_mlp_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, FW_SMEM));
        g_fwd_attr_set = true;
    }
    if (B == 0) return FPIC_OK;
    FwdK k{m->d, X, Y, B, count, m->err};
    const long long ntiles = (B + 127) / 128;
    // two CTAs per SM (~110 KB of shared memory and 128 TMEM columns each) so
    // one CTA's epilogue overlaps the other's MMAs
    const long long cap = 2LL * m->sm_count;
    const unsigned grid = (unsigned)(ntiles < cap ? ntiles : cap);
    k_mlp_fwd<<<grid, FW_THREADS, FW_SMEM, s>>>(k);
    FPIC_CUDA(cudaGetLastError());
    return FPIC_OK;
}

namespace fpic {
int mlp_forward_dev(fpic_mlp* m, const float* X, float* Y, long long B, cudaStream_t s)
{
    return mlp_forward_impl(m, X, Y, B, nullptr, s);
}

int mlp_forward_dev_count(fpic_mlp* m, const float* X, float* Y, long long B, const long long* count,
                          cudaStream_t s)
{
    return mlp_forward_impl(m, X, Y, B, count, s);
}
}  // namespace fpic

extern "C" int fpic_mlp_forward(fpic_mlp* m, const float* X, float* Y, long long B, void* stream)
{
    if (!m || (B > 0 && (!X || !Y))) return set_error(FPIC_EINVAL, "fpic_mlp_forward: NULL argument");
    if (B < 0) return set_error(FPIC_EINVAL, "fpic_mlp_forward: B < 0");
    FPIC_CUDA(cudaSetDevice(m->device));
    return mlp_forward_impl(m, X, Y, B, nullptr, (cudaStream_t)stream);
}

extern "C" int fpic_mlp_status(fpic_mlp* m, int* status)
{
    if (!m || !status) return set_error(FPIC_EINVAL, "fpic_mlp_status: NULL argument");
    FPIC_CUDA(cudaMemcpy(status, m->err, sizeof(int), cudaMemcpyDeviceToHost));
    return *status ? set_error(FPIC_ETIMEOUT, "a tensor-core wait timed out") : FPIC_OK;
}


namespace {

struct TrainBufs {
    long long B = 0;
    void* buf = nullptr;
    float *rowloss, *part;
    double* db;
    uint16_t *H, *dZ, *Xb, *dY;
};

TrainBufs g_tb;   // one training workspace per process (training is serial)

int train_bufs(long long B)
{
    if (g_tb.buf && g_tb.B == B) return 0;
    if (g_tb.buf) FPIC_CUDA(cudaFree(g_tb.buf));
    g_tb.buf = nullptr;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += (b + 255) & ~(size_t)255; return o; };
    const size_t orl = take(B * 4), opart = take((dw_part_off(3) + TRAIN_SPLITS * 128 * 16) * 4),
                 odb = take((size_t)TRAIN_MAX_CTAS * TRAIN_NDB * 8), oH = take(3 * B * 128 * 2),
                 odZ = take(3 * B * 128 * 2), oXb = take(B * 16 * 2), odY = take(B * 16 * 2);
    FPIC_CUDA(cudaMalloc(&g_tb.buf, off));
    char* b = (char*)g_tb.buf;
    g_tb.B = B;
    g_tb.rowloss = (float*)(b + orl);
    g_tb.part = (float*)(b + opart);
    g_tb.db = (double*)(b + odb);
    g_tb.H = (uint16_t*)(b + oH);
    g_tb.dZ = (uint16_t*)(b + odZ);
    g_tb.Xb = (uint16_t*)(b + oXb);
    g_tb.dY = (uint16_t*)(b + odY);
    return 0;
}

// Gradient of the batch loss into grad (nullable) and, with P, the Adam step;
// the loss value when loss_host is given.
int train_impl(fpic_mlp* m, const float* X, const float* T, const float* S, const float* lossw, long long B,
               ApplyK ap, float* loss_host, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        FPIC_CUDA(cudaFuncSetAttribute(k_train_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, TR_SMEM));
        FPIC_CUDA(cudaFuncSetAttribute(k_train_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, DW_SMEM));
        attr = true;
    }
    int rc = train_bufs(B);
    if (rc) return rc;
    TrainBufs& t = g_tb;
    LossW lw;
    for (int k = 0; k < 16; ++k) lw.m[k] = k < 9 ? lossw[k] : 0.f;
    const long long ntiles = B / 128;
    const int cap = m->sm_count < TRAIN_MAX_CTAS ? m->sm_count : TRAIN_MAX_CTAS;
    const int ncta = (int)(ntiles < cap ? ntiles : cap);
    const TrainK tk{m->d, X, T, S, lw, B, 1.0f / (float)B, t.rowloss, t.H, t.dZ, t.Xb, t.dY, t.db, m->err};
    k_train_tile<<<ncta, FW_THREADS, TR_SMEM, s>>>(tk);
    const DwK dk{t.H, t.dZ, t.Xb, t.dY, B, t.part, m->err};
    k_train_dw<<<dim3(TRAIN_SPLITS, 4), FW_THREADS, DW_SMEM, s>>>(dk);
    ap.w = m->d;
    ap.part = t.part;
    ap.db = t.db;
    ap.ncta = ncta;
    k_train_apply<<<(unsigned)((MLP_NPARAM + 127) / 128), 128, 0, s>>>(ap);
    FPIC_CUDA(cudaGetLastError());
    if (loss_host) {
        std::vector<float> h(B);
        FPIC_CUDA(cudaMemcpyAsync(h.data(), t.rowloss, B * 4, cudaMemcpyDeviceToHost, s));
        FPIC_CUDA(cudaStreamSynchronize(s));
        double L = 0.0;
        for (long long b = 0; b < B; ++b) L += h[b];
        *loss_host = (float)(L / (double)B);
    }
    return FPIC_OK;
}

bool mlp_batch_ok(long long B)
{
    return B >= 16 * TRAIN_SPLITS && (B & (B - 1)) == 0 && B <= (1LL << 24);
}

}  // namespace

extern "C" int fpic_mlp_grad(fpic_mlp* m, const float* X, const float* T, const float* S, const float* lossw,
                             long long B, float* grad, float* loss, void* stream)
{
    if (!m || !X || !T || !S || !lossw || !grad) return set_error(FPIC_EINVAL, "fpic_mlp_grad: NULL argument");
    if (!mlp_batch_ok(B)) return set_error(FPIC_EINVAL, "fpic_mlp_grad: B must be a power of two in [256, 2^24]");
    FPIC_CUDA(cudaSetDevice(m->device));
    ApplyK ap{};
    ap.grad = grad;
    return train_impl(m, X, T, S, lossw, B, ap, loss, (cudaStream_t)stream);
}

extern "C" int fpic_mlp_train_step(fpic_mlp* m, float* P, float* mom, float* vel, const float* X, const float* T,
                                   const float* S, const float* lossw, long long B, int step, float lr, float beta1,
                                   float beta2, float eps, float* loss, void* stream)
{
    if (!m || !P || !mom || !vel || !X || !T || !S || !lossw) return set_error(FPIC_EINVAL, "fpic_mlp_train_step: NULL argument");
    if (!mlp_batch_ok(B)) return set_error(FPIC_EINVAL, "fpic_mlp_train_step: B must be a power of two in [256, 2^24]");
    if (step < 1 || !(lr > 0.f)) return set_error(FPIC_EINVAL, "fpic_mlp_train_step: step >= 1 and lr > 0 required");
    FPIC_CUDA(cudaSetDevice(m->device));
    ApplyK ap{};
    ap.P = P;
    ap.mom = mom;
    ap.vel = vel;
    ap.lr = lr;
    ap.b1 = beta1;
    ap.b2 = beta2;
    ap.eps = eps;
    ap.c1 = 1.0f - powf(beta1, (float)step);
    ap.c2 = 1.0f - powf(beta2, (float)step);
    return train_impl(m, X, T, S, lossw, B, ap, loss, (cudaStream_t)stream);
}
