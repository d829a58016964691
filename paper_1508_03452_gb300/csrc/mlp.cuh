// mlp.cuh -- the learned seed of the primitive recovery: a 20-64-64-64-4 ReLU
// network mapping normalised moments to the velocity (and eps / T^00 - 1).
// It only supplies the starting vector of the Landau eigen-solve; the solve
// itself (and its result) is the method's.
//
// Parameters (float32 master copy, MLP_NPARAM values): W1[64][20] b1[64]
// W2[64][64] b2[64] W3[64][64] b3[64] W4[4][64] b4[4], W[out][in].
//
// Inference inside the tile, batched and persistent step kernels and the standalone one
// use warp-level bf16 tensor-core MMA (mma.sync m16n8k16, float32 accumulation): each
// warp owns the 32 cells (rows) of its threads, so no block-wide barrier is needed and no
// block holds tensor memory while it waits for another. The one-run step kernel uses
// the tensor-memory form (mlp_tc.cuh), whose sums agree with these bit for bit.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include <cstring>

namespace lb {

constexpr int MLP_IN = 20, MLP_H = 64, MLP_OUT = 4;
constexpr int MLP_W1 = 0, MLP_B1 = MLP_W1 + MLP_H * MLP_IN, MLP_W2 = MLP_B1 + MLP_H,
              MLP_B2 = MLP_W2 + MLP_H * MLP_H, MLP_W3 = MLP_B2 + MLP_H, MLP_B3 = MLP_W3 + MLP_H * MLP_H,
              MLP_W4 = MLP_B3 + MLP_H, MLP_B4 = MLP_W4 + MLP_OUT * MLP_H, MLP_NPARAM = MLP_B4 + MLP_OUT;

// Shared feature rows: 40 bf16 (80 bytes, a multiple of 16 for ldmatrix) per
// cell, 20 features and zeros up to 32, so the 8 rows of one 8x8 fragment fall in
// distinct banks. The network's outputs come back as floats in the same rows.
constexpr int MLP_FROW = 40;
// Device inference blob: bf16 weights in MMA fragment order, then float32
// biases. Layer l (K inputs padded to 32 or 64, N outputs padded to a
// multiple of 8, zero padding) stores, for output row r, k-tile kt (16 wide)
// and lane column group t (0..3), the 4 values W[r][16 kt + 2t + {0, 1, 8, 9}]
// at ((r * K/16 + kt) * 4 + t) * 4: the B fragment of one lane is one 8-byte load.
constexpr int MLP_K1 = 32;  // first-layer inputs, padded
constexpr int MLPD_W1 = 0, MLPD_W2 = MLPD_W1 + MLP_H * MLP_K1, MLPD_W3 = MLPD_W2 + MLP_H * MLP_H,
              MLPD_W4 = MLPD_W3 + MLP_H * MLP_H, MLPD_NBF16 = MLPD_W4 + 8 * MLP_H;
constexpr int MLPD_NBIAS = 3 * MLP_H + 8;                                // float32 biases after the bf16 block
constexpr int MLPD_BYTES = MLPD_NBF16 * 2 + MLPD_NBIAS * 4;              // device inference blob
constexpr int MLP_ACT_BYTES_PER_CELL = MLP_FROW * 2;                     // shared feature row per cell

// blob index of weight (r, k) of a layer with K inputs (fragment order above)
__host__ __device__ constexpr int mlpd_frag_index(int r, int k, int K)
{
    return ((r * (K / 16) + k / 16) * 4 + (k % 8) / 2) * 4 + ((k % 16) / 8) * 2 + (k % 2);
}

// normalised features of one cell: T^{mu nu} / T^00 (9), N^a / N^0 (3),
// N^0 / T^00, E_old / sqrt(T^00) (3), B_old / sqrt(T^00) (3), 1
template <class R>
__device__ __forceinline__ void mlp_features(R T00, const R* T0a, const R* Tab /* xx yy zz xy xz yz */, R N0,
                                             const R* Na, const R* E_old, const R* B_old, float* x)
{
    const R it = R(1) / T00;
    const R is = sqrt(it);
    for (int a = 0; a < 3; ++a) x[a] = (float)(T0a[a] * it);
    for (int m = 0; m < 6; ++m) x[3 + m] = (float)(Tab[m] * it);
    const R in = R(1) / N0;
    for (int a = 0; a < 3; ++a) x[9 + a] = (float)(Na[a] * in);
    x[12] = (float)(N0 * it);
    for (int a = 0; a < 3; ++a) {
        x[13 + a] = (float)(E_old[a] * is);
        x[16 + a] = (float)(B_old[a] * is);
    }
    x[19] = 1.0f;
}

// four 8x8 bf16 matrices from shared memory (row addresses from lanes 0..31)
__device__ __forceinline__ void ldmatrix_x4(uint32_t* r, const __nv_bfloat16* row_addr)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(row_addr);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Warp order of the blob's weights: 8-byte fragment i of the blob (row r, k-tile
// kt, lane column group t of its layer) goes where the fragments of the 32 lanes
// that use them together, for two k-tiles at a time, are consecutive: a warp's
// load is 512 bytes in a row. In the blob's own order the 8 rows of a fragment
// lie K * 2 bytes apart, in the same shared-memory banks.
// (i = base + at; a constant `at` that is the same side of the layers' starts for every
// `base` settles the layer at compile time)
__device__ __forceinline__ int mlp_warp_order(int base, int at)
{
    const int first = at < MLPD_W2 / 4 ? 0 : (at < MLPD_W3 / 4 ? MLPD_W2 / 4 : (at < MLPD_W4 / 4 ? MLPD_W3 / 4 : MLPD_W4 / 4));
    const int kt_count = first == 0 ? MLP_K1 / 16 : MLP_H / 16;
    const int j = base + (at - first), t = j % 4, kt = (j / 4) % kt_count, r = j / (4 * kt_count);
    const int lane = (r % 8) * 4 + t;
    return first + ((r / 8) * kt_count + (kt & ~1)) * 32 + 2 * lane + (kt & 1);
}
__device__ __forceinline__ int mlp_warp_order(int i) { return mlp_warp_order(0, i); }

// a vector of the blob, in global memory (read-only path) or the block's shared copy
template <bool GLOBAL, class T>
__device__ __forceinline__ T mlp_ld(const T* p)
{
    if constexpr (GLOBAL)
        return __ldg(p);
    else
        return *p;
}

// One hidden layer with the activations kept in registers: the accumulator
// fragment of two 8-wide output tiles is, packed to bf16, the A fragment of one
// 16-wide k-tile of the next layer, so no activation goes through shared memory.
// A: [m-tile][k-tile][register] of the K inputs; on return the 64 outputs. The
// weights are in warp order (mlp_warp_order): two k-tiles' fragments of the 32
// lanes are 512 consecutive bytes, one 16-byte load a lane.
template <int K, int MT, bool GLOBAL>
__device__ __forceinline__ void mlp_layer_frag(uint32_t (&A)[MT][4][4], const __nv_bfloat16* W, const float* bias)
{
    const int lane = threadIdx.x & 31, tig = lane & 3;
    constexpr int KT = K / 16;
    const __nv_bfloat162 zero2 = __floats2bfloat162_rn(0.0f, 0.0f);
    uint32_t N[MT][4][4];
#pragma unroll
    for (int np = 0; np < 4; ++np) {  // output tiles 2 np, 2 np + 1: four independent chains of products
        float acc[2][MT][4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float2 b = mlp_ld<GLOBAL>(reinterpret_cast<const float2*>(bias + 8 * (2 * np + q) + 2 * tig));
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                acc[q][mt][0] = acc[q][mt][2] = b.x;
                acc[q][mt][1] = acc[q][mt][3] = b.y;
            }
        }
#pragma unroll
        for (int kt = 0; kt < KT; kt += 2) {
            uint4 bw[2];
#pragma unroll
            for (int q = 0; q < 2; ++q)
                bw[q] = mlp_ld<GLOBAL>(reinterpret_cast<const uint4*>(W + (((2 * np + q) * KT + kt) * 32 + 2 * lane) * 4));
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const uint32_t b[2] = {h ? bw[q].z : bw[q].x, h ? bw[q].w : bw[q].y};
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) mma_bf16(acc[q][mt], A[mt][kt + h], b);
                }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const __nv_bfloat162 v =
                        __hmax2(__floats2bfloat162_rn(acc[q][mt][2 * hh], acc[q][mt][2 * hh + 1]), zero2);
                    memcpy(&N[mt][np][2 * q + hh], &v, 4);
                }
    }
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int kt = 0; kt < 4; ++kt)
#pragma unroll
            for (int r = 0; r < 4; ++r) A[mt][kt][r] = N[mt][kt][r];
}

// Forward pass of 16 MT of the warp's rows: `rows` (shared) holds MLP_FROW bf16 per row,
// 20 features then zeros up to 32; `wts` the inference blob in warp order
// (GLOBAL: in global memory).
// y[mt]: the accumulator fragment of rows 16 mt.. (columns 0..3 are the outputs:
// lanes with lane % 4 < 2 hold columns 2 (lane % 4), + 1 of rows lane / 4, + 8).
template <int MT, bool GLOBAL>
__device__ __forceinline__ void mlp_forward_frag(const __nv_bfloat16* rows, const unsigned char* wts, float (&y)[MT][4])
{
    const int lane = threadIdx.x & 31, tig = lane & 3;
    const __nv_bfloat16* W = reinterpret_cast<const __nv_bfloat16*>(wts);
    const float* bias = reinterpret_cast<const float*>(wts + MLPD_NBF16 * 2);
    uint32_t A[MT][4][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int kt = 0; kt < 2; ++kt) ldmatrix_x4(A[mt][kt], rows + (16 * mt + (lane & 15)) * MLP_FROW + 16 * kt + (lane >> 4) * 8);
    mlp_layer_frag<MLP_K1, MT, GLOBAL>(A, W + MLPD_W1, bias);
    mlp_layer_frag<MLP_H, MT, GLOBAL>(A, W + MLPD_W2, bias + MLP_H);
    mlp_layer_frag<MLP_H, MT, GLOBAL>(A, W + MLPD_W3, bias + 2 * MLP_H);
    const float2 b = mlp_ld<GLOBAL>(reinterpret_cast<const float2*>(bias + 3 * MLP_H + 2 * tig));
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        y[mt][0] = y[mt][2] = b.x;
        y[mt][1] = y[mt][3] = b.y;
    }
#pragma unroll
    for (int kt = 0; kt < 4; kt += 2) {
        const uint4 bw = mlp_ld<GLOBAL>(reinterpret_cast<const uint4*>(W + MLPD_W4 + (kt * 32 + 2 * lane) * 4));
        const uint32_t b0[2] = {bw.x, bw.y}, b1[2] = {bw.z, bw.w};
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) mma_bf16(y[mt], A[mt][kt], b0);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) mma_bf16(y[mt], A[mt][kt + 1], b1);
    }
}

// float32 parameters (device) -> the step kernels' copies of the weights
// (mlp_step_weight_bytes() bytes), on stream s: the blob with its fragments in warp
// order, then the tensor core's order
int mlp_step_weight_bytes();
cudaError_t launch_mlp_pack_step(const float* params, unsigned char* blob, cudaStream_t s);

}  // namespace lb
