// mlp.cu -- training and standalone inference kernels of the learned recovery
// seed (see mlp.cuh), and their C-ABI entry points.
//
// Training runs in float32 on the CUDA cores. A block takes kTS samples at a
// time through the whole network: weights and activations in shared memory,
// every thread a fixed set of gradient entries in registers over all the
// block's samples. The blocks' partial sums are added in a fixed order by the
// kernel that also takes the Adam step, so a gradient (and a training run) is
// bit-reproducible. Samples are rows of 24 float32: 20 features then 4 targets
// (beta, eps / T^00 - 1). Loss: mean over samples of the squared error summed
// over the 4 outputs.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "lbrmhd.h"
#include "mlp.cuh"
#include "mlp_tc.cuh"
#include "tma.cuh"

namespace lb {

constexpr int MLP_ROW = MLP_IN + MLP_OUT;
static_assert(MLP_NPARAM == LBRMHD_MLP_NPARAM && MLP_IN == LBRMHD_MLP_NFEAT && MLP_ROW == LBRMHD_MLP_ROW,
              "network layout differs from the C ABI");
constexpr int kTrainThreads = 256;
constexpr int kTS = 8;                                // samples per block and pass
constexpr int kTrainStride = (MLP_NPARAM + 1 + 3) / 4 * 4;  // floats per block of partial sums (16-byte rows)
// shared-memory rows: 68 floats per 64-wide row (16-byte vectors of 8
// consecutive rows fall in distinct banks), 20 per first-layer row
constexpr int kWRow = 68;
constexpr int TS_W1 = 0, TS_W2 = TS_W1 + MLP_H * MLP_IN, TS_W3 = TS_W2 + MLP_H * kWRow, TS_W4 = TS_W3 + MLP_H * kWRow,
              TS_B = TS_W4 + MLP_OUT * MLP_H, TS_X = TS_B + 3 * MLP_H + 4, TS_A = TS_X + kTS * MLP_ROW;
constexpr int kActs = 6;  // h1, h2, h3, d3, d2, d1
constexpr int TS_DY = TS_A + kActs * kTS * MLP_H, TS_LOSS = TS_DY + kTS * MLP_OUT,
              kTrainSmem = (TS_LOSS + kTS) * 4;
static_assert(TS_W2 % 4 == 0 && TS_W4 % 4 == 0 && TS_X % 4 == 0 && TS_A % 4 == 0 && TS_DY % 4 == 0,
              "16-byte alignment of the shared-memory arrays");

__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// 16 bytes from global memory (through L2) into shared memory, and the wait for
// all of a thread's copies
__device__ __forceinline__ void cp_async16(float* dst, const float* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ float dot4(float4 a, float4 b, float s)
{
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
}

// one hidden layer of the block's kTS samples: out[s][o] = relu(b[o] + W[o] . in[s])
// (thread: neuron o = t % 64, samples t / 64 and t / 64 + 4)
template <int K>
__device__ __forceinline__ void train_layer(const float* W, int wrow, const float* bias, const float* in, int irow,
                                            float* out)
{
    const int o = threadIdx.x % MLP_H, s0 = threadIdx.x / MLP_H;
    float a0 = bias[o], a1 = a0;
    const float4* w = reinterpret_cast<const float4*>(W + o * wrow);
    const float4* x0 = reinterpret_cast<const float4*>(in + s0 * irow);
    const float4* x1 = reinterpret_cast<const float4*>(in + (s0 + 4) * irow);
#pragma unroll
    for (int k = 0; k < K / 4; ++k) {
        const float4 wk = w[k];
        a0 = dot4(wk, x0[k], a0);
        a1 = dot4(wk, x1[k], a1);
    }
    out[s0 * MLP_H + o] = fmaxf(a0, 0.0f);
    out[(s0 + 4) * MLP_H + o] = fmaxf(a1, 0.0f);
}

// delta of the layer below: out[s][k] = (h[s][k] > 0) sum_o W[o][k] d[s][o]
__device__ __forceinline__ void train_delta(const float* W, const float* d, const float* h, float* out)
{
    const int k = threadIdx.x % MLP_H, s0 = threadIdx.x / MLP_H;
    float a0 = 0.0f, a1 = 0.0f;
    const float4* d0 = reinterpret_cast<const float4*>(d + s0 * MLP_H);
    const float4* d1 = reinterpret_cast<const float4*>(d + (s0 + 4) * MLP_H);
#pragma unroll
    for (int o = 0; o < MLP_H; o += 4) {
        const float4 w = make_float4(W[o * kWRow + k], W[(o + 1) * kWRow + k], W[(o + 2) * kWRow + k],
                                     W[(o + 3) * kWRow + k]);
        a0 = dot4(w, d0[o / 4], a0);
        a1 = dot4(w, d1[o / 4], a1);
    }
    out[s0 * MLP_H + k] = h[s0 * MLP_H + k] > 0.0f ? a0 : 0.0f;
    out[(s0 + 4) * MLP_H + k] = h[(s0 + 4) * MLP_H + k] > 0.0f ? a1 : 0.0f;
}

// 4 x 4 entries of a 64 x 64 weight gradient: g[i][j] += sum_s d[s][o0 + i] h[s][k0 + j]
__device__ __forceinline__ void train_outer(const float* d, const float* h, int o0, int k0, float (&g)[4][4])
{
#pragma unroll
    for (int s = 0; s < kTS; ++s) {
        const float4 dv = *reinterpret_cast<const float4*>(d + s * MLP_H + o0);
        const float4 hv = *reinterpret_cast<const float4*>(h + s * MLP_H + k0);
        const float dd[4] = {dv.x, dv.y, dv.z, dv.w}, hh[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) g[i][j] = fmaf(dd[i], hh[j], g[i][j]);
    }
}

// Loss and gradient sums of a block's share of `count` samples. Sample j of the
// batch is row (sample_seed ? hash(sample_seed, j) mod n : j).
// What bounds it: a batch is little work (60 kFLOP a sample, 61 MFLOP for 1024:
// 1 us at the float32 rate) in a chain of seven dependent layers, so latency
// does; 8 samples a block spread a batch of 1024 over 128 of the 152 SMs, and
// each layer is one pass of 256 threads between two barriers. The one warp per
// sample kernel before it read the weights from L1 at a stride (and added into
// shared memory with 32-way bank conflicts): 164 us per batch of 1024, now 12 us.
__global__ void __launch_bounds__(kTrainThreads) mlp_grad_kernel(const float* P,
                                                                 const float* __restrict__ data, int64_t n,
                                                                 int64_t count, uint64_t sample_seed,
                                                                 float* partial, float inv_count)
{
    extern __shared__ __align__(16) float sm[];
    const int t = threadIdx.x;
    grid_release();
    // a thread's share of a tile's rows: one 16-byte vector of kTS x 24 floats
    constexpr int kRowVecs = MLP_ROW / 4;
    const int64_t ntiles = (count + kTS - 1) / kTS;
    auto fetch = [&](int64_t tile) {
        const int64_t j = tile * kTS + t / kRowVecs;
        if (t >= kTS * kRowVecs || tile >= ntiles || j >= count) return make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const int64_t row = sample_seed ? (int64_t)(splitmix64(sample_seed ^ (uint64_t)j * 0x2545F4914F6CDD1Dull) %
                                                    (uint64_t)n)
                                        : j;
        const float* p = data + row * MLP_ROW + 4 * (t % kRowVecs);
        return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));  // the caller's rows may be 4-byte aligned
    };
    float4 next = fetch(blockIdx.x);
    grid_wait();  // the parameters are the previous step's output
    const bool aligned = (reinterpret_cast<uintptr_t>(P) & 15) == 0;
    // from L2 (an L1 line could hold the step before the last), all in flight at once
    auto copy = [&](int dst, int src) {  // 4 parameters
        if (aligned) {
            cp_async16(sm + dst, P + src);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) sm[dst + q] = __ldcg(P + src + q);
        }
    };
    for (int i = t; i < MLP_H * MLP_IN / 4; i += kTrainThreads) copy(TS_W1 + 4 * i, MLP_W1 + 4 * i);
#pragma unroll
    for (int r = 0; r < MLP_H * MLP_H / 4 / kTrainThreads; ++r) {
        const int i = t + r * kTrainThreads, at = (i / (MLP_H / 4)) * kWRow + 4 * (i % (MLP_H / 4));
        copy(TS_W2 + at, MLP_W2 + 4 * i);
        copy(TS_W3 + at, MLP_W3 + 4 * i);
    }
    if (t < MLP_OUT * MLP_H / 4)
        copy(TS_W4 + 4 * t, MLP_W4 + 4 * t);
    else if (t < MLP_OUT * MLP_H / 4 + 3 * MLP_H / 4) {
        const int i = t - MLP_OUT * MLP_H / 4, l = i / (MLP_H / 4), q = 4 * (i % (MLP_H / 4));
        copy(TS_B + l * MLP_H + q, (l == 0 ? MLP_B1 : (l == 1 ? MLP_B2 : MLP_B3)) + q);
    } else if (t == MLP_OUT * MLP_H / 4 + 3 * MLP_H / 4) {
        copy(TS_B + 3 * MLP_H, MLP_B4);
    }
    static_assert(MLP_OUT * MLP_H == kTrainThreads, "one output weight per thread");
    static_assert(MLP_W2 % 4 == 0 && MLP_W3 % 4 == 0 && MLP_W4 % 4 == 0 && MLP_B1 % 4 == 0 && MLP_B4 % 4 == 0, "vectors");
    cp_async_wait();
    float* x = sm + TS_X;
    float* h1 = sm + TS_A;
    float* h2 = h1 + kTS * MLP_H;
    float* h3 = h2 + kTS * MLP_H;
    float* d3 = h3 + kTS * MLP_H;
    float* d2 = d3 + kTS * MLP_H;
    float* d1 = d2 + kTS * MLP_H;
    float* dy = sm + TS_DY;
    float* ls = sm + TS_LOSS;
    // this thread's gradient entries: 4 x 4 of W2 and of W3 (rows 4 (t / 16),
    // columns 4 (t % 16)), 5 of W1 (row t / 4), one of W4, one bias
    const int o0 = 4 * (t / 16), k0 = 4 * (t % 16), o1 = t / 4, k1 = 5 * (t % 4);
    float g2[4][4] = {}, g3[4][4] = {}, g1[5] = {}, g4 = 0.0f, gb = 0.0f, loss = 0.0f;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        if (t < kTS * kRowVecs) reinterpret_cast<float4*>(x)[t] = next;
        __syncthreads();
        next = fetch(tile + gridDim.x);
        train_layer<MLP_IN>(sm + TS_W1, MLP_IN, sm + TS_B, x, MLP_ROW, h1);
        __syncthreads();
        train_layer<MLP_H>(sm + TS_W2, kWRow, sm + TS_B + MLP_H, h1, MLP_H, h2);
        __syncthreads();
        train_layer<MLP_H>(sm + TS_W3, kWRow, sm + TS_B + 2 * MLP_H, h2, MLP_H, h3);
        __syncthreads();
        {  // outputs: 8 lanes per (sample, output), 8 inputs each
            const int o = (t / 8) % MLP_OUT, s = t / (8 * MLP_OUT), q = t % 8;
            const float4* w = reinterpret_cast<const float4*>(sm + TS_W4 + o * MLP_H + 8 * q);
            const float4* h = reinterpret_cast<const float4*>(h3 + s * MLP_H + 8 * q);
            float a = dot4(w[1], h[1], dot4(w[0], h[0], 0.0f));
#pragma unroll
            for (int m = 4; m > 0; m >>= 1) a += __shfl_xor_sync(0xffffffffu, a, m);
            const bool in = tile * kTS + s < count;
            const float e = in ? a + sm[TS_B + 3 * MLP_H + o] - x[s * MLP_ROW + MLP_IN + o] : 0.0f;
            float e2 = e * e;  // summed over the 4 outputs of the sample
            e2 += __shfl_xor_sync(0xffffffffu, e2, 8);
            e2 += __shfl_xor_sync(0xffffffffu, e2, 16);
            if (q == 0) dy[s * MLP_OUT + o] = 2.0f * e * inv_count;
            if (t % 32 == 0) ls[s] = e2 * inv_count;
        }
        __syncthreads();
        {  // output layer's gradient and the delta of layer 3
            const int o = t / MLP_H, k = t % MLP_H;
#pragma unroll
            for (int s = 0; s < kTS; ++s) g4 = fmaf(dy[s * MLP_OUT + o], h3[s * MLP_H + k], g4);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int s = o + 4 * r;
                const float4 dv = *reinterpret_cast<const float4*>(dy + s * MLP_OUT);
                const float4 w = make_float4(sm[TS_W4 + k], sm[TS_W4 + MLP_H + k], sm[TS_W4 + 2 * MLP_H + k],
                                             sm[TS_W4 + 3 * MLP_H + k]);
                d3[s * MLP_H + k] = h3[s * MLP_H + k] > 0.0f ? dot4(w, dv, 0.0f) : 0.0f;
            }
            if (t == 0)
#pragma unroll
                for (int s = 0; s < kTS; ++s) loss += ls[s];
        }
        __syncthreads();
        train_delta(sm + TS_W3, d3, h2, d2);
        train_outer(d3, h2, o0, k0, g3);
        __syncthreads();
        train_delta(sm + TS_W2, d2, h1, d1);
        train_outer(d2, h1, o0, k0, g2);
        __syncthreads();
#pragma unroll
        for (int s = 0; s < kTS; ++s) {
            const float dv = d1[s * MLP_H + o1];
#pragma unroll
            for (int j = 0; j < 5; ++j) g1[j] = fmaf(dv, x[s * MLP_ROW + k1 + j], g1[j]);
        }
        {  // biases: threads 0..63 layer 1, ..127 layer 2, ..191 layer 3, ..195 the outputs
            const float* d = t < MLP_H ? d1 : (t < 2 * MLP_H ? d2 : d3);
            if (t < 3 * MLP_H) {
#pragma unroll
                for (int s = 0; s < kTS; ++s) gb += d[s * MLP_H + t % MLP_H];
            } else if (t < 3 * MLP_H + MLP_OUT) {
#pragma unroll
                for (int s = 0; s < kTS; ++s) gb += dy[s * MLP_OUT + t - 3 * MLP_H];
            }
        }
        __syncthreads();  // x, the deltas and dy are rewritten by the next tile
    }
    float* out = partial + (int64_t)blockIdx.x * kTrainStride;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        *reinterpret_cast<float4*>(out + MLP_W2 + (o0 + i) * MLP_H + k0) =
            make_float4(g2[i][0], g2[i][1], g2[i][2], g2[i][3]);
        *reinterpret_cast<float4*>(out + MLP_W3 + (o0 + i) * MLP_H + k0) =
            make_float4(g3[i][0], g3[i][1], g3[i][2], g3[i][3]);
    }
#pragma unroll
    for (int j = 0; j < 5; ++j) out[MLP_W1 + o1 * MLP_IN + k1 + j] = g1[j];
    out[MLP_W4 + t] = g4;
    if (t < MLP_H)
        out[MLP_B1 + t] = gb;
    else if (t < 2 * MLP_H)
        out[MLP_B2 + t - MLP_H] = gb;
    else if (t < 3 * MLP_H)
        out[MLP_B3 + t - 2 * MLP_H] = gb;
    else if (t < 3 * MLP_H + MLP_OUT)
        out[MLP_B4 + t - 3 * MLP_H] = gb;
    if (t == 0) out[MLP_NPARAM] = loss;
}

// Adam's constants of one step (ADAM), c1 and c2 the bias corrections
struct AdamStep {
    float lr, b1, b2, eps, c1, c2;
};

// Adds the blocks' partial sums (8 interleaved shares, each in block order, then
// the shares in order) and either writes the gradient and the loss, or takes
// the Adam step m = b1 m + (1 - b1) g, v = b2 v + (1 - b2) g^2, p -= lr mhat /
// (sqrt(vhat) + eps). 32 entries a block: 311 blocks read the partials at once
// (a batch of 1024: 5 MB from L2), and the step that follows needs no launch of its
// own. 18 us a step of 1024 samples in all, 181 us before.
constexpr int kReduceShares = 8;
template <bool ADAM>
__global__ void __launch_bounds__(32 * kReduceShares) mlp_reduce_kernel(const float* partial, int nblocks,
                                                                                 float* grad, float* P, float* m, float* v,
                                                                                 float* loss, AdamStep a)
{
    __shared__ float sh[kReduceShares][32];
    const int lane = threadIdx.x % 32, share = threadIdx.x / 32, i = blockIdx.x * 32 + lane;
    grid_release();
    grid_wait();
    float s = 0.0f;
    if (i <= MLP_NPARAM) {
#pragma unroll 8
        for (int b = share; b < nblocks; b += kReduceShares) s += __ldcg(partial + (int64_t)b * kTrainStride + i);  // L2, as the parameters above
    }
    sh[share][lane] = s;
    __syncthreads();
    if (share || i > MLP_NPARAM) return;
    float g = 0.0f;
#pragma unroll
    for (int q = 0; q < kReduceShares; ++q) g += sh[q][lane];
    if constexpr (!ADAM) {
        grad[i] = g;
    } else {
        if (i == MLP_NPARAM) {
            if (loss) *loss = g;
            return;
        }
        // from L2: a launch that started early may share its SM with a block of the
        // step before the last, whose L1 lines of m and v reach into this block's
        const float mi = a.b1 * __ldcg(m + i) + (1.0f - a.b1) * g;
        const float vi = a.b2 * __ldcg(v + i) + (1.0f - a.b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        P[i] = __ldcg(P + i) - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
    }
}

// float32 parameters -> bf16 inference blob in fragment order (zero padding); STEP:
// the step kernels' own two copies instead, fragments in warp order (mma.sync), then
// the tensor core's order (mlp_tc.cuh)
template <bool STEP>
__global__ void mlp_pack_kernel(const float* __restrict__ P, unsigned char* __restrict__ blob)
{
    __nv_bfloat16* W = reinterpret_cast<__nv_bfloat16*>(blob);
    __nv_bfloat16* C = reinterpret_cast<__nv_bfloat16*>(blob + MLPD_BYTES);
    float* bias = reinterpret_cast<float*>(blob + MLPD_NBF16 * 2);
    // weight (r, k) of the layer that starts at `at` of the blob and `tc` of the tensor core's copy
    auto put = [&](int at, int tc, int r, int k, int K, float v) {
        const int e = at + mlpd_frag_index(r, k, K);
        const __nv_bfloat16 b = __float2bfloat16_rn(v);
        W[STEP ? 4 * mlp_warp_order(e / 4) + e % 4 : e] = b;
        if constexpr (STEP) C[tc + mlpt_index(r, MLPT_KB + k, MLPT_KB + K)] = b;
    };
    const int total = MLP_H * MLP_K1 + 2 * MLP_H * MLP_H + 8 * MLP_H + MLPD_NBIAS;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        // i enumerates (layer, r, k) in row-major order, then the biases
        if (i < MLP_H * MLP_K1) {
            const int r = i / MLP_K1, k = i % MLP_K1;
            put(MLPD_W1, MLPT_W1, r, k, MLP_K1, k < MLP_IN ? P[MLP_W1 + r * MLP_IN + k] : 0.0f);
        } else if (i < MLP_H * MLP_K1 + MLP_H * MLP_H) {
            const int j = i - MLP_H * MLP_K1, r = j / MLP_H, k = j % MLP_H;
            put(MLPD_W2, MLPT_W2, r, k, MLP_H, P[MLP_W2 + r * MLP_H + k]);
        } else if (i < MLP_H * MLP_K1 + 2 * MLP_H * MLP_H) {
            const int j = i - MLP_H * MLP_K1 - MLP_H * MLP_H, r = j / MLP_H, k = j % MLP_H;
            put(MLPD_W3, MLPT_W3, r, k, MLP_H, P[MLP_W3 + r * MLP_H + k]);
        } else if (i < MLP_H * MLP_K1 + 2 * MLP_H * MLP_H + 8 * MLP_H) {
            const int j = i - MLP_H * MLP_K1 - 2 * MLP_H * MLP_H, r = j / MLP_H, k = j % MLP_H;
            put(MLPD_W4, MLPT_W4, r, k, MLP_H, r < MLP_OUT ? P[MLP_W4 + r * MLP_H + k] : 0.0f);
            if constexpr (STEP) C[MLPT_W4 + mlpt_index(r + 8, MLPT_KB + k, MLPT_K)] = __float2bfloat16_rn(0.0f);
        } else {
            const int j = i - (MLP_H * MLP_K1 + 2 * MLP_H * MLP_H + 8 * MLP_H);
            float val = 0.0f;
            if (j < 64) val = P[MLP_B1 + j];
            else if (j < 128) val = P[MLP_B2 + j - 64];
            else if (j < 192) val = P[MLP_B3 + j - 128];
            else if (j < 192 + MLP_OUT) val = P[MLP_B4 + j - 192];
            bias[j] = val;
            if constexpr (STEP) {
                mlpt_put_bias(C, j / MLP_H, j % MLP_H, val);
                if (j >= 3 * MLP_H) mlpt_put_bias(C, 3, j % MLP_H + 8, 0.0f);
            }
        }
    }
}

// Standalone inference: a warp takes 32 rows at a time through the network, the
// activations staying in its registers from layer to layer (mlp_forward_frag),
// the weights read from the block's shared copy; same products and sums in the
// same order as the batched step kernels'. Bound by the warp-level matrix instructions
// (168 mma.sync per 32 rows): 55 us for 1,000,003 rows. The rows arrive as coalesced
// 16-byte loads for the next tile while this one is computed. Before, activations went
// through shared memory, and the rows and the weight fragments were loaded at
// strides: L1 92 % busy, 121 us.
constexpr int kInferWarps = 4, kInferBlocks = 3;  // warps per block, blocks per SM (4: 128 registers spill, 74 us)
__global__ void __launch_bounds__(32 * kInferWarps, kInferBlocks) mlp_infer_kernel(const unsigned char* __restrict__ blob,
                                                                        const float* __restrict__ feat, int64_t n,
                                                                        float* __restrict__ out)
{
    __shared__ __align__(16) unsigned char wts[(MLPD_BYTES + 15) / 16 * 16];
    __shared__ __align__(16) __nv_bfloat16 rows[kInferWarps][32 * MLP_FROW];
    const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
    // the blob's fragments (8 bytes a lane), those of a warp's lanes side by side
    // (unrolled, all loads in flight at once: a call of few rows is mostly this, 100 to
    // 10,000 rows 3.3 us where the first kernel took 5.4)
    constexpr int kFrags = MLPD_NBF16 / 4, kInferThreads = 32 * kInferWarps;
    static_assert(kFrags % kInferThreads == 0 && MLPD_W2 / 4 % kInferThreads == 0 && MLPD_W3 / 4 % kInferThreads == 0 &&
                      MLPD_W4 / 4 % kInferThreads == 0,
                  "a pass of the threads stays in one layer");
    uint2 frag[kFrags / kInferThreads];
#pragma unroll
    for (int j = 0; j < kFrags / kInferThreads; ++j)
        frag[j] = __ldg(reinterpret_cast<const uint2*>(blob) + threadIdx.x + j * kInferThreads);
#pragma unroll
    for (int j = 0; j < kFrags / kInferThreads; ++j)
        reinterpret_cast<uint2*>(wts)[mlp_warp_order(threadIdx.x, j * kInferThreads)] = frag[j];
    for (int i = threadIdx.x; i < MLPD_NBIAS; i += 32 * kInferWarps)
        reinterpret_cast<float*>(wts + MLPD_NBF16 * 2)[i] = __ldg(reinterpret_cast<const float*>(blob + MLPD_NBF16 * 2) + i);
    __nv_bfloat16* mine = rows[w];
    for (int i = lane; i < 32 * MLP_FROW; i += 32) mine[i] = __float2bfloat16_rn(0.0f);
    __syncthreads();
    constexpr int kVecs = MLP_IN / 4;  // 16-byte vectors per row
    const int64_t ntiles = (n + 31) / 32, total = n * kVecs;
    const int64_t nw = (int64_t)gridDim.x * kInferWarps;
    const bool aligned = (reinterpret_cast<uintptr_t>(feat) & 15) == 0;
    float4 f[kVecs];
    auto fetch = [&](int64_t tile) {
#pragma unroll
        for (int j = 0; j < kVecs; ++j) {
            const int64_t i = tile * 32 * kVecs + 32 * j + lane;
            f[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (i < total) {
                const float* p = feat + 4 * i;
                f[j] = aligned ? __ldg(reinterpret_cast<const float4*>(p))
                               : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
            }
        }
    };
    int64_t tile = (int64_t)blockIdx.x * kInferWarps + w;
    fetch(tile);
    for (; tile < ntiles; tile += nw) {
        __syncwarp();  // the previous tile's fragments have been read
#pragma unroll
        for (int j = 0; j < kVecs; ++j) {
            const int i = 32 * j + lane;
            __nv_bfloat162* p = reinterpret_cast<__nv_bfloat162*>(mine + (i / kVecs) * MLP_FROW + 4 * (i % kVecs));
            p[0] = __floats2bfloat162_rn(f[j].x, f[j].y);
            p[1] = __floats2bfloat162_rn(f[j].z, f[j].w);
        }
        __syncwarp();
        fetch(tile + nw);
        float y[2][4];
        mlp_forward_frag<2, false>(mine, wts, y);
        const int gid = lane >> 2, tig = lane & 3;
        if (tig < 2) {
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int64_t r = tile * 32 + 16 * mt + gid + 8 * hh;
                    if (r < n) {
                        float* p = out + r * MLP_OUT + 2 * tig;
                        p[0] = y[mt][2 * hh];
                        p[1] = y[mt][2 * hh + 1];
                    }
                }
        }
    }
}

int mlp_step_weight_bytes() { return MLPD_BYTES + MLPT_BYTES; }

cudaError_t launch_mlp_pack_step(const float* params, unsigned char* blob, cudaStream_t s)
{
    mlp_pack_kernel<true><<<32, 256, 0, s>>>(params, blob);
    return cudaGetLastError();
}

}  // namespace lb

namespace {
bool train_configured()
{
    static bool ok = cudaFuncSetAttribute(lb::mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          lb::kTrainSmem) == cudaSuccess;
    return ok;
}

// blocks of a gradient: one per kTS samples, up to a fixed number (three for each SM of a
// GB300, which is what the shared memory holds), each then walking several tiles. Fixed,
// not asked of the device: it sets the order in which a gradient is summed, and a
// training run's bits are not to depend on where it runs.
constexpr int kTrainBlocks = 456;
int g_train_blocks(int64_t count)
{
    const int64_t b = (count + lb::kTS - 1) / lb::kTS;
    return (int)(b < 1 ? 1 : (b > kTrainBlocks ? kTrainBlocks : b));
}

// launches a kernel that, unless it is the `first` of a call, may start while its
// predecessor on the stream drains (it waits for it itself before it reads what
// that wrote; the first one's predecessor may have written the samples)
template <class... KArgs, class... Args>
cudaError_t launch_overlapped(bool first, void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t s,
                              Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = first ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// Device memory of a training or gradient call (18 MB at most) from a pool of
// this library, so that a call does not pay for cudaMalloc / cudaFree (215 us a
// call, with the device-wide wait of the free; 45 us from the pool). The pool is
// the driver's: safe with several threads and streams, it keeps at most
// kPoolKeep bytes per device between calls and returns the rest when a stream
// synchronises. A stream under capture takes the plain allocation, which CUDA
// refuses there.
constexpr uint64_t kPoolKeep = 32ull << 20;
constexpr int kPoolDevices = 32;

cudaMemPool_t workspace_pool()
{
    static std::mutex mu;
    static cudaMemPool_t pools[kPoolDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kPoolDevices) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!pools[dev]) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        uint64_t keep = kPoolKeep;
        if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) cudaGetLastError();
        pools[dev] = p;
    }
    return pools[dev];
}

struct Workspace {
    float* p = nullptr;
    cudaStream_t s = nullptr;
    bool pooled = false;
    bool alloc(size_t bytes, cudaStream_t stream)
    {
        s = stream;
        cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &st) != cudaSuccess) cudaGetLastError();
        cudaMemPool_t pool = st == cudaStreamCaptureStatusNone ? workspace_pool() : nullptr;
        if (pool) {
            if (cudaMallocFromPoolAsync((void**)&p, bytes, pool, stream) == cudaSuccess) return pooled = true;
            cudaGetLastError();
        }
        return cudaMalloc((void**)&p, bytes) == cudaSuccess;
    }
    ~Workspace()
    {
        if (p && pooled)
            cudaFreeAsync(p, s);
        else if (p)
            cudaFree(p);
    }
};

constexpr int kReduceGrid = (lb::MLP_NPARAM + 1 + 31) / 32;
}  // namespace

extern "C" {

int lbrmhd_mlp_nparams(void) { return lb::MLP_NPARAM; }

int lbrmhd_mlp_blob_bytes(void) { return lb::MLPD_BYTES; }

int lbrmhd_mlp_pack(const float* d_params, void* d_blob, void* stream)
{
    if (!d_params || !d_blob) return LBRMHD_ERR_BAD_ARG;
    lb::mlp_pack_kernel<false><<<32, 256, 0, (cudaStream_t)stream>>>(d_params, (unsigned char*)d_blob);
    return cudaGetLastError() == cudaSuccess ? LBRMHD_OK : LBRMHD_ERR_CUDA;
}

int lbrmhd_mlp_infer(const void* d_blob, const float* d_features, int64_t n, float* d_out, void* stream)
{
    if (!d_blob || !d_features || !d_out || n < 0) return LBRMHD_ERR_BAD_ARG;
    if (n == 0) return LBRMHD_OK;
    const int64_t grid = (int64_t)lb::device_sms() * lb::kInferBlocks;  // one wave
    const int64_t tiles = (n + 31) / 32, blocks = (tiles + lb::kInferWarps - 1) / lb::kInferWarps;
    lb::mlp_infer_kernel<<<(unsigned)(blocks < grid ? blocks : grid), 32 * lb::kInferWarps, 0, (cudaStream_t)stream>>>(
        (const unsigned char*)d_blob, d_features, n, d_out);
    return cudaGetLastError() == cudaSuccess ? LBRMHD_OK : LBRMHD_ERR_CUDA;
}

int lbrmhd_mlp_grad(const float* d_params, const float* d_data, int64_t n, float* d_grad, void* stream)
{
    if (!d_params || !d_data || !d_grad || n < 1) return LBRMHD_ERR_BAD_ARG;
    const int nb = g_train_blocks(n);
    cudaStream_t s = (cudaStream_t)stream;
    Workspace ws;
    if (!ws.alloc((size_t)nb * lb::kTrainStride * sizeof(float), s)) return LBRMHD_ERR_OOM;
    float* partial = ws.p;
    if (!train_configured()) return LBRMHD_ERR_CUDA;
    cudaError_t e1 = launch_overlapped(true, lb::mlp_grad_kernel, nb, lb::kTrainThreads, lb::kTrainSmem, s, d_params, d_data,
                                       n, n, 0, partial, 1.0f / (float)n);
    if (e1 == cudaSuccess)
        e1 = launch_overlapped(false, lb::mlp_reduce_kernel<false>, kReduceGrid, 32 * lb::kReduceShares, 0, s, partial, nb,
                               d_grad, nullptr, nullptr, nullptr, nullptr, lb::AdamStep{});
    const cudaError_t e2 = cudaStreamSynchronize(s);
    return (e1 == cudaSuccess && e2 == cudaSuccess) ? LBRMHD_OK : LBRMHD_ERR_CUDA;
}

int lbrmhd_mlp_train(float* d_params, float* d_adam, const float* d_data, int64_t n, int steps, int batch, float lr,
                     uint64_t seed, float* d_loss, void* stream)
{
    if (!d_params || !d_adam || !d_data || n < 1 || steps < 0 || batch < 1 || !(lr > 0)) return LBRMHD_ERR_BAD_ARG;
    const int nb = g_train_blocks(batch);
    cudaStream_t s = (cudaStream_t)stream;
    Workspace ws;
    if (!ws.alloc((size_t)nb * lb::kTrainStride * sizeof(float), s)) return LBRMHD_ERR_OOM;
    float* partial = ws.p;
    if (!train_configured()) return LBRMHD_ERR_CUDA;
    const float b1 = 0.9f, b2 = 0.999f;
    float c1 = 1.0f, c2 = 1.0f;
    cudaError_t e1 = cudaSuccess;
    for (int t = 0; t < steps && e1 == cudaSuccess; ++t) {
        c1 *= b1;
        c2 *= b2;
        e1 = launch_overlapped(t == 0, lb::mlp_grad_kernel, nb, lb::kTrainThreads, lb::kTrainSmem, s, d_params, d_data, n,
                               batch, lb::splitmix64(seed + (uint64_t)t + 1) | 1ull, partial, 1.0f / (float)batch);
        if (e1 == cudaSuccess)
            e1 = launch_overlapped(false, lb::mlp_reduce_kernel<true>, kReduceGrid, 32 * lb::kReduceShares, 0, s, partial, nb,
                                   nullptr, d_params, d_adam, d_adam + lb::MLP_NPARAM, d_loss ? d_loss + t : nullptr,
                                   lb::AdamStep{lr, b1, b2, 1e-8f, 1.0f - c1, 1.0f - c2});
    }
    const cudaError_t e2 = cudaStreamSynchronize(s);
    return (e1 == cudaSuccess && e2 == cudaSuccess) ? LBRMHD_OK : LBRMHD_ERR_CUDA;
}

}  // extern "C"
