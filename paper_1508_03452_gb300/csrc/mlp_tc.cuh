// mlp_tc.cuh -- forward pass of the learned seed's network on the fifth-generation
// tensor cores: 128 rows (one per thread of a 128-thread block) at a time.
//
// Activations never leave the tensor memory and the registers: a thread owns row t
// of the tile in both (lane t of the tensor memory). Its bf16 inputs are stored to
// the operand columns, one thread issues the layer's products (operand A in tensor
// memory, the weights in shared memory, float32 sums in tensor memory), and every
// thread reads its row of sums back, applies the ReLU and stores the next operand; the
// biases start the sums, as products of constant inputs. What bounds it: the chain of
// four layers (store, products, commit, load: ~700 clocks each), so several blocks share
// an SM; the products themselves are a sixth of what mma.sync takes (one 128 x 64 x 16
// product in ~34 clocks against 128 mma.sync of 16).
#pragma once

#include "mlp.cuh"
#include "tma.cuh"

namespace lb {

constexpr int kTcRows = 128;    // rows of a tile, threads of its block
constexpr int kTcCols = 128;    // tensor-memory columns of a block: 64 sums, 40 operand, rounded to a power of two
constexpr int kTcOperand = 64;  // first operand column: 32 of activations, 8 of the constant inputs

// Weights as the tensor core reads them from shared memory (K-major, no swizzle):
// core matrices of 8 output rows x 8 inputs (8 rows of 16 bytes), those of a row
// group side by side along K (128 bytes apart), row groups K * 16 bytes apart. The first
// 16 inputs of a layer are the constants 1, 1, 1, 0, ..., whose weights add up to its
// bias: their product starts the sums, as the bias starts those of the mma.sync form,
// and the two forms' sums agree bit for bit (with the bias after the inputs, or added
// to the outputs, a hidden unit's bf16 rounding could fall otherwise, and with it
// the seed of a run depended on the launch schedule). The output layer is padded to 16
// rows (the smallest N of a 128-row product).
constexpr int MLPT_KB = 16;  // inputs of the bias
constexpr int MLPT_K1 = MLPT_KB + MLP_K1, MLPT_K = MLPT_KB + MLP_H;
constexpr int MLPT_W1 = 0, MLPT_W2 = MLPT_W1 + MLP_H * MLPT_K1, MLPT_W3 = MLPT_W2 + MLP_H * MLPT_K,
              MLPT_W4 = MLPT_W3 + MLP_H * MLPT_K, MLPT_BYTES = 2 * (MLPT_W4 + 16 * MLPT_K);
static_assert(MLPT_BYTES % 16 == 0, "one bulk copy");

// element of weight (r, k) of a layer with K inputs, from the layer's start
__host__ __device__ constexpr int mlpt_index(int r, int k, int K)
{
    return (r / 8) * (K * 8) + (k / 8) * 64 + (r % 8) * 8 + k % 8;
}

// the bias inputs' weights of layer l (0..3), output r: three bf16 values, each
// what the one before leaves of b, cut off, so that they add up to b exactly (an
// infinity or NaN as the first alone)
__device__ __forceinline__ void mlpt_put_bias(__nv_bfloat16* W, int l, int r, float b)
{
    const int K = l == 0 ? MLPT_K1 : MLPT_K;
    __nv_bfloat16* w = W + (l == 0 ? MLPT_W1 : (l == 1 ? MLPT_W2 : (l == 2 ? MLPT_W3 : MLPT_W4)));
    float rest = b;
#pragma unroll
    for (int j = 0; j < MLPT_KB; ++j) {
        const float v = isfinite(rest) ? __uint_as_float(__float_as_uint(rest) & 0xffff0000u) : rest;
        w[mlpt_index(r, j, K)] = __float2bfloat16_rn(j < 3 ? v : 0.0f);
        rest = isfinite(rest) ? rest - v : 0.0f;
    }
}

// --- tensor memory ----------------------------------------------------------
// (.sync.aligned: the whole warp, converged)
__device__ __forceinline__ void tc_alloc(uint32_t* addr_sh)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(addr_sh)),
                 "r"(kTcCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc(uint32_t addr)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(kTcCols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 words of this thread's lane to 16 columns
__device__ __forceinline__ void tc_st16(uint32_t addr, const uint32_t* v)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            addr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tc_st8(uint32_t addr, uint32_t v0, uint32_t v1, uint32_t rest)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%3,%3,%3,%3,%3};" ::"r"(addr), "r"(v0), "r"(v1),
                 "r"(rest)
                 : "memory");
}
__device__ __forceinline__ void tc_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 32 (4) columns of this thread's lane
__device__ __forceinline__ void tc_ld32(uint32_t addr, float (&v)[32])
{
    uint32_t u[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
        "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
          "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), "=r"(u[16]),
          "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), "=r"(u[24]),
          "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
        : "r"(addr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(u[i]);
}
__device__ __forceinline__ void tc_ld4(uint32_t addr, float (&v)[4])
{
    uint32_t u[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3])
                 : "r"(addr)
                 : "memory");
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(u[i]);
}

// products of a layer: D (float32, 128 x N) = A (bf16, tensor memory, 128 x K) W^T,
// then the commit that arrives on *bar (one thread)
// (K with the bias inputs, which lie behind the activations in the operand)
template <int K, int N>
__device__ __forceinline__ void tc_layer(uint32_t tmem, uint32_t w_smem, uint64_t* bar)
{
    // instruction: float32 sums, bf16 operands, both K-major, N / 8, M / 16
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N / 8) << 17) | ((uint32_t)(kTcRows / 16) << 24);
    // shared-memory matrix: start, K step and row-group step in 16-byte units, version 1, no swizzle
    constexpr uint64_t steps = ((uint64_t)(128 / 16) << 16) | ((uint64_t)(K * 16 / 16) << 32) | (1ull << 46);
#pragma unroll
    for (int k = 0; k < K / 16; ++k) {
        const uint64_t desc = steps | (uint64_t)(((w_smem + 256u * k) & 0x3ffffu) >> 4);
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem),
            "r"(tmem + kTcOperand + (k == 0 ? MLP_H / 2 : 8 * (k - 1))), "l"(desc), "r"(idesc), "r"(k)
            : "memory");
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    uint32_t u;
    memcpy(&u, &v, 4);
    return u;
}
__device__ __forceinline__ uint32_t pack_relu_bf16(float a, float b)  // (a in the low half; -0 and NaN as max(., 0) gives them)
{
    const __nv_bfloat162 v = __hmax2(__floats2bfloat162_rn(a, b), __floats2bfloat162_rn(0.0f, 0.0f));
    uint32_t u;
    memcpy(&u, &v, 4);
    return u;
}

constexpr uint32_t kTcOnes = 0x3f803f80u, kTcOne = 0x00003f80u;  // bf16 pairs (1, 1) and (1, 0)

// the bias inputs (once per block, all of its threads)
__device__ __forceinline__ void mlp_tc_constants(uint32_t tmem, int tid)
{
    tc_st8(tmem + ((uint32_t)(tid & ~31) << 16) + kTcOperand + MLP_H / 2, kTcOnes, kTcOne, 0u);
}

// a wait of the tensor core's own products, a few polls before the bounded one reads the clock
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity)
{
#pragma unroll 1
    for (int i = 0; i < 32; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_bounded(bar, parity);
}

// The network on the block's 128 rows: x[10] this thread's 20 features as bf16 pairs,
// y its outputs; mlp_tc_constants has been called. `w`: the weights in shared memory (MLPT_ order,
// visible to the asynchronous proxy); tmem: the block's kTcCols columns; *bar: an
// mbarrier of count 1 whose next phase has parity *phase; ok: whether the thread's
// inputs have arrived. All 128 threads call it; false (for all of them) if an input
// had not, or the products did not complete within the wait limit.
__device__ __forceinline__ bool mlp_forward_tc(const uint32_t (&x)[MLP_IN / 2], const unsigned char* w, uint32_t tmem,
                                               uint64_t* bar, uint32_t& phase, int tid, float (&y)[4], bool ok)
{
    const uint32_t mine = tmem + ((uint32_t)(tid & ~31) << 16);  // this warp's lanes
    const uint32_t ws = smem_u32(w);
    {
        uint32_t a[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) a[j] = j < MLP_IN / 2 ? x[j] : 0u;
        tc_st16(mine + kTcOperand, a);
    }
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        tc_st_wait();
        tc_fence_before();
        ok = __syncthreads_and(ok);
        if (!ok) return false;
        if (tid == 0) {
            tc_fence_after();
            if (l == 0)
                tc_layer<MLPT_K1, MLP_H>(tmem, ws + 2 * MLPT_W1, bar);
            else if (l == 1)
                tc_layer<MLPT_K, MLP_H>(tmem, ws + 2 * MLPT_W2, bar);
            else if (l == 2)
                tc_layer<MLPT_K, MLP_H>(tmem, ws + 2 * MLPT_W3, bar);
            else
                tc_layer<MLPT_K, 16>(tmem, ws + 2 * MLPT_W4, bar);
        }
        ok = tc_wait(bar, phase);
        phase ^= 1u;
        __syncwarp();
        tc_fence_after();
        if (l == 3) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[32];
            tc_ld32(mine + 32 * h, v);
            uint32_t a[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) a[j] = pack_relu_bf16(v[2 * j], v[2 * j + 1]);
            tc_st16(mine + kTcOperand + 16 * h, a);
        }
    }
    tc_ld4(mine, y);
    tc_fence_before();
    return __syncthreads_and(ok);  // every row has been read: the columns are free again
}

// A block's use of the network: tc_open takes its tensor memory and starts the copy of
// the weights (all threads; a block barrier in it), tc_run takes the thread's row
// through the network and gives the tensor memory back (all threads, once; false for
// all of them if a wait ran out).
struct TcCtx {
    const unsigned char* w;  // weights in shared memory, arriving on bar[0]
    uint64_t* bar;           // [0] the weights, [1] the products
    uint32_t tmem;           // the block's columns
};
constexpr size_t kTcSmem = MLPT_BYTES + 3 * sizeof(uint64_t);  // weights, barriers, the columns' address

__device__ __forceinline__ TcCtx tc_open(unsigned char* smem, const unsigned char* weights, int tid)
{
    TcCtx tm;
    tm.w = smem;
    tm.bar = reinterpret_cast<uint64_t*>(smem + MLPT_BYTES);
    uint32_t* tmem_sh = reinterpret_cast<uint32_t*>(tm.bar + 2);
    if (tid == 0) {
        mbar_init(&tm.bar[0], 1u);
        mbar_init(&tm.bar[1], 1u);
        mbar_init_fence();
        mbar_arrive_expect_tx(&tm.bar[0], MLPT_BYTES);
        bulk_load(smem, weights, MLPT_BYTES, &tm.bar[0]);
    }
    if (tid < 32) tc_alloc(tmem_sh);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    tm.tmem = *tmem_sh;
    mlp_tc_constants(tm.tmem, tid);
    return tm;
}

__device__ __forceinline__ bool tc_run(const TcCtx& tm, const float (&feat)[MLP_IN], int tid, float (&y)[MLP_OUT])
{
    uint32_t xb[MLP_IN / 2];
#pragma unroll
    for (int j = 0; j < MLP_IN / 2; ++j) xb[j] = pack_bf16(feat[2 * j], feat[2 * j + 1]);
    const bool in = mbar_wait_bounded(&tm.bar[0], 0u);
    __syncwarp();
    uint32_t phase = 0;
    const bool got = mlp_forward_tc(xb, tm.w, tm.tmem, &tm.bar[1], phase, tid, y, in);
    if (!got) {
        // a wait ran out: wait again, with a limit, for the copy and the products issued
        // last, which must not outlive the block's memory (before the first products
        // the parity is that of the barrier's past phase, and the wait returns at once)
        mbar_wait_bounded(&tm.bar[0], 0u);
        mbar_wait_bounded(&tm.bar[1], phase ^ 1u);
        __syncwarp();
    }
    if (tid < 32) tc_dealloc(tm.tmem);
    return got;
}

}  // namespace lb
