// Device functions of the library's headers behind plain C entries, for tests that
// compare them on their own (tests/device_checks.py builds this file).
#include "lattice.cuh"
#include "mlp_tc.cuh"

namespace {

// 128 rows a block through the tensor-memory network, as the one-run step kernel takes
// its cells; rows past the end repeat the last one and are not stored
__global__ void __launch_bounds__(lb::kTcRows) seed_kernel(const unsigned char* w, const float* feat, int64_t n, float* out,
                                                           int* failed)
{
    __shared__ __align__(16) unsigned char sm[lb::kTcSmem];
    const int tid = threadIdx.x;
    const lb::TcCtx tm = lb::tc_open(sm, w, tid);
    const int64_t row = blockIdx.x * (int64_t)lb::kTcRows + tid, r = row < n ? row : n - 1;
    float x[lb::MLP_IN], y[lb::MLP_OUT];
#pragma unroll
    for (int j = 0; j < lb::MLP_IN; ++j) x[j] = feat[r * lb::MLP_IN + j];
    if (!lb::tc_run(tm, x, tid, y)) {
        if (tid == 0) atomicAdd(failed, 1);
        return;
    }
    if (row < n)
#pragma unroll
        for (int j = 0; j < lb::MLP_OUT; ++j) out[row * lb::MLP_OUT + j] = y[j];
}

// the same with weights that never arrive: the barrier expects their bytes, no copy is
// started, and the block's waits run out; out counts the threads that were told so
__global__ void __launch_bounds__(lb::kTcRows) late_seed_kernel(int* told)
{
    __shared__ __align__(16) unsigned char sm[lb::kTcSmem];
    const int tid = threadIdx.x;
    lb::TcCtx tm;
    tm.w = sm;
    tm.bar = reinterpret_cast<uint64_t*>(sm + lb::MLPT_BYTES);
    uint32_t* columns = reinterpret_cast<uint32_t*>(tm.bar + 2);
    if (tid == 0) {
        lb::mbar_init(&tm.bar[0], 1u);
        lb::mbar_init(&tm.bar[1], 1u);
        lb::mbar_init_fence();
        lb::mbar_arrive_expect_tx(&tm.bar[0], lb::MLPT_BYTES);
    }
    if (tid < 32) lb::tc_alloc(columns);
    lb::tc_fence_before();
    __syncthreads();
    lb::tc_fence_after();
    tm.tmem = *columns;
    lb::mlp_tc_constants(tm.tmem, tid);
    const float x[lb::MLP_IN] = {};
    float y[lb::MLP_OUT];
    if (!lb::tc_run(tm, x, tid, y)) atomicAdd(told, 1);
}

__global__ void reciprocal_kernel(const double* x, int64_t n, double* rcp, double* rsqrt)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    rcp[i] = lb::rcp_approx(x[i]);
    rsqrt[i] = lb::rsqrt_newton(x[i]);
}

}  // namespace

// the float64 reciprocals of n values; 0, or -1 on a CUDA error
extern "C" int check_reciprocals(const double* d_x, int64_t n, double* d_rcp, double* d_rsqrt)
{
    if (n < 1) return -1;
    reciprocal_kernel<<<(unsigned)((n + 127) / 128), 128>>>(d_x, n, d_rcp, d_rsqrt);
    return cudaGetLastError() == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess ? 0 : -1;
}

// threads of one block that were told that the weights did not arrive (128 expected)
extern "C" int check_late_seed()
{
    int *d_told = nullptr, told = -1;
    if (cudaMalloc((void**)&d_told, sizeof(int)) != cudaSuccess) return -1;
    if (cudaMemset(d_told, 0, sizeof(int)) == cudaSuccess) {
        late_seed_kernel<<<1, lb::kTcRows>>>(d_told);
        if (cudaGetLastError() != cudaSuccess || cudaMemcpy(&told, d_told, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
            told = -1;
    }
    cudaFree(d_told);
    return told;
}

// blocks whose waits ran out (0 expected), or -1 on a CUDA error
extern "C" int check_seed(const float* d_params, const float* d_feat, int64_t n, float* d_out)
{
    unsigned char* w = nullptr;
    int* d_failed = nullptr;
    int failed = -1;
    if (n < 1 || cudaMalloc((void**)&w, lb::mlp_step_weight_bytes()) != cudaSuccess) return -1;
    if (cudaMalloc((void**)&d_failed, sizeof(int)) == cudaSuccess && cudaMemset(d_failed, 0, sizeof(int)) == cudaSuccess &&
        lb::launch_mlp_pack_step(d_params, w, nullptr) == cudaSuccess) {
        seed_kernel<<<(unsigned)((n + lb::kTcRows - 1) / lb::kTcRows), lb::kTcRows>>>(w + lb::MLPD_BYTES, d_feat, n, d_out,
                                                                                      d_failed);
        if (cudaGetLastError() != cudaSuccess || cudaMemcpy(&failed, d_failed, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
            failed = -1;
    }
    cudaFree(d_failed);
    cudaFree(w);
    return failed;
}
