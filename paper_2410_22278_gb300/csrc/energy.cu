// E_J = 1/2 sum D o J and E_K = -1/4 sum D o K of matrices on the device
// (jk_energy): one launch, the sums written straight into pinned host memory.
//
// The reduction reads 3 n^2 doubles (16.6 MB for the 64-water box: 2.5 us at
// the copy rate, from L2 when a build has just written them); what a call
// took was everything around it -- a stream-ordered allocation and free, a
// memset, a copy into pageable memory and 2432 blocks adding to two addresses
// (201 us a call, 20 of them the kernel).
#include <cuda_runtime.h>

#include <algorithm>

#include "plan.h"

namespace jk {
namespace {

// two blocks per SM cover the load latency; each block's partial is added by
// the last block to finish, in block order, so the result is reproducible
constexpr int kEnergyGrid = 304, kEnergyBlock = 512;

__device__ __forceinline__ void block_sum2(double &a, double &b, double (*sh)[2])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sh[threadIdx.x >> 5][0] = a;
        sh[threadIdx.x >> 5][1] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a = b = 0.0;
        for (int w = 0; w < kEnergyBlock / 32; ++w) {
            a += sh[w][0];
            b += sh[w][1];
        }
    }
}

// part: gridDim.x pairs, then the counter of finished blocks (zero between
// launches).  vec: all pointers are 16-byte aligned.
__global__ void __launch_bounds__(kEnergyBlock) k_energy(size_t n2, const double *__restrict__ D, const double *__restrict__ J,
                                                         const double *__restrict__ K, int vec, double *part, double *out)
{
    __shared__ double sh[kEnergyBlock / 32][2];
    __shared__ int last;
    const size_t t = blockIdx.x * (size_t)kEnergyBlock + threadIdx.x, step = (size_t)gridDim.x * kEnergyBlock;
    double a = 0.0, b = 0.0;
    if (vec) {
        const double2 *D2 = reinterpret_cast<const double2 *>(D), *J2 = reinterpret_cast<const double2 *>(J),
                      *K2 = reinterpret_cast<const double2 *>(K);
#pragma unroll 4
        for (size_t i = t; i < n2 / 2; i += step) {
            const double2 d = __ldg(D2 + i);
            if (J) {
                const double2 x = __ldg(J2 + i);
                a = fma(d.x, x.x, fma(d.y, x.y, a));
            }
            if (K) {
                const double2 x = __ldg(K2 + i);
                b = fma(d.x, x.x, fma(d.y, x.y, b));
            }
        }
        if (t == 0 && (n2 & 1)) {
            if (J) a = fma(D[n2 - 1], J[n2 - 1], a);
            if (K) b = fma(D[n2 - 1], K[n2 - 1], b);
        }
    } else {
        for (size_t i = t; i < n2; i += step) {
            const double d = __ldg(D + i);
            if (J) a = fma(d, __ldg(J + i), a);
            if (K) b = fma(d, __ldg(K + i), b);
        }
    }
    block_sum2(a, b, sh);
    unsigned *done = reinterpret_cast<unsigned *>(part + 2 * kEnergyGrid);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = a;
        part[2 * blockIdx.x + 1] = b;
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    a = b = 0.0;
    for (unsigned i = threadIdx.x; i < gridDim.x; i += kEnergyBlock) {
        a += __ldcg(part + 2 * i);
        b += __ldcg(part + 2 * i + 1);
    }
    block_sum2(a, b, sh);
    if (threadIdx.x == 0) {
        *done = 0u;
        out[0] = a;
        out[1] = b;
        __threadfence_system();
    }
}

int make_slot(EnergySlot &s, cudaStream_t st)
{
    const size_t bytes = (2 * kEnergyGrid + 1) * sizeof(double);
    if (cudaMalloc((void **)&s.part, bytes) != cudaSuccess) return fail_cuda(JK_ERR_OOM, "energy scratch");
    if (cudaMemsetAsync(s.part, 0, bytes, st) != cudaSuccess || cudaHostAlloc((void **)&s.host, 2 * sizeof(double), cudaHostAllocMapped) != cudaSuccess) {
        cudaFree(s.part);
        return fail_cuda(JK_ERR_OOM, "energy scratch");
    }
    return JK_OK;
}

}  // namespace

// one slot with the plan, so that the first call allocates nothing
int energy_reserve(Plan *P)
{
    EnergySlot s;
    const int rc = make_slot(s, 0);
    if (rc == JK_OK) P->energy_free.push_back(s);
    return rc;
}

void energy_release(Plan *P)
{
    for (auto *slots : {&P->energy_free, &P->energy_lost}) {
        for (auto &s : *slots) {
            cudaFree(s.part);
            cudaFreeHost(s.host);
        }
        slots->clear();
    }
}

int energy(Plan *P, const double *D, const double *J, const double *K, double *e_coul, double *e_exch, cudaStream_t st)
{
    EnergySlot s;
    {
        std::lock_guard<std::mutex> g(P->energy_mu);
        if (!P->energy_free.empty()) {
            s = P->energy_free.back();
            P->energy_free.pop_back();
        }
    }
    if (!s.part) {
        const int rc = make_slot(s, st);
        if (rc) return rc;
    }
    const size_t n2 = (size_t)P->nbf * P->nbf;
    const int vec = (((uintptr_t)D | (uintptr_t)J | (uintptr_t)K) & 15) == 0;
    const unsigned grid = (unsigned)std::min<size_t>((n2 + 2 * kEnergyBlock - 1) / (2 * kEnergyBlock), kEnergyGrid);
    // The launch is judged by its own status, not by an error that an earlier
    // call left in this thread, and the stream is waited for whatever it says:
    // the kernel reads the caller's matrices and owns the slot until it ends.
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kEnergyBlock);
    cfg.stream = st;
    const cudaError_t launched = cudaLaunchKernelEx(&cfg, k_energy, n2, D, J, K, vec, s.part, s.host);
    const cudaError_t done = cudaStreamSynchronize(st);
    const bool ok = launched == cudaSuccess && done == cudaSuccess;
    if (ok) {
        *e_coul = 0.5 * s.host[0];
        *e_exch = -0.25 * s.host[1];
    }
    {
        std::lock_guard<std::mutex> g(P->energy_mu);
        (ok ? P->energy_free : P->energy_lost).push_back(s);
    }
    return ok ? JK_OK : fail_cuda(JK_ERR_CUDA, "energy reduction failed");
}

}  // namespace jk
