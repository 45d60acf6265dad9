// Self-tests.  Square roots: the FP64 roots of pm_roots.cuh on the caller's
// arguments.  Failure detection: one block waits, with the bounded wait the
// FFT passes use for their tensor copies (%globaltimer, 2 s), on an
// mbarrier that nothing ever arrives at.  The wait gives up, the block
// records the error in the flag the passes use, and the host reads it as it
// reads an expired wait of a pass.  No fault, trap or unbounded wait.
#include "pm_launch.h"
#include "pm_passes.cuh"
#include "pm_roots.cuh"

namespace {

__global__ void k_wait_expiry(int *err) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        pmk::mbar_init(&bar, 1);   // one arrival expected; none comes
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0 && !pmk::mbar_wait(&bar, 0)) atomicExch(err, 1);
}

__global__ void k_roots(const double *r, long long n, double *inv_sqrt, double *root, double *inv) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        inv_sqrt[i] = pmroot::inv_sqrt(r[i], (float)r[i]);
        pmroot::root_inv(r[i], root[i], inv[i]);
    }
}

}  // namespace

cudaError_t pm_launch_roots(const double *r, long long n, double *inv_sqrt, double *root, double *inv, cudaStream_t st) {
    if (n > 0) k_roots<<<256, 256, 0, st>>>(r, n, inv_sqrt, root, inv);
    return cudaGetLastError();
}

cudaError_t pm_launch_wait_expiry(int *err, cudaStream_t st) {
    k_wait_expiry<<<1, 32, 0, st>>>(err);
    return cudaGetLastError();
}
