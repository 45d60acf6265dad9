// CIC variant and adjoint kernels, both precisions.
#include "pm_launch.h"
#include "pm_cic.cuh"
PM_CIC_INSTANTIATE(float)
PM_CIC_INSTANTIATE(double)
cudaError_t pm_launch_cic_slots(long long *a, long long *b, long long n, cudaStream_t st) { return cic_slots(a, b, n, st); }
