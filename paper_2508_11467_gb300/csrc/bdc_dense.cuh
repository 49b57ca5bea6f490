// Shared by the dense front and back end's translation units: the grid
// barrier of the cooperative kernels, the Householder scalars and the panel
// launchers of bdc_reduce.cu.
#pragma once
#include "bdc_internal.cuh"

namespace bdc {

// count, gen: the reusable barrier of k_geqr2 and k_labrd (bdc_dense.cu);
// mono: the monotonic arrival counter of the kernels of bdc_reduce.cu; err:
// set by the barrier wait that gave up (all CTAs leave at their next barrier)
struct GridBar {
    unsigned count, gen, mono;
    int err;
};
constexpr unsigned long long kBarNs = 2000000000ull;

__device__ __forceinline__ unsigned long long gtime() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// CTAs of the resident kernels at most (their exchange buffers are sized by it)
constexpr int kResGrid = 160;
// scratch doubles of the resident reduction of an m x n matrix (any m >= n
// that resident_fits() accepts)
size_t resident_scratch_doubles(int n);
// whether the m x n matrix fits the shared memory of the device's SMs as one
// block of rows per CTA
bool resident_fits(int m, int n);
// bidiagonalization of the m x n matrix A (m >= n, lda) held on chip; bars:
// running arrival count of bar->mono over the launches of one call
cudaError_t launch_gebd2_resident(int m, int n, double *A, int lda, double *d, double *e, double *tauq, double *taup,
                                  double *scratch, GridBar *bar, unsigned *bars, cudaStream_t st);

}  // namespace bdc
