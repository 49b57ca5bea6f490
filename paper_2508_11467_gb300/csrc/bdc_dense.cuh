// Shared by the dense front and back end's translation units: the grid
// barrier of the cooperative kernels, the Householder scalars and the panel
// launchers of bdc_reduce.cu.
#pragma once
#include "bdc_internal.cuh"

namespace bdc {

// count, gen: the reusable barrier of k_geqr2 (bdc_dense.cu);
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
constexpr int kQp = 32;            // columns of a QR panel at most: a lane each
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

// one panel of nb <= 32 columns and rows of the blocked reduction of the m x n
// matrix A: V, X at PW (m x 32 each), Y, U at QW (n x 32 each)
size_t labrd_scratch_doubles(int m, int n);
cudaError_t launch_labrd_panel(int m, int n, int nb, double *A, int lda, double *d, double *e, double *tauq,
                               double *taup, double *PW, double *QW, double *scratch, GridBar *bar, unsigned *bars,
                               cudaStream_t st);
// QR of an m x nb panel (nb <= 32) held on chip, likewise; gram[c ldg + i] =
// v_c^T v_i for c < i
bool geqr2_resident_fits(int m, int nb);
cudaError_t launch_geqr2_resident(int m, int nb, double *A, int lda, double *tau, double *gram, int ldg,
                                  double *scratch, GridBar *bar, unsigned *bars, cudaStream_t st);

// One operand of a product of split_products(): n vectors of K entries (the
// rows of A, the columns of B).  tr = 0: vector v at p + v ld, along K; tr =
// 1: entry k of vector v at p + k ld + v.  parts > 1: the sum of `parts`
// copies pstride apart.  mask: a panel of reflectors, the stored entries
// where row > reflector, 0 above: row moff + k of reflector v (mask = 1), or
// row moff + v of reflector k (mask = 2, mask = 3), the unit entry left out but
// for mask = 2.  mask = 4: entry k = v left out.
// add: add[v add_v + k add_k] is added to entry k of vector v.
struct SplitSide {
    const double *p;
    long long pstride;
    int ld, tr, n, parts, mask, moff;
    int row0;   // set by split_products
    const double *add;
    long long add_v, add_k;
};
struct SplitProd {
    SplitSide a, b;
    double *C;   // a.n x b.n, column-major
    int ldc, K, sub;   // 0: C = A B, 1: C -= A B, 2: C += A B
};
constexpr int kSplitMax = 32, kSplitMostK = 16384;
// rows of A and columns of B at most: a tile list entry holds the row block
// (of 128) in 15 bits, the column block in 16
constexpr int kSplitMostRows = 32767 * 128;
// products on the tensor cores by error-free BF16 slices (bdc_gemm_mixed.cu),
// at most kSplitMax in one launch set, K up to kSplitMostK and a.n, b.n up to
// kSplitMostRows (cudaErrorInvalidValue beyond); scratch of split_scratch(sum of a.n,
// sum of b.n, largest K, sum of ceil(a.n/128) ceil(b.n/128)) bytes; *err
// (device) is set when a bounded wait gave up.  The products of a launch set
// have results of their own; chained = 1: two products of one shape
// subtracted from one C, each at a scale of its own.
size_t split_scratch(long long rowsA, long long colsB, int K, long long tiles);
cudaError_t split_products(SplitProd *prods, int count, void *scratch, size_t bytes, int *err, cudaStream_t st,
                           int chained = 0);

}  // namespace bdc
