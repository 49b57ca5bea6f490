// Dense front and back end of the SVD (FP64), all on the GPU:
//
//   Sec. 4.1, Algorithm 1  bidiagonalization A = Q1 B P1^T (m >= n) by blocks
//             of b columns and rows: one cooperative panel kernel (k_labrd_panel, bdc_reduce.cu)
//             forms the b column reflectors H_i, row reflectors G_i and the
//             vectors y_i, x_i of Eqs. (bidiag-y-k3) and (bidiag-x-k3), the
//             corrections of the not yet updated trailing matrix merged into
//             one pair of matrices P = [V X], Q = [Y U]; the trailing matrix
//             then takes the merged rank-(2b) update A -= P Q^T of Eq.
//             (bidiag-A-trail3): ONE product in FP64, the halves V Y^T and
//             X U^T at a scale of their own when sliced.
//   Sec. 4.3  QR of a tall-and-skinny A (cooperative panel k_geqr2 plus a
//             block-reflector update of the trailing columns), the explicit Q
//             (Eq. orgqr-q), and the back-transformations U = Q1 U2 and
//             V^T = V2^T P1^T.  A block reflector I - Y T Y^T is applied with
//             T formed explicitly from the modified compact-WY relation of
//             Eqs. (inv_t, larft_update), T^{-1} = the upper part of Y^T Y with
//             the diagonal 1 / tau: products only, no solve per column.
//
// Products: from 64 reflectors on (and for the trailing updates) error-free
// BF16 slices on the tcgen05 tensor cores (split_products, bdc_gemm_mixed.cu:
// 56 bits below each row's maximum), smaller ones FP64 mma.sync.m8n8k4
// (k_dgemm: C = alpha op(A) op(B) + beta C with either operand transposed).
// mma.sync FP64 runs at 1.67 multiply-adds a clock and SM on GB300 (measured,
// any shape and occupancy; the plain FMA 1.9), so the FP64 products were
// most of a large SVD: back-transformation of 4096 x 4096, one side, 181 ms
// (165 ms without the triangular solves) -> 10.5 ms; trailing updates of its
// reduction about 85 -> 25 ms; 333 x 333, one side, 2.4 -> 0.64 ms.  Error
// against twice the precision, FP64 products and blocks of 64 -> these: explicit
// Q of 257 x 257, 1000 x 1000, 10000 x 300 6.3e-16, 6.7e-16, 1.5e-16 -> 6.0e-16,
// 4.1e-16, 1.1e-16; Q C of a Gaussian C 9.4e-16, 9.7e-16, 2.6e-16 -> 6.2e-16,
// 4.6e-16, 1.0e-16; backward error of geqrf 6.8e-16, 7.2e-16, 2.9e-16 -> 6.2e-16,
// 4.6e-16, 2.7e-16; U^T U - I of gesvd 333, 2000 5.3e-14, 4.0e-13 -> 4.8e-14,
// 4.0e-13.  (Q C of an identity, whose ones scale the slices of C's first rows:
// 6.3e-16, 6.7e-16, 1.5e-16 -> 6.7e-16, 5.3e-16, 3.5e-16.)
//
// The panel
// kernels run as cooperative launches (all CTAs resident) and separate their
// phases with a grid barrier whose wait is bounded (2 s of %globaltimer): a
// barrier that gives up sets an error word, every CTA leaves at its next
// barrier, and the entry point reports BDC_ERR_TIMEOUT (the products' bounded
// waits set the same word; the entry points without a status fill their
// result with NaN then).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "bdc_dense.cuh"

namespace bdc {

namespace {

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// ------------------------------------------------------------------ GEMM
struct DGemm {
    const double *A, *B;
    double *C;
    int lda, ldb, ldc, M, N, K;
    int ta, tb;            // op(A) = A^T, op(B) = B^T
    double alpha, beta;    // beta = 0: C is not read
    int kchunk;            // split K: CTA row blockIdx.y multiplies K range [y kchunk, (y+1) kchunk)
    double *part;          // split K: partial products part[y][M x N] (then alpha, beta unused)
};

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
                 : "+d"(c[0]), "+d"(c[1])
                 : "d"(a), "d"(b));
}

// Four warps of 32 x 32 (4 x 4 fragments 8 x 8), K step 16, operands staged
// k-major in padded shared tiles, next step prefetched.  CTA tile 64 x 64, or
// 32 x 128 for products of at most 32 rows (the QR panels' Y^T C), where the
// lower half of a 64 x 64 tile would leave two SM sub-partitions idle.
constexpr int DBK = 16, DSB = DBK + 4;
template <int DBM, int DBN>
__global__ void __launch_bounds__(128) k_dgemm(DGemm g) {
    pdl_begin();
    constexpr int DSA = DBM + 8, WN = DBN / 32;
    static_assert(DBM / 32 * WN == 4, "four warps");
    __shared__ double As[DBK * DSA];   // As[k][m]
    __shared__ double Bs[DBN * DSB];   // Bs[n][k]
    const int tilesN = (g.N + DBN - 1) / DBN;
    const int m0 = (blockIdx.x / tilesN) * DBM, n0 = (blockIdx.x % tilesN) * DBN;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = (warp / WN) * 32, wn = (warp % WN) * 32;
    const int gr = lane >> 2, tg = lane & 3;
    double acc[4][4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
    constexpr int LA = DBM * DBK / 128, LB = DBN * DBK / 128;   // elements per thread per operand
    double ra[LA], rb[LB];
    auto load = [&](int k0) {
#pragma unroll
        for (int r = 0; r < LA; ++r) {
            const int idx = tid + r * 128;
            int am, ak;
            if (!g.ta) { am = idx % DBM; ak = idx / DBM; } else { ak = idx % DBK; am = idx / DBK; }
            const int gm = m0 + am, gk = k0 + ak;
            ra[r] = (gm < g.M && gk < g.K) ? (g.ta ? g.A[(size_t)gm * g.lda + gk] : g.A[(size_t)gk * g.lda + gm])
                                           : 0.0;
        }
#pragma unroll
        for (int r = 0; r < LB; ++r) {
            const int idx = tid + r * 128;
            int bk, bn;
            if (!g.tb) { bk = idx % DBK; bn = idx / DBK; } else { bn = idx % DBN; bk = idx / DBN; }
            const int gn = n0 + bn, gk2 = k0 + bk;
            rb[r] = (gn < g.N && gk2 < g.K) ? (g.tb ? g.B[(size_t)gk2 * g.ldb + gn] : g.B[(size_t)gn * g.ldb + gk2])
                                            : 0.0;
        }
    };
    auto store = [&]() {
#pragma unroll
        for (int r = 0; r < LA; ++r) {
            const int idx = tid + r * 128;
            int am, ak;
            if (!g.ta) { am = idx % DBM; ak = idx / DBM; } else { ak = idx % DBK; am = idx / DBK; }
            As[ak * DSA + am] = ra[r];
        }
#pragma unroll
        for (int r = 0; r < LB; ++r) {
            const int idx = tid + r * 128;
            int bk, bn;
            if (!g.tb) { bk = idx % DBK; bn = idx / DBK; } else { bn = idx % DBN; bk = idx / DBN; }
            Bs[bn * DSB + bk] = rb[r];
        }
    };
    // K range of this CTA (all of K unless split)
    const int kb = g.part ? (int)blockIdx.y * g.kchunk : 0;
    const int ke = g.part ? min(g.K, kb + g.kchunk) : g.K;
    // operand loads are bounded by the K range end
    const int Kfull = g.K;
    g.K = ke;
    load(kb);
    for (int k0 = kb; k0 < ke; k0 += DBK) {
        __syncthreads();
        store();
        __syncthreads();
        if (k0 + DBK < ke) load(k0 + DBK);
#pragma unroll
        for (int kk = 0; kk < DBK; kk += 4) {
            if (k0 + kk >= ke) break;
            double af[4], bf[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) af[i] = As[(kk + tg) * DSA + wm + i * 8 + gr];
#pragma unroll
            for (int j = 0; j < 4; ++j) bf[j] = Bs[(wn + j * 8 + gr) * DSB + kk + tg];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (m0 + wm + i * 8 < g.M && n0 + wn + j * 8 < g.N) dmma(acc[i][j], af[i], bf[j]);
        }
    }
    (void)Kfull;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int gm = m0 + wm + i * 8 + gr;
        if (gm >= g.M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int gn = n0 + wn + j * 8 + 2 * tg + h;
                if (gn >= g.N) continue;
                if (g.part) {
                    g.part[((size_t)blockIdx.y * g.N + gn) * g.M + gm] = acc[i][j][h];
                    continue;
                }
                double *c = g.C + (size_t)gn * g.ldc + gm;
                const double v = g.alpha * acc[i][j][h];
                *c = (g.beta == 0.0) ? v : fma(g.beta, *c, v);
            }
        }
    }
}

// scratch for split-K partial products (set per call sequence by the driver)
thread_local double *g_split_buf = nullptr;
thread_local size_t g_split_cap = 0;   // doubles

int sm_count_dense() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    }
    return n;
}

cudaError_t dgemm_launch(const DGemm &g, int splits, cudaStream_t st) {
    if (g.M <= 32) {
        const long long tiles = (long long)((g.M + 31) / 32) * ((g.N + 127) / 128);
        if (tiles > 0x7fffffffll) return cudaErrorInvalidValue;
        launch_pdl(k_dgemm<32, 128>, dim3((unsigned)tiles, (unsigned)splits), 128, 0, st, g);
    } else {
        const long long tiles = (long long)((g.M + 63) / 64) * ((g.N + 63) / 64);
        if (tiles > 0x7fffffffll) return cudaErrorInvalidValue;
        launch_pdl(k_dgemm<64, 64>, dim3((unsigned)tiles, (unsigned)splits), 128, 0, st, g);
    }
    return cudaGetLastError();
}

// C = alpha op(A) op(B) + beta C
cudaError_t dgemm(int ta, int tb, int M, int N, int K, double alpha, const double *A, int lda, const double *B,
                  int ldb, double beta, double *C, int ldc, cudaStream_t st) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    return dgemm_launch(DGemm{A, B, C, lda, ldb, ldc, M, N, std::max(K, 0), ta, tb, alpha, beta, 0, nullptr}, 1, st);
}

// op(A) op(B) as `splits` partial products over ranges of K, part y at
// g_split_buf + y M N (column-major M x N): the products with few output
// tiles and a long K (Y^T C and C Y of the block reflectors) then use the
// whole GPU.  The split count fills whole rounds of two CTAs per SM (the
// FP64 tensor pipe is full with one warp per sub-partition, so a round's time
// does not depend on how full it is) and keeps at least 64 of K per part.
cudaError_t dgemm_parts(int ta, int tb, int M, int N, int K, const double *A, int lda, const double *B, int ldb,
                        int &splits, cudaStream_t st) {
    const long long tiles = M <= 32 ? (long long)((N + 127) / 128) : (long long)((M + 63) / 64) * ((N + 63) / 64);
    const long long sms = sm_count_dense();
    const long long cap = std::max<long long>(1, (long long)(g_split_cap / ((size_t)M * N)));
    const long long most = std::max<long long>(1, std::min<long long>({cap, 64, K / 64}));
    // the split with the least work on the fullest SM, the smallest within 3 %
    splits = 1;
    double best = 0.0;
    for (long long s = 1; s <= most; ++s) {
        const double c = (double)((tiles * s + sms - 1) / sms) / (double)s;
        if (s == 1 || c < 0.97 * best) {
            best = c;
            splits = (int)s;
        }
    }
    DGemm g{A, B, nullptr, lda, ldb, 0, M, N, K, ta, tb, 1.0, 0.0, 0, g_split_buf};
    g.kchunk = ((K + splits - 1) / splits + DBK - 1) / DBK * DBK;
    splits = (K + g.kchunk - 1) / g.kchunk;
    return dgemm_launch(g, splits, st);
}

// ------------------------------------------------------------ grid barrier
// all CTAs of a cooperative launch; false (and the error word set) when the
// wait gave up or another CTA gave up before
__device__ bool grid_sync(GridBar *gb) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile GridBar *v = gb;
        int ok = v->err == 0;
        if (ok) {
            const unsigned g0 = v->gen;
            __threadfence();
            const unsigned arrived = atomicAdd(&gb->count, 1u);
            if (arrived == gridDim.x - 1) {
                gb->count = 0;
                __threadfence();
                atomicAdd(&gb->gen, 1u);
            } else {
                const unsigned long long t0 = gtime();
                while (v->gen == g0) {
                    if (v->err) { ok = 0; break; }
                    if (gtime() - t0 > kBarNs) {
                        atomicExch(&gb->err, 1);
                        ok = 0;
                        break;
                    }
                }
            }
            __threadfence();
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// block sum of a double over blockDim.x threads (result in every thread)
__device__ double block_sum(double v, double *sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double r = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) r += sh[k];
    return r;
}

// sum over the grid's CTAs of part[k * stride] (k < count), by the whole
// block: strided loads, four in flight per thread, then a block reduction
__device__ double grid_partials(const double *part, int count, int stride, double *sh) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    const int T = blockDim.x;
    int k = threadIdx.x;
    for (; k + 3 * T < count; k += 4 * T) {
        s0 += part[(size_t)k * stride];
        s1 += part[(size_t)(k + T) * stride];
        s2 += part[(size_t)(k + 2 * T) * stride];
        s3 += part[(size_t)(k + 3 * T) * stride];
    }
    for (; k < count; k += T) s0 += part[(size_t)k * stride];
    return block_sum((s0 + s1) + (s2 + s3), sh);
}

// Householder reflector from alpha and ||x_2..||^2 = sig2 (LAPACK's sign
// convention, Sec. 4.1's first display): beta = -sign(alpha) ||x||, tau =
// (beta - alpha) / beta, the vector's tail scaled by 1 / (alpha - beta);
// sig2 = 0 gives tau = 0 (H = I).  Returns the tail scale.
__device__ __forceinline__ double reflector(double alpha, double sig2, double &tau, double &beta) {
    if (sig2 == 0.0) {
        tau = 0.0;
        beta = alpha;
        return 0.0;
    }
    const double nrm = sqrt(fma(alpha, alpha, sig2));
    beta = alpha >= 0.0 ? -nrm : nrm;
    tau = (beta - alpha) / beta;
    return 1.0 / (alpha - beta);
}

// ---------------------------------------------------------- QR panel
// geqr2 on the local m x nb panel A (Sec. 4.3, step 1): column reflectors
// with the panel's later columns updated after each one.  part[grid][b]:
// partial products v^T A[:, c] per CTA.
struct Geqr2Args {
    double *A;
    int lda, m, nb, b;
    double *tau;
    double *part;
    GridBar *bar;
};

__global__ void __launch_bounds__(256) k_geqr2(Geqr2Args a) {
    __shared__ double sh[32];
    __shared__ double sw[64];
    const int T = blockDim.x, G = gridDim.x;
    const int gtid = blockIdx.x * T + threadIdx.x, gthreads = G * T;
    const int m = a.m, nb = a.nb, b = a.b;
    double *A = a.A;
    const long long lda = a.lda;
    for (int i = 0; i < nb; ++i) {
        double ss = 0.0;
        for (int r = i + 1 + gtid; r < m; r += gthreads) ss = fma(A[(size_t)i * lda + r], A[(size_t)i * lda + r], ss);
        ss = block_sum(ss, sh);
        if (threadIdx.x == 0) a.part[(size_t)blockIdx.x * (b + 1) + b] = ss;
        if (!grid_sync(a.bar)) return;
        double sig2 = grid_partials(a.part + b, G, b + 1, sh);
        const double alpha = A[(size_t)i * lda + i];
        double tau, beta;
        const double sc = reflector(alpha, sig2, tau, beta);
        // w_c = v^T A[i:, c] for every later panel column at once, from the
        // column before scaling (v_r = sc A[r, i] for r > i, v_i = 1; the
        // scaled v is written in the update phase, after the barrier, so no
        // CTA reads a row another one is scaling): each warp sums its rows for
        // column c = i + 1 + lane (lanes over columns, the warp's rows in
        // turn), then the warps' sums are added in shared memory in a fixed
        // order
        {
            __shared__ double wsum[8][33];
            const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
            const int c = i + 1 + lane;
            double acc = 0.0;
            if (c < nb) {
                for (int r = i + 1 + blockIdx.x * nwarp + wid; r < m; r += G * nwarp)
                    acc = fma(A[(size_t)i * lda + r], A[(size_t)c * lda + r], acc);
                acc *= sc;
                if (gtid < 32) acc += A[(size_t)c * lda + i];           // v_i = 1 at row i (one warp of CTA 0)
            }
            if (wid < 8) wsum[wid][lane] = acc;
            __syncthreads();
            if (threadIdx.x < 32) {
                double t = 0.0;
                for (int q = 0; q < nwarp && q < 8; ++q) t += wsum[q][threadIdx.x];
                if (i + 1 + (int)threadIdx.x < nb) a.part[(size_t)blockIdx.x * (b + 1) + i + 1 + threadIdx.x] = t;
            }
        }
        if (gtid == 0) a.tau[i] = tau;
        if (!grid_sync(a.bar)) return;
        // A[i:, c] -= tau v w_c, w_c summed over the CTAs: thread t takes
        // column offset t % 32 and every eighth CTA from t / 32
        {
            __shared__ double red[8][33];
            const int co = threadIdx.x & 31, kk = threadIdx.x >> 5, c = i + 1 + co;
            double w = 0.0;
            if (c < nb && kk < 8)
                for (int k = kk; k < G; k += 8) w += a.part[(size_t)k * (b + 1) + c];
            if (kk < 8) red[kk][co] = w;
            __syncthreads();
            if (threadIdx.x < 32) {
                double t = 0.0;
                for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
                sw[threadIdx.x] = tau * t;
            }
            __syncthreads();
        }
        for (int r = i + gtid; r < m; r += gthreads) {
            double v = 1.0;
            if (r > i) {
                v = A[(size_t)i * lda + r] * sc;        // the reflector's entry, stored scaled
                A[(size_t)i * lda + r] = v;
            }
            for (int c = i + 1; c < nb; ++c) A[(size_t)c * lda + r] -= v * sw[c - i - 1];
        }
        if (gtid == 0) A[(size_t)i * lda + i] = beta;
        if (!grid_sync(a.bar)) return;
    }
}

// ------------------------------------------------ block reflector helpers
// Y (rows x nb, ld rows) from the stored reflectors: column j is zero above
// row j + off, 1 at row j + off, then the stored entries src[j * ldsrc + r]
// (column reflectors: off = 0, src = A's panel; row reflectors: the entries
// of row j of A's panel, read with ldsrc = 1 and stride lda, off = 0 on the
// shifted rows).
__global__ void k_form_y(double *Y, int rows, int nb, const double *src, long long sr, long long sc) {
    pdl_begin();
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)rows * nb) return;
    const int j = (int)(k / rows), r = (int)(k % rows);
    Y[k] = (r < j) ? 0.0 : (r == j) ? 1.0 : src[(size_t)j * sc + (size_t)r * sr];
}

// ---- T of the compact WY form I - Y T Y^T = H_1 ... H_nb, for every block
// of kTB reflectors of a call at once.  T^{-1} is the strictly upper part of
// Y^T Y plus the diagonal 1 / tau (Eqs. inv_t, larft_update); it is inverted
// here once (zero row and column where tau = 0), so that applying a block is
// two products and a small one with T instead of a triangular solve per right
// hand side (one thread each, 64 x 64 / 2 dependent FMAs: 4096 x 4096, one
// side, 181 ms of which the solves were about 130).
constexpr int kTB = 64;

// the reflectors of a call: block j holds kTB of them from reflector i0 = j
// kTB, entry r of reflector i0 + c at src + i0 (sr + sc) + r sr + c sc for r
// > c (1 at r = c, 0 above), rows - i0 entries long
struct Reflectors {
    const double *src;
    long long sr, sc;
    int rows, count;
};

// partial Y^T Y of block blockIdx.x over the rows of chunk blockIdx.y
__global__ void __launch_bounds__(128) k_gram(Reflectors f, int kchunk, double *part) {
    pdl_begin();
    constexpr int LD = kTB + 4;
    __shared__ double Ys[16 * LD];   // [row][reflector]
    const int i0 = blockIdx.x * kTB, nb = min(kTB, f.count - i0), rows = f.rows - i0;
    const double *src = f.src + (size_t)i0 * (f.sr + f.sc);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32, gr = lane >> 2, tg = lane & 3;
    const int kb = blockIdx.y * kchunk, ke = min(rows, kb + kchunk);
    double acc[4][4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
    for (int k0 = kb; k0 < ke; k0 += 16) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 16 * kTB / 128; ++q) {
            const int idx = tid + q * 128;
            int r, c;   // the contiguous index fastest
            if (f.sr == 1) { r = idx % 16; c = idx / 16; } else { c = idx % kTB; r = idx / kTB; }
            const int gk = k0 + r;
            double v = 0.0;
            if (gk < ke && c < nb && gk >= c) v = (gk == c) ? 1.0 : src[(size_t)gk * f.sr + (size_t)c * f.sc];
            Ys[r * LD + c] = v;
        }
        __syncthreads();
        if (wm > wn || wn >= nb) continue;   // below the diagonal, past the reflectors
#pragma unroll
        for (int kk = 0; kk < 16; kk += 4) {
            double af[4], bf[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                af[i] = Ys[(kk + tg) * LD + wm + i * 8 + gr];
                bf[i] = Ys[(kk + tg) * LD + wn + i * 8 + gr];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dmma(acc[i][j], af[i], bf[j]);
        }
    }
    double *out = part + ((size_t)blockIdx.x * gridDim.y + blockIdx.y) * kTB * kTB;
    if (wm <= wn)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    out[(size_t)(wm + i * 8 + gr) * kTB + wn + j * 8 + 2 * tg + h] = acc[i][j][h];
}

// C (rm x cn, row stride ldc) = sgn A (rm x kn) B (kn x cn) in shared memory, 8 x 8 fragments over the CTA's warps
__device__ __forceinline__ void smem_mm(double *C, int ldc, const double *A, int lda, const double *B, int ldb, int rm,
                                        int cn, int kn, double sgn) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int gr = lane >> 2, tg = lane & 3;
    const int tn = cn / 8, tiles = rm / 8 * tn;
    for (int q = warp; q < tiles; q += nw) {
        const int r0 = q / tn * 8, c0 = q % tn * 8;
        double acc[2] = {0.0, 0.0};
        for (int k = 0; k < kn; k += 4) dmma(acc, A[(r0 + gr) * lda + k + tg], B[(k + tg) * ldb + c0 + gr]);
        C[(r0 + gr) * ldc + c0 + 2 * tg] = sgn * acc[0];
        C[(r0 + gr) * ldc + c0 + 2 * tg + 1] = sgn * acc[1];
    }
}

// T (kTB x kTB, row-major, zero below the diagonal and beyond the block's
// reflectors) of block blockIdx.x: the 16 x 16 diagonal blocks by the column
// recursion T(:, j) = -tau_j T G(:, j), a warp each; then pairs of blocks by
// T_12 = -T_11 G_12 T_22.  Block x is sub-block x % per of group x / per:
// its G and T lie at group (x / per) gstride + (x % per) kTB (ld + 1), row
// stride ld; G is the sum of `chunks` copies cstride apart.
constexpr int kTLd = kTB + 4;
struct TForm {
    const double *G;
    double *T;
    const double *tau;
    int ld, per, chunks, count;
    long long gstride_g, gstride_t, cstride;
};
constexpr int kPair = 2;   // sets of reflectors (Q1 and P1) served by one launch
struct TForms {
    TForm f[kPair];
};
__global__ void __launch_bounds__(256) k_tform(const __grid_constant__ TForms fs) {
    pdl_begin();
    const TForm &f = fs.f[blockIdx.y];
    if ((int)blockIdx.x * kTB >= f.count) return;
    extern __shared__ double tsm[];
    double *Gs = tsm, *Ts = tsm + kTB * kTLd, *Xs = Ts + kTB * kTLd;   // G, T, 32 x 32 product
    const int i0 = blockIdx.x * kTB, nb = min(kTB, f.count - i0);
    const int sub = blockIdx.x % f.per, grp = blockIdx.x / f.per;
    const double *p = f.G + grp * f.gstride_g + (long long)sub * kTB * (f.ld + 1);
    const double *tau = f.tau;
    double *Tall = f.T + grp * f.gstride_t + (long long)sub * kTB * (f.ld + 1);
    for (int k = threadIdx.x; k < kTB * kTB; k += blockDim.x) {
        const int r = k / kTB, c = k % kTB;
        double s = 0.0;
        if (r < c && c < nb)
#pragma unroll 8
            for (int y = 0; y < f.chunks; ++y) s += p[y * f.cstride + (long long)r * f.ld + c];
        Gs[r * kTLd + c] = s;
        Ts[r * kTLd + c] = 0.0;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < kTB / 16) {
        const int o = warp * 16;
        for (int j = 0; j < 16; ++j) {
            const double tj = (o + j < nb) ? tau[i0 + o + j] : 0.0;
            double s = 0.0;
            if (lane < j)
                for (int k = lane; k < j; ++k) s = fma(Ts[(o + lane) * kTLd + o + k], Gs[(o + k) * kTLd + o + j], s);
            if (lane <= j) Ts[(o + lane) * kTLd + o + j] = (lane == j) ? tj : -tj * s;
            __syncwarp();
        }
    }
    __syncthreads();
    for (int h = 16; h < kTB && h < nb; h *= 2)
        for (int o = 0; o < kTB; o += 2 * h) {
            smem_mm(Xs, kTLd, Gs + o * kTLd + o + h, kTLd, Ts + (o + h) * kTLd + o + h, kTLd, h, h, h, 1.0);
            __syncthreads();
            smem_mm(Ts + o * kTLd + o + h, kTLd, Ts + o * kTLd + o, kTLd, Xs, kTLd, h, h, h, -1.0);
            __syncthreads();
        }
    for (int k = threadIdx.x; k < kTB * kTB; k += blockDim.x)
        Tall[(long long)(k / kTB) * f.ld + k % kTB] = Ts[(k / kTB) * kTLd + k % kTB];
}
constexpr size_t kTformSmem = sizeof(double) * (2 * kTB + 32) * kTLd;
cudaError_t launch_tform(const TForm *f, int jobs, int blocks, cudaStream_t st) {
    TForms fs{};
    for (int q = 0; q < jobs; ++q) fs.f[q] = f[q];
    cudaError_t e =
        cudaFuncSetAttribute(k_tform, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTformSmem);
    if (e != cudaSuccess) return e;
    launch_pdl(k_tform, dim3(blocks, jobs), 256, kTformSmem, st, fs);
    return cudaGetLastError();
}

// T of every block of the reflectors into Tall (blocks x kTB x kTB)
cudaError_t form_t(const Reflectors &f, const double *tau, double *Tall, cudaStream_t st) {
    if (f.count <= 0) return cudaSuccess;
    const int blocks = (f.count + kTB - 1) / kTB;
    // chunks of at least 256 rows, about four CTAs per SM over all blocks
    const long long cap = (long long)(g_split_cap / ((size_t)blocks * kTB * kTB));
    long long chunks = std::min<long long>((f.rows + 255) / 256, std::max(1, 4 * sm_count_dense() / blocks));
    chunks = std::max<long long>(1, std::min(chunks, cap));
    if (cap < 1) return cudaErrorInvalidValue;
    int kchunk = (int)((f.rows + chunks - 1) / chunks + 15) / 16 * 16;
    chunks = (f.rows + kchunk - 1) / kchunk;
    launch_pdl(k_gram, dim3(blocks, (unsigned)chunks), 128, 0, st, f, kchunk, g_split_buf);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const TForm tf{g_split_buf, Tall, tau, kTB, 1, (int)chunks, f.count, (long long)chunks * kTB * kTB,
                   (long long)kTB * kTB, (long long)kTB * kTB};
    return launch_tform(&tf, 1, blocks, st);
}

// W = M Z for the summed partial products Z of dgemm_parts, M = T or T^T
// (tr), nb x nb.  left: Z is nb x count (column-major), a vector per column;
// right: Z is count x nb, a vector per row (W^T = M Z^T).  V = 16 vectors per
// CTA, 8 while that leaves SMs without one (the sums of the partial products
// take most of it: 480 vectors of 31 parts 46 us with 16, 28 with 8); each warp
// takes 8 rows of M, its fragments straight from L2.  add: Z += the first nb
// rows of add (left; the unit entries' share).
template <int V>
__global__ void __launch_bounds__(256) k_tz(const double *__restrict__ T, int nb, int tr, const double *__restrict__ part,
                                            int splits, int right, int count, double *__restrict__ W,
                                            const double *__restrict__ add, int ldadd) {
    pdl_begin();
    constexpr int LD = V + 4;
    __shared__ double Zs[kTB * LD];   // [k][vector]
    const int v0 = blockIdx.x * V;
    const size_t mn = (size_t)nb * count;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gr = lane >> 2, tg = lane & 3;
    const int i0 = warp * 8;
    double mf[kTB / 4];
#pragma unroll
    for (int k = 0; k < kTB / 4; ++k) {
        const int i = i0 + gr, j = 4 * k + tg;
        mf[k] = T[tr ? j * kTB + i : i * kTB + j];
    }
    for (int k = threadIdx.x; k < kTB * V; k += blockDim.x) {
        int p, v;
        if (right) { v = k % V; p = k / V; } else { p = k % kTB; v = k / kTB; }
        double s = 0.0;
        if (p < nb && v0 + v < count) {
            const double *q = part + (right ? (size_t)p * count + v0 + v : (size_t)(v0 + v) * nb + p);
#pragma unroll 16
            for (int y = 0; y < splits; ++y) s += q[(size_t)y * mn];
            if (add) s += add[(size_t)(v0 + v) * ldadd + p];
        }
        Zs[p * LD + v] = s;
    }
    __syncthreads();
    if (i0 >= nb) return;
    double acc[V / 8][2];
#pragma unroll
    for (int j = 0; j < V / 8; ++j) acc[j][0] = acc[j][1] = 0.0;
#pragma unroll
    for (int k = 0; k < kTB / 4; ++k) {
        // M is triangular: T has only k >= i, T^T only k <= i
        if (tr ? 4 * k > i0 + 7 : 4 * k + 3 < i0) continue;
#pragma unroll
        for (int j = 0; j < V / 8; ++j) dmma(acc[j], mf[k], Zs[(4 * k + tg) * LD + j * 8 + gr]);
    }
#pragma unroll
    for (int j = 0; j < V / 8; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int v = v0 + j * 8 + 2 * tg + h, i = i0 + gr;
            if (i < nb && v < count) W[right ? (size_t)i * count + v : (size_t)v * nb + i] = acc[j][h];
        }
}

template <typename... Args>
void launch_tz(int count, cudaStream_t st, Args... args) {
    if (count <= 8 * sm_count_dense()) launch_pdl(k_tz<8>, (count + 7) / 8, 256, 0, st, args...);
    else launch_pdl(k_tz<16>, (count + 15) / 16, 256, 0, st, args...);
}

// C (rows x cols, ldc) := H C or H^T C (left) or C H or C H^T (right), H =
// I - Y T Y^T = H_1 ... H_nb for the explicit Y (left: rows x nb; right:
// cols x nb) and its T: Z = Y^T C (or C Y) in partial products, W = T Z or
// T^T Z (or Z T, Z T^T), C -= Y W (or W Y^T).
cudaError_t apply_block(int left, int trans, int rows, int cols, const double *Y, int nb, const double *T, double *C,
                        int ldc, double *W, cudaStream_t st) {
    if (rows <= 0 || cols <= 0 || nb <= 0) return cudaSuccess;
    cudaError_t e;
    int splits;
    if (left) {
        if ((e = dgemm_parts(1, 0, nb, cols, rows, Y, rows, C, ldc, splits, st)) != cudaSuccess) return e;
        launch_tz(cols, st, T, nb, trans ? 1 : 0, g_split_buf, splits, 0, cols, W, nullptr, 0);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        return dgemm(0, 0, rows, cols, nb, -1.0, Y, rows, W, nb, 1.0, C, ldc, st);
    }
    if ((e = dgemm_parts(0, 0, rows, nb, cols, C, ldc, Y, cols, splits, st)) != cudaSuccess) return e;
    launch_tz(rows, st, T, nb, trans ? 0 : 1, g_split_buf, splits, 1, rows, W, nullptr, 0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return dgemm(0, 1, rows, cols, nb, -1.0, W, rows, Y, cols, 1.0, C, ldc, st);
}

// ---- blocks of kWide reflectors on the split-BF16 products (split_products):
// V = Y T is formed for every block of a call at once (Y read in place from
// the panel through the slicing's mask), then per block Z = Y^T C (partial
// products over K) and C -= V Z.
constexpr int kWide = 256;
// partial products of a block's Y^T Y: rows of each, and how many (eight at most)
int gram_chunk(int rows) { return std::max(512, ((rows + 7) / 8 + 31) / 32 * 32); }
int gram_chunks(int rows) { return (rows + gram_chunk(rows) - 1) / gram_chunk(rows); }

// G = Y^T Y above the diagonal from the partial products of Y without its unit
// entries (symmetric): entry (r, c), r < c, adds reflector r's row c times
// reflector c's unit entry.  T zeroed.
struct GramSum {
    const double *part;
    Reflectors f;
    int chunk, chunks;
    double *G, *T;
};
struct GramSums {
    GramSum g[kPair];
};
__global__ void k_gram_sum(const __grid_constant__ GramSums gs) {
    pdl_begin();
    const GramSum &a = gs.g[blockIdx.z];
    const Reflectors &f = a.f;
    const size_t w2 = (size_t)kWide * kWide;
    const int k = blockIdx.x * blockDim.x + threadIdx.x, r = k / kWide, c = k % kWide;
    const int i0 = blockIdx.y * kWide, nb = min(kWide, f.count - i0);
    if (nb <= 0) return;
    const double *p = a.part + (size_t)blockIdx.y * a.chunks * w2 + k;
    double s = 0.0;
    if (r < c && c < nb) {
        const int own = (f.rows - i0 + a.chunk - 1) / a.chunk;   // this block's partial products
#pragma unroll 4
        for (int y = 0; y < own; ++y) s += p[(size_t)y * w2];
        s += f.src[(size_t)i0 * (f.sr + f.sc) + (size_t)c * f.sr + (size_t)r * f.sc];
    }
    a.G[blockIdx.y * w2 + k] = s;
    a.T[blockIdx.y * w2 + k] = 0.0;
}

// the off-diagonal blocks of T from its h x h diagonal blocks, one 8 x 8
// fragment per warp, operands from L2: phase 0: X = G_12 T_22, phase 1: T_12 =
// -T_11 X (row-major, kWide x kWide per block; a fragment's K range skips the
// zero half of the triangular factor).  The products cancel, and the rounding
// of one long sum was most of the error of an explicit Q of about kWide
// reflectors: sums of 8 terms, four of them as a tree, then those in turn
// (explicit Q of 257 x 257 against twice the precision: one sum 9.6e-16, so
// 5.8e-16, blocks of 64 in FP64 6.3e-16).
struct TMerge {
    const double *G[kPair];
    double *T[kPair], *X[kPair];
    int blocks[kPair];
};
__global__ void __launch_bounds__(128) k_tmerge(const __grid_constant__ TMerge a, int h, int phase) {
    pdl_begin();
    if ((int)blockIdx.y >= a.blocks[blockIdx.z]) return;
    const size_t w2 = (size_t)kWide * kWide;
    const double *g = a.G[blockIdx.z] + blockIdx.y * w2;
    double *t = a.T[blockIdx.z] + blockIdx.y * w2, *x = a.X[blockIdx.z] + blockIdx.y * w2;
    const int lane = threadIdx.x & 31, gr = lane >> 2, tg = lane & 3;
    const int per = (h / 8) * (h / 8);
    const int q = blockIdx.x * 4 + (threadIdx.x >> 5);
    const int o = q / per * 2 * h, r0 = q % per / (h / 8) * 8, c0 = q % per % (h / 8) * 8;
    if (o + 2 * h > kWide) return;
    const double *A = phase == 0 ? g + (size_t)o * kWide + o + h : t + (size_t)o * kWide + o;
    const double *B = phase == 0 ? t + (size_t)(o + h) * kWide + o + h : x + (size_t)o * kWide + o + h;
    double acc[2] = {0.0, 0.0};
    const int kb = phase == 0 ? 0 : r0, ke = phase == 0 ? c0 + 8 : h;   // (multiples of 8)
    for (int k0 = kb; k0 < ke; k0 += 32) {
        double a[8], b[8], c[4][2];
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int k = k0 + 4 * s + tg;
            a[s] = k < ke ? A[(size_t)(r0 + gr) * kWide + k] : 0.0;
            b[s] = k < ke ? B[(size_t)k * kWide + c0 + gr] : 0.0;
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            c[s][0] = c[s][1] = 0.0;
            if (k0 + 8 * s >= ke) continue;
            dmma(c[s], a[2 * s], b[2 * s]);
            dmma(c[s], a[2 * s + 1], b[2 * s + 1]);
        }
        acc[0] += (c[0][0] + c[1][0]) + (c[2][0] + c[3][0]);
        acc[1] += (c[0][1] + c[1][1]) + (c[2][1] + c[3][1]);
    }
    double *out = (phase == 0 ? x : t) + (size_t)(o + r0 + gr) * kWide + o + h + c0 + 2 * tg;
    out[0] = phase == 0 ? acc[0] : -acc[0];
    out[1] = phase == 0 ? acc[1] : -acc[1];
}

// workspace of the split path: G, T, X (blocks x kWide^2), V (rows x count,
// also the partial Y^T Y before it), Z parts, slices
struct SplitWs {
    double *G, *T, *X, *V, *Z;
    size_t zcap;       // doubles at Z
    char *slices;
    size_t slice_bytes;
    int *err;
};

// op(Y) sides of a block (reflectors i0 .. i0 + nb - 1 of f, rows k0 ..).  The
// vectors leave out the unit entry: it would be the maximum that scales the
// slices of a reflector whose other entries are about 1 / sqrt(rows), and its
// product is the row of C itself, added in FP64 (I - Q^T Q of 1000 x 1000:
// 4.0e-14 by FP64 products, 5.3e-14 with the unit entry sliced).
SplitSide y_vectors(const Reflectors &f, int i0, int nb, int k0) {   // a vector per reflector, K = rows
    const double *p = f.src + (size_t)i0 * (f.sr + f.sc) + (size_t)k0 * f.sr;
    return f.sr == 1 ? SplitSide{p, 0, (int)f.sc, 0, nb, 1, 1, k0, 0} : SplitSide{p, 0, (int)f.sr, 1, nb, 1, 1, k0, 0};
}
SplitSide y_rows(const Reflectors &f, int i0, int rows, int mask) {  // a vector per row, K = reflectors
    const double *p = f.src + (size_t)i0 * (f.sr + f.sc);
    return f.sr == 1 ? SplitSide{p, 0, (int)f.sc, 1, rows, 1, mask, 0, 0} : SplitSide{p, 0, (int)f.sr, 0, rows, 1, mask, 0, 0};
}

// runs products in sets that fit kSplitMax and the slice scratch
struct SplitSet {
    const SplitWs &w;
    cudaStream_t st;
    std::vector<SplitProd> v;
    long long rows = 0, cols = 0, tiles = 0;
    int kmax = 0;
    cudaError_t add(const SplitProd &p) {
        auto need = [&](long long r, long long c, int k, long long t) { return split_scratch(r, c, k, t); };
        const long long t = (long long)((p.a.n + 127) / 128) * ((p.b.n + 127) / 128);
        const int k = std::max(kmax, p.K);
        if (!v.empty() && ((int)v.size() == kSplitMax || need(rows + p.a.n, cols + p.b.n, k, tiles + t) > w.slice_bytes)) {
            if (cudaError_t e = run()) return e;
        }
        v.push_back(p);
        rows += p.a.n; cols += p.b.n; tiles += t;
        kmax = std::max(kmax, p.K);
        return cudaSuccess;
    }
    cudaError_t run() {
        cudaError_t e = split_products(v.data(), (int)v.size(), w.slices, w.slice_bytes, w.err, st);
        v.clear();
        rows = cols = tiles = 0;
        kmax = 0;
        return e;
    }
};

// A set of reflectors to apply: left: C := Q C (C f.rows x other), right: C
// := C P^T (other x f.rows; C's first column is the reflectors' first row),
// with workspace of its own (slices and the error word may be shared).
struct WideJob {
    Reflectors f;
    const double *tau;
    int left, other;
    double *C;
    int ldc;
    SplitWs w;
    int blocks() const { return (f.count + kWide - 1) / kWide; }
};

// V = Y T but for the products with T's entries above the diagonal (of Y
// without its unit entries): tau_c y_rc below the diagonal, T_rc from Y's unit
// entry on and above it
struct VStart {
    Reflectors f;
    const double *T, *tau;
    double *V;
};
struct VStarts {
    VStart v[kPair];
};
__global__ void k_v_start(const __grid_constant__ VStarts vs) {
    pdl_begin();
    const VStart &a = vs.v[blockIdx.z];
    const Reflectors &f = a.f;
    const int j = blockIdx.y, i0 = j * kWide, rows = f.rows - i0, k = blockIdx.x * blockDim.x + threadIdx.x;
    if (i0 >= f.count) return;
    const int c = k / rows, r = k - c * rows;
    if (c >= min(kWide, f.count - i0)) return;
    const double *src = f.src + (size_t)i0 * (f.sr + f.sc);
    a.V[(size_t)(i0 + c) * f.rows + r] = r > c ? a.tau[i0 + c] * src[(size_t)r * f.sr + (size_t)c * f.sc]
                                               : a.T[((size_t)j * kWide + r) * kWide + c];
}

// V = Y T of every kWide block of the jobs' reflectors (row-major T): V of
// block j at w.V + i0 f.rows, column-major, f.rows - i0 rows, leading
// dimension f.rows.  T's diagonal and Y's unit entries are about sqrt(rows)
// times the others and would set their scale in the slices: their share is
// formed in FP64 (k_v_start).  (Explicit Q of 10000 x 300, error against
// twice the precision: FP64 products 1.5e-16, all of T sliced 5.0e-16.)
cudaError_t form_v(const WideJob *jobs, int njobs, cudaStream_t st) {
    const size_t w2 = (size_t)kWide * kWide;
    cudaError_t e;
    SplitSet set{jobs[0].w, st};
    GramSums gs{};
    TForm tf[kPair];
    TMerge tm{};
    int most = 0, count = 0;
    for (int q = 0; q < njobs; ++q) {
        const Reflectors &f = jobs[q].f;
        const SplitWs &w = jobs[q].w;
        const int blocks = jobs[q].blocks();
        // (a block below the first has as many chunks or fewer)
        const int chunk = gram_chunk(f.rows), chunks = gram_chunks(f.rows);
        for (int j = 0; j < blocks; ++j) {
            const int i0 = j * kWide, nb = std::min(kWide, f.count - i0), rows = f.rows - i0;
            for (int y = 0, k0 = 0; k0 < rows; ++y, k0 += chunk) {
                SplitProd p{};
                p.a = p.b = y_vectors(f, i0, nb, k0);
                p.C = w.V + ((size_t)j * chunks + y) * w2;
                p.ldc = kWide;
                p.K = std::min(chunk, rows - k0);
                if ((e = set.add(p)) != cudaSuccess) return e;
            }
        }
        gs.g[q] = GramSum{w.V, f, chunk, chunks, w.G, w.T};
        tf[q] = TForm{w.G, w.T, jobs[q].tau, kWide, kWide / kTB, 1, f.count, (long long)w2, (long long)w2, 0};
        tm.G[q] = w.G; tm.T[q] = w.T; tm.X[q] = w.X; tm.blocks[q] = blocks;
        most = std::max(most, blocks);
        count = std::max(count, f.count);
    }
    if ((e = set.run()) != cudaSuccess) return e;
    launch_pdl(k_gram_sum, dim3((unsigned)(w2 / 256), most, njobs), 256, 0, st, gs);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_tform(tf, njobs, (count + kTB - 1) / kTB, st)) != cudaSuccess) return e;
    for (int h = kTB; h < kWide && h < count; h *= 2)
        for (int phase = 0; phase < 2; ++phase) {
            const int tiles = kWide / (2 * h) * (h / 8) * (h / 8);
            launch_pdl(k_tmerge, dim3((tiles + 3) / 4, most, njobs), 128, 0, st, tm, h, phase);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    VStarts vs{};
    int rmost = 0;
    for (int q = 0; q < njobs; ++q) {
        vs.v[q] = VStart{jobs[q].f, jobs[q].w.T, jobs[q].tau, jobs[q].w.V};
        rmost = std::max(rmost, jobs[q].f.rows);
    }
    launch_pdl(k_v_start, dim3(rmost * (kWide / 256), most, njobs), 256, 0, st, vs);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int q = 0; q < njobs; ++q)
        for (int j = 0; j < jobs[q].blocks(); ++j) {
            const Reflectors &f = jobs[q].f;
            const int i0 = j * kWide, nb = std::min(kWide, f.count - i0);
            SplitProd p{};
            p.a = y_rows(f, i0, f.rows - i0, 3);
            p.b = SplitSide{jobs[q].w.T + j * w2, 0, kWide, 1, nb, 1, 4, 0, 0};
            p.sub = 2;
            p.C = jobs[q].w.V + (size_t)i0 * f.rows;
            p.ldc = f.rows;
            p.K = nb;
            if ((e = set.add(p)) != cudaSuccess) return e;
        }
    return set.run();
}

// One block of a job on ns rows or columns of C from s0: C := (I - V Y^T) C
// (left) or C (I - Y V^T) (right).  yk(k0): the block's reflectors as K-along
// vectors from row k0.
struct WideStep {
    int left, rows, nb, np, kc, ns;   // rows of the block's reflectors; np products of kc rows each
    double *c;
    int ldc;
    const double *V;
    int ldv;
    double *Z;
    void cut(int parts) {             // K = rows in `parts` products at most
        np = std::max({1, (rows + kSplitMostK - 1) / kSplitMostK, std::min(parts, rows / 256)});
        kc = ((rows + np - 1) / np + 31) / 32 * 32;
        np = (rows + kc - 1) / kc;
    }
    int tiles() const { return (nb + 127) / 128 * ((ns + 127) / 128); }
    template <typename YK>
    cudaError_t products(YK yk, SplitSet &set) const {
        for (int y = 0; y < np; ++y) {
            SplitProd p{};
            p.K = std::min(kc, rows - y * kc);
            p.C = Z + (long long)y * nb * ns;
            if (left) {        // Z (nb x ns) = Y^T C
                p.a = yk(y * kc);
                p.b = SplitSide{c + y * kc, 0, ldc, 0, ns, 1, 0, 0, 0};
                p.ldc = nb;
            } else {           // Z (ns x nb) = C Y
                p.a = SplitSide{c + (size_t)y * kc * ldc, 0, ldc, 1, ns, 1, 0, 0, 0};
                p.b = yk(y * kc);
                p.ldc = ns;
            }
            if (cudaError_t e = set.add(p)) return e;
        }
        return cudaSuccess;
    }
    cudaError_t update(SplitSet &set) const {
        const long long zs = (long long)nb * ns;
        SplitProd p{};
        p.K = nb;
        p.C = c;
        p.ldc = ldc;
        p.sub = 1;
        if (left) {            // C -= V Z
            p.a = SplitSide{V, 0, ldv, 1, rows, 1, 0, 0, 0};
            p.b = SplitSide{Z, zs, nb, 0, ns, np, 0, 0, 0, c, ldc, 1};   // + C's first nb rows
        } else {               // C -= Z V^T
            p.a = SplitSide{Z, zs, ns, 1, ns, np, 0, 0, 0, c, 1, ldc};   // + C's first nb columns
            p.b = SplitSide{V, 0, ldv, 1, rows, 1, 0, 0, 0};
        }
        return set.add(p);
    }
};

// the step of the whole untouched dimension; its block's C starts at c
WideStep wide_step(int left, int rows, int other, int nb, const double *V, int ldv, double *c, int ldc,
                   const SplitWs &w) {
    return WideStep{left, rows, nb, 1, 0, other, c, ldc, V, ldv, w.Z};
}

// products along K of a block applied alone: a wave of tiles or so
void cut_alone(WideStep &x) { x.cut(std::min(kSplitMax, 152 / std::max(x.tiles(), 1))); }
// slice scratch of the step's products and of its update
size_t step_slices(const WideStep &x) {
    const long long nt = (x.ns + 127) / 128, t = nt * ((x.rows + 127) / 128);
    return std::max({split_scratch((long long)x.np * x.nb, (long long)x.np * x.ns, x.kc, (long long)x.np * x.tiles()),
                     split_scratch(x.ns, x.rows, x.nb, t), split_scratch(x.rows, x.ns, x.nb, t)});
}

// one block, in slabs of the untouched dimension that fit the slice scratch and the Z parts
// (also: one more product for the launches of the last update)
template <typename YK>
cudaError_t apply_wide(int left, int rows, int other, YK yk, int nb, const double *V, int ldv, double *C, int ldc,
                       const SplitWs &w, cudaStream_t st, const SplitProd *also = nullptr) {
    cudaError_t e;
    int slab = other < kSplitMostRows ? (other + 127) / 128 * 128 : kSplitMostRows;
    auto step_of = [&](int s) {
        WideStep x = wide_step(left, rows, s, nb, V, ldv, C, ldc, w);
        cut_alone(x);
        return x;
    };
    for (; slab > 128; slab = (slab / 2 + 127) / 128 * 128) {
        const WideStep x = step_of(slab);
        if ((size_t)x.np * nb * slab <= w.zcap && step_slices(x) <= w.slice_bytes)
            break;
    }
    SplitSet set{w, st};
    for (int s0 = 0; s0 < other; s0 += slab) {
        WideStep x = step_of(std::min(slab, other - s0));
        x.c = C + (left ? (size_t)s0 * ldc : (size_t)s0);
        if ((e = x.products(yk, set)) != cudaSuccess || (e = set.run()) != cudaSuccess ||
            (e = x.update(set)) != cudaSuccess)
            return e;
        if (s0 + slab < other && (e = set.run()) != cudaSuccess) return e;
    }
    if (also && (e = set.add(*also)) != cudaSuccess) return e;
    return set.run();
}

// where block i0 of a job starts in its C
double *job_c(const WideJob &j, int i0) { return j.C + (j.left ? (size_t)i0 : (size_t)i0 * j.ldc); }

// the blocks of one job from the last to the first
cudaError_t apply_job(const WideJob &j, cudaStream_t st) {
    if (cudaError_t e = form_v(&j, 1, st)) return e;
    for (int i0 = (j.blocks() - 1) * kWide; i0 >= 0; i0 -= kWide) {
        const int nb = std::min(kWide, j.f.count - i0), rows = j.f.rows - i0;
        auto yk = [&](int k0) { return y_vectors(j.f, i0, nb, k0); };
        if (cudaError_t e = apply_wide(j.left, rows, j.other, yk, nb, j.w.V + (size_t)i0 * j.f.rows, j.f.rows,
                                       job_c(j, i0), j.ldc, j.w, st))
            return e;
    }
    return cudaSuccess;
}

// Two jobs side by side (the back-transformations of U and V^T), their
// products in the same launches: below about order 2000 a block's products
// leave most SMs without a tile and its time is the launches' and the K loop
// of a tile's (gesvd of 333 x 333: 4.57 ms one after the other, 4.11 ms so).
cudaError_t apply_pair(const WideJob (&j)[kPair], cudaStream_t st) {
    cudaError_t e;
    if ((e = form_v(j, kPair, st)) != cudaSuccess) return e;
    SplitSet set{j[0].w, st};
    for (int b = std::max(j[0].blocks(), j[1].blocks()) - 1; b >= 0; --b) {
        WideStep x[kPair];
        int tiles = 0;
        bool live[kPair];
        for (int q = 0; q < kPair; ++q) {
            const int i0 = b * kWide;
            if (!(live[q] = b < j[q].blocks())) continue;
            x[q] = wide_step(j[q].left, j[q].f.rows - i0, j[q].other, std::min(kWide, j[q].f.count - i0),
                             j[q].w.V + (size_t)i0 * j[q].f.rows, j[q].f.rows, job_c(j[q], i0), j[q].ldc, j[q].w);
            tiles += x[q].tiles();
        }
        for (int q = 0; q < kPair; ++q)
            if (live[q]) {
                const int fit = (int)(j[q].w.zcap / ((size_t)x[q].nb * x[q].ns));
                x[q].cut(std::min({kSplitMax / kPair, 152 / std::max(tiles, 1), fit}));
                if ((e = x[q].products([&](int k0) { return y_vectors(j[q].f, b * kWide, x[q].nb, k0); }, set)) !=
                    cudaSuccess)
                    return e;
            }
        if ((e = set.run()) != cudaSuccess) return e;
        for (int q = 0; q < kPair; ++q)
            if (live[q] && (e = x[q].update(set)) != cudaSuccess) return e;
        if ((e = set.run()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// How Z = Y^T C of a QR panel is cut along K = rows: np products of kc rows,
// a wave of tiles or so, no product longer than kSplitMostK.  (rows up to
// kSplitMax (kSplitMostK - 64) give np <= kSplitMax and kc <= kSplitMostK.)
struct PanelCut {
    int np, kc;
};
PanelCut panel_cut(int rows, int cols) {
    const int tiles = (cols + 127) / 128, least = (rows + kSplitMostK - 33) / (kSplitMostK - 32);
    const int np = std::max({1, least, std::min({kSplitMax, 152 / std::max(tiles, 1), rows / 256})});
    const int kc = ((rows + np - 1) / np + 31) / 32 * 32;
    return PanelCut{(rows + kc - 1) / kc, kc};
}

// H^T C for one panel of at most kTB reflectors with its T (row-major, ld
// kTB): Z = Y^T C in split-K parts, W = T^T Z in FP64 (small), C -= Y W
cudaError_t apply_panel(const Reflectors &f, const double *T, int rows, int cols, double *C, int ldc, double *W,
                        const SplitWs &w, cudaStream_t st) {
    const int nb = f.count;
    const auto [np, kc] = panel_cut(rows, cols);
    const long long zs = (long long)nb * cols;
    cudaError_t e;
    SplitSet set{w, st};
    for (int y = 0; y < np; ++y) {
        SplitProd p{};
        p.a = y_vectors(f, 0, nb, y * kc);
        p.b = SplitSide{C + y * kc, 0, ldc, 0, cols, 1, 0, 0, 0};
        p.C = w.Z + y * zs;
        p.ldc = nb;
        p.K = std::min(kc, rows - y * kc);
        if ((e = set.add(p)) != cudaSuccess) return e;
    }
    if ((e = set.run()) != cudaSuccess) return e;
    launch_tz(cols, st, T, nb, 1, w.Z, np, 0, cols, W, C, ldc);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    SplitProd p{};
    p.a = y_rows(f, 0, rows, 2);
    p.b = SplitSide{W, 0, nb, 0, cols, 1, 0, 0, 0};
    p.C = C;
    p.ldc = ldc;
    p.K = nb;
    p.sub = 1;
    if ((e = set.add(p)) != cudaSuccess) return e;
    return set.run();
}

// a bounded wait of the products gave up: the result must not pass for one
__global__ void k_poison(const int *err, double *C, long long rows, long long cols, long long ld) {
    if (*err == 0) return;
    for (long long k = threadIdx.x; k < rows * cols; k += blockDim.x)
        C[k / rows * ld + k % rows] = __longlong_as_double(0x7ff8000000000000ll);
}

__global__ void k_fill(double *X, long long rows, long long cols, long long ld, double diag_val) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= rows * cols) return;
    const long long c = k / rows, r = k % rows;
    X[c * ld + r] = (r == c) ? diag_val : 0.0;
}

// columns of the identity less V: column c has its one in row r0 + c, V's rows
// begin there
__global__ void k_identity_less(double *X, long long rows, long long cols, long long ld, int r0, const double *V,
                                long long ldv) {
    pdl_begin();
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= rows * cols) return;
    const long long c = k / rows, r = k % rows;
    X[c * ld + r] = r < r0 ? 0.0 : ((r == c + r0) ? 1.0 : 0.0) - V[c * ldv + r - r0];
}

__global__ void k_copy_upper(const double *A, long long lda, double *R, long long ldr, int n) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)n * n) return;
    const int c = (int)(k / n), r = (int)(k % n);
    R[(size_t)c * ldr + r] = (r <= c) ? A[(size_t)c * lda + r] : 0.0;
}

__global__ void k_zero_rows(double *X, long long ld, int r0, int r1, int cols) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int rows = r1 - r0;
    if (rows <= 0 || k >= (long long)rows * cols) return;
    const int c = (int)(k / rows), r = r0 + (int)(k % rows);
    X[(size_t)c * ld + r] = 0.0;
}

__global__ void k_clear_bar(GridBar *bar) { *bar = GridBar{0, 0, 0, 0}; }
__global__ void k_read_err(const GridBar *bar, int *info) {
    if (bar->err) *info = BDC_ERR_TIMEOUT;
}

int coop_blocks(const void *fn, int threads, size_t smem) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem);
    per = std::min(per, 2);
    return std::max(1, sms * std::max(per, 1));
}

// panel and block sizes
constexpr int kDenseBlock = 32;   // b: columns / rows per panel (reflectors per block)
// reflectors per block when they are applied (back-transformation, explicit
// Q) in FP64: wider blocks pass over C fewer times (Z = Y^T C and C -= Y W
// with K = kApplyBlock)
constexpr int kApplyBlock = kTB;
static_assert(kDenseBlock <= 32 && kDenseBlock <= kTB, "k_geqr2: a lane per later panel column; T of a panel");

constexpr double kQrRatio = 1.6;  // m >= 1.6 n: QR first (Sec. 4.3)
constexpr int kPairMost = 2048;   // largest dimension of back-transformations done side by side

// Blocks of kWide reflectors on the split products, or of kTB in FP64: the
// split path's fixed cost (about 50 launches) is below one FP64 block's three
// products from 64 reflectors on (100 x 100: 0.4 ms either way; 333 x 333:
// 0.64 against 1.39 ms; 600 x 600: 0.88 against 2.3 ms)
bool use_wide(int refl, int rows, int other) {
    return refl >= 64 && other >= 64 && rows <= 8 * kSplitMostK;   // (gram_chunk)
}
// ---- workspaces: every routine lays out what it can reach at its shape
// (bytes from an aligned base; the barrier and error word come first in all).
// A workspace asked for with some sizes serves all smaller ones: the sizes
// here are bounds that grow with every dimension (the cuts along K do not),
// and the *_bytes functions take in what smaller shapes run instead.
struct DenseWs {
    size_t bar = 0, total = 256;
    size_t PW = 0, QW = 0, lab = 0, res = 0;                             // reduction
    size_t part = 0, Y = 0, Ti = 0, Z = 0, split = 0, split_doubles = 0; // QR panels, block reflectors in FP64
    size_t wG[kPair] = {}, wT[kPair] = {}, wX[kPair] = {}, wV[kPair] = {}, wZ[kPair] = {}, wZcap = 0;   // per job
    size_t wS = 0, wSbytes = 0;                                          // slices
    size_t add(size_t bytes) {
        const size_t at = total;
        total += al256(bytes);
        return at;
    }
    size_t doubles(size_t n) { return add(sizeof(double) * n); }
    // block reflectors in FP64: copied reflectors, T, sums, and the partial
    // products that dgemm_parts may use (one per 64 of K, 64 at most; 16 of as
    // many columns as the longest dimension; one where the tiles alone fill the
    // chip 33 times over) or k_gram's
    void fp64(size_t rows, size_t refl, size_t other) {
        constexpr size_t kManyTiles = 340000;
        const size_t len = std::max({rows, refl, other});
        Y = doubles(rows * kTB);
        Ti = doubles((size_t)kTB * (refl + kTB));
        Z = doubles((size_t)kTB * other);
        const size_t parts = std::max<size_t>(1, std::min<size_t>(64, rows / 64));
        split_doubles = std::max({kTB * other, std::min(parts * kTB * std::min(other, kManyTiles), 16 * kTB * len),
                                  (size_t)kTB * kTB * std::max<size_t>(16, std::min(len / 4 + 16, (size_t)4 * sm_count_dense()))});
        split = doubles(split_doubles);
    }
    void slices(size_t bytes) {
        wSbytes = std::max(wSbytes, bytes);
        wS = add(bytes);
    }
};

// Slices held at most, in bytes: whole products of up to 24 M entries (340 MB),
// or of 1024 vectors as long as the longest (`len`); above that products go in
// slabs or sets, or in FP64
size_t slice_cap(size_t len) {
    const size_t lp = (len + 31) / 32 * 32 + 32;
    return 14 * std::max<size_t>((size_t)24 << 20, (size_t)(2 * kWide + 512) * lp) + (size_t)64 * (len + 4096) +
           ((size_t)1 << 20);
}

// Bounds over every cut of `rows` along K into products of nb reflectors on up
// to ns vectors (np kc < rows + 32 np; np a wave's worth of the 152 / tiles, or
// what the length of a product asks for): doubles of the partial results, and
// slices of the products' operands.
int cuts_most(int rows) { return std::max((rows + kSplitMostK - 33) / (kSplitMostK - 32), std::min(kSplitMax, std::max(1, rows / 256))); }
size_t cut_doubles(int rows, int nb, int ns) {
    const size_t one = (size_t)nb * ns, least = (rows + kSplitMostK - 33) / (kSplitMostK - 32);
    return std::max(least * one, std::min(cuts_most(rows) * one, (size_t)152 * 128 * 128));
}
size_t cut_slices(int rows, int nb, int ns) {
    const size_t np = cuts_most(rows), len = rows + 32 * np, v = (size_t)nb + ns;
    return 14 * (v * len + 256 * (size_t)std::min((rows + 31) / 32 * 32 + 32, kSplitMostK)) + 24 * np * (v + 256) +
           8 * (np * 2 * ((ns + 127) / 128 + 1) + 152) + 65536;
}

DenseWs ws_gebrd(int m, int n) {
    DenseWs w;
    constexpr int b = kDenseBlock;
    w.PW = w.doubles(2 * (size_t)b * m);
    w.QW = w.doubles(2 * (size_t)b * n);
    w.lab = w.doubles(labrd_scratch_doubles(m, n));
    w.res = w.doubles(resident_scratch_doubles(n));
    const long long tr = std::min(m - b, kSplitMostRows), tc = std::min<long long>(n - b, tr);
    if (tc > 0) w.slices(split_scratch(2 * tr, 2 * tc, b, ((tr + 127) / 128) * ((tc + 127) / 128)));
    return w;
}

// a QR panel's trailing update on the split products: from about 300 x 300,
// while its slices and Z parts stay below the caps of the m x n matrix
size_t panel_slices(int rows, int cols, const PanelCut &c) {
    const long long tn = (cols + 127) / 128;
    return std::max(split_scratch((long long)c.np * 32, (long long)c.np * cols, c.kc, c.np * tn),
                    split_scratch(rows, cols, 32, (long long)((rows + 127) / 128) * tn));
}
bool panel_split(int rows, int cols, size_t len) {
    if ((long long)rows * cols < 100 * 1000 || cols > kSplitMostRows || rows > kSplitMax * (kSplitMostK - 64)) return false;
    const PanelCut c = panel_cut(rows, cols);
    return c.np <= kSplitMax && c.kc <= kSplitMostK &&
           (size_t)cols * 32 * kSplitMax <= std::max<size_t>((size_t)2 * kWide * (len + 256), (size_t)kWide * 4096) &&
           panel_slices(rows, cols, c) <= slice_cap(len);
}

DenseWs ws_geqrf(int m, int n) {
    DenseWs w;
    constexpr int b = kDenseBlock;
    const size_t len = std::max(m, n);
    w.part = w.doubles((size_t)4 * 256 * (b + 1));   // k_geqr2's partial sums (its grid is at most this)
    w.res = w.doubles(resident_scratch_doubles(kQp));
    w.Ti = w.doubles((size_t)2 * kTB * kTB);         // T, Y^T Y of a panel
    w.Z = w.doubles((size_t)b * n);
    w.Y = w.doubles((size_t)b * m);
    // The largest update that panel_split may take (its columns: at most half
    // the longer side and 128, or 1024; a wide matrix has no fewer than n - m
    // left); one in FP64 is small or larger than that.
    const int rows = std::min(m, kSplitMax * (kSplitMostK - 64));
    const long long side = std::max<long long>(m, std::min<long long>(n, 2ll * m + 256));
    const int cols = (int)std::min<long long>({std::max(n - 1, 0), std::max((side + 256) / 2, 1024ll), kSplitMostRows});
    const long long tiles = (long long)((rows + 127) / 128) * ((cols + 127) / 128);
    const size_t need = std::max(cut_slices(rows, 32, cols), split_scratch(rows, cols, 32, tiles));
    const bool large = m > rows || n - 1 > cols || need > slice_cap(len);
    // Y^T Y of a panel that is too long for the chip: up to four CTAs an SM
    const size_t gram = (size_t)kTB * kTB * std::max(16, std::min((m + 255) / 256, 4 * sm_count_dense()));
    // partial products as in DenseWs::fp64
    const size_t parts = large ? std::max(1, std::min(64, m / 64)) : 1;
    w.split_doubles = std::max({gram, std::min((size_t)b * n * parts, 16 * b * len), (size_t)b * n, (size_t)52000});
    w.split = w.doubles(w.split_doubles);
    if ((long long)rows * cols >= 100 * 1000) {
        w.wZcap = cut_doubles(rows, 32, cols);
        w.wZ[0] = w.doubles(w.wZcap);
        w.slices(std::min(need, slice_cap(len)));
    }
    return w;
}

// the split path of one job, or of two side by side
struct WideShape {
    int left, rows, count, other;   // reflectors of `rows` entries on `other` vectors
    int own;                        // 1: with a product on a block's own columns beside each update (explicit Q)
};
void ws_wide(DenseWs &w, const WideShape *jobs, int njobs) {
    const size_t w2 = (size_t)kWide * kWide;
    size_t need = 0, cap = 0;
    long long gram = 0, vrows = 0, vcols = 0, vtiles = 0;
    int chunk = 0;
    w.wZcap = 0;
    for (int q = 0; q < njobs; ++q) {
        const WideShape &j = jobs[q];
        const int blocks = (j.count + kWide - 1) / kWide, nb = std::min(j.count, kWide);
        const int ns = j.other < kSplitMostRows ? (j.other + 127) / 128 * 128 : kSplitMostRows;
        const int parts = std::min((j.rows + 511) / 512, 8);       // gram_chunks() at most
        w.wG[q] = w.doubles(blocks * w2);
        w.wT[q] = w.doubles(blocks * w2);
        w.wX[q] = w.doubles(blocks * w2);
        w.wV[q] = w.doubles(std::max((size_t)j.rows * j.count, (size_t)blocks * parts * w2));   // V, before it Y^T Y's parts
        gram += (long long)blocks * parts;
        chunk = std::max(chunk, gram_chunk(j.rows));
        for (int b = 0; b < blocks; ++b) {
            const int rows = j.rows - b * kWide, c = std::min(kWide, j.count - b * kWide);
            vrows += rows;
            vcols += c;
            vtiles += (long long)((rows + 127) / 128) * ((c + 127) / 128);
        }
        // products Y^T C and the update, whole
        const long long mt = (j.rows + 127) / 128, nt = (ns + 127) / 128 + (j.own ? (nb + 127) / 128 : 0);
        need += std::max({cut_slices(j.rows, nb, ns), split_scratch((j.own ? 2ll : 1ll) * j.rows, ns + (j.own ? nb : 0), nb, mt * nt),
                          split_scratch(ns, j.rows, nb, mt * nt)});
        const size_t len = std::max(j.rows, std::min(j.other, 1 << 16));
        cap = std::max(cap, slice_cap(len));
        // (the second bound: slabs of the vectors)
        w.wZcap = std::max(w.wZcap, std::min(cut_doubles(j.rows, nb, ns),
                                             std::max<size_t>((size_t)2 * kWide * (len + 256), (size_t)kWide * 4096)));
    }
    gram = std::min<long long>(gram, kSplitMax);
    need = std::max({need, split_scratch(gram * kWide, gram * kWide, chunk, gram * (kWide / 128) * (kWide / 128)),
                     split_scratch(vrows, vcols, kWide, vtiles)});
    for (int q = 0; q < njobs; ++q) w.wZ[q] = w.doubles(w.wZcap);
    w.slices(std::min(need, cap));
}

DenseWs ws_orgqr(int m, int n) {
    DenseWs w;
    if (use_wide(n, m, n)) {
        w.Y = w.doubles((size_t)m * kWide);
        const WideShape j{1, m, n, n, 1};
        ws_wide(w, &j, 1);
    } else {
        w.fp64(m, n, n);
    }
    return w;
}

DenseWs ws_ormbr(int vect, int m, int n, int cdim) {
    DenseWs w;
    const int refl = vect == 0 ? n : n - 1, rows = vect == 0 ? m : n - 1;
    if (use_wide(refl, rows, cdim)) {
        const WideShape j{vect == 0, rows, refl, cdim, 0};
        ws_wide(w, &j, 1);
    } else {
        w.fp64(rows, std::max(refl, 0), cdim);
    }
    return w;
}

// U and V^T of an m x n SVD
bool both_at_once(int m, int n) { return std::max(m, n) <= kPairMost && use_wide(n - 1, m, n); }
DenseWs ws_both(int m, int n) {
    DenseWs w;
    const WideShape j[kPair] = {{1, m, n, n, 0}, {0, n - 1, n - 1, n, 0}};
    ws_wide(w, j, kPair);
    return w;
}

// slices of an m x n by n x n product
DenseWs ws_product(int m, int n) {
    DenseWs w;
    const int rows = std::min(m, kSplitMostRows);
    if (n >= 64 && n <= kSplitMostK)
        w.slices(std::min(slice_cap(std::min(m, 1 << 17)),
                          split_scratch(rows, n, n, (long long)((rows + 127) / 128) * ((n + 127) / 128))));
    return w;
}

// `refl` reflectors of `rows` entries on `other` vectors, and on fewer of each
size_t apply_bytes(int left, int rows, int refl, int other, int own) {
    constexpr int kLongest = 8 * kSplitMostK;
    const bool many = refl >= 64 && other >= 64;
    DenseWs w;
    w.fp64(rows, std::max(refl, 0), other);
    size_t most = w.total;
    if (many) {
        if (rows <= kLongest) {   // fewer than 64 of one
            DenseWs a, b;
            a.fp64(rows, 63, other);
            b.fp64(rows, refl, 63);
            most = std::max(a.total, b.total);
        }
        DenseWs c;
        const WideShape j{left, std::min(rows, kLongest), std::min(refl, kLongest), other, own};
        if (own) c.Y = c.doubles((size_t)j.rows * kWide);
        ws_wide(c, &j, 1);
        most = std::max(most, c.total);
    }
    return most;
}

SplitWs split_ws(char *ws, const DenseWs &w, int job = 0) {
    return SplitWs{(double *)(ws + w.wG[job]), (double *)(ws + w.wT[job]), (double *)(ws + w.wX[job]),
                   (double *)(ws + w.wV[job]), (double *)(ws + w.wZ[job]), w.wZcap, ws + w.wS, w.wSbytes,
                   &((GridBar *)(ws + w.bar))->err};
}

// the split-K scratch of the calling thread's dense routine
struct SplitScope {
    SplitScope(char *ws, const DenseWs &w) {
        g_split_buf = (double *)(ws + w.split);
        g_split_cap = w.split_doubles;
    }
    ~SplitScope() {
        g_split_buf = nullptr;
        g_split_cap = 0;
    }
};

cudaError_t launch_coop(const void *fn, int grid, void *args, cudaStream_t st) {
    void *params[] = {args};
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(256), params, 0, st);
}

}  // namespace

// ---------------------------------------------------------------- drivers
// Bidiagonalization, Algorithm 1 (m >= n): on chip once it fits; before that,
// per panel of b, k_labrd_panel, then the merged rank-(2b) update of the trailing matrix.
cudaError_t dense_gebrd(int m, int n, double *A, int lda, double *d, double *e, double *tauq, double *taup,
                        char *ws, cudaStream_t st) {
    const DenseWs w = ws_gebrd(m, n);
    constexpr int b = kDenseBlock;
    GridBar *bar = (GridBar *)(ws + w.bar);
    cudaError_t err = cudaMemsetAsync(bar, 0, 3 * sizeof(unsigned), st);   // the counters (not the error word)
    if (err != cudaSuccess) return err;
    unsigned bars = 0;
    for (int i0 = 0; i0 < n; i0 += b) {
        const int nb = std::min(b, n - i0), ml = m - i0, nl = n - i0;
        if (resident_fits(ml, nl))
            return launch_gebd2_resident(ml, nl, A + i0 + (size_t)i0 * lda, lda, d + i0, e + i0, tauq + i0, taup + i0,
                                         (double *)(ws + w.res), bar, &bars, st);
        if ((err = launch_labrd_panel(ml, nl, nb, A + i0 + (size_t)i0 * lda, lda, d + i0, e + i0, tauq + i0, taup + i0,
                                      (double *)(ws + w.PW), (double *)(ws + w.QW), (double *)(ws + w.lab), bar, &bars,
                                      st)) != cudaSuccess)
            return err;
        if (nb < nl) {
            // the merged rank-(2b) update A[nb:, nb:] -= P Q^T (Eq. bidiag-A-trail3):
            // P = [V X] (ml x 2b) and Q = [Y U] (nl x 2b) are contiguous column
            // blocks.  Sliced, it is two products of K = b, A -= V Y^T and A -= X U^T:
            // V and U are of order one, X and Y of the trailing matrix's, and
            // the slices keep 56 bits below a vector's maximum, which must not
            // be the other half's: one product of K = 2b under any common
            // scale loses V Y^T where the two differ (1900 x 1900 Gaussian,
            // first column times 1e-8: 1.8e-9 of ||A||; so 1e-15).  Two halves
            // cost 182 ms for 4096 x 4096, one would take 174
            const double *P = (const double *)(ws + w.PW), *Q = (const double *)(ws + w.QW);
            const SplitWs sw = split_ws(ws, w);
            const long long tr = ml - nb, tc = nl - nb;
            if (tr <= kSplitMostRows &&
                split_scratch(2 * tr, 2 * tc, b, ((tr + 127) / 128) * ((tc + 127) / 128)) <= sw.slice_bytes) {
                SplitProd p[2]{};
                for (int h = 0; h < 2; ++h) {
                    p[h].a = SplitSide{P + (size_t)h * b * ml + nb, 0, ml, 1, (int)tr, 1, 0, 0, 0};
                    p[h].b = SplitSide{Q + (size_t)h * b * nl + nb, 0, nl, 1, (int)tc, 1, 0, 0, 0};
                    p[h].C = A + i0 + nb + (size_t)(i0 + nb) * lda;
                    p[h].ldc = lda;
                    p[h].K = b;
                    p[h].sub = 1;
                }
                if ((err = split_products(p, 2, sw.slices, sw.slice_bytes, sw.err, st, 1)) != cudaSuccess) return err;
                continue;
            }
            if ((err = dgemm(0, 1, ml - nb, nl - nb, 2 * b, -1.0, P + nb, ml, Q + nb, nl, 1.0,
                             A + i0 + nb + (size_t)(i0 + nb) * lda, lda, st)) != cudaSuccess)
                return err;
        }
    }
    return cudaSuccess;
}

// QR (Sec. 4.3): per panel, k_geqr2 and the update of the trailing columns by
// H^T = I - Y T^T Y^T in modified compact WY
cudaError_t dense_geqrf(int m, int n, double *A, int lda, double *tau, char *ws, cudaStream_t st) {
    const DenseWs w = ws_geqrf(m, n);
    constexpr int b = kDenseBlock;
    SplitScope split_scope(ws, w);
    GridBar *bar = (GridBar *)(ws + w.bar);
    cudaError_t err = cudaMemsetAsync(bar, 0, 3 * sizeof(unsigned), st);   // the counters (not the error word)
    if (err != cudaSuccess) return err;
    // enough CTAs for ~4 panel rows per thread: the per-column reductions over
    // the CTAs' partial sums grow with the grid
    const int grid = std::max(1, std::min(coop_blocks((const void *)k_geqr2, 256, 0), (m + 1023) / 1024));
    double *Y = (double *)(ws + w.Y), *Ti = (double *)(ws + w.Ti), *Z = (double *)(ws + w.Z);
    const int kmax = std::min(m, n);
    const SplitWs sw = split_ws(ws, w);
    unsigned bars = 0;
    for (int i0 = 0; i0 < kmax; i0 += b) {
        const int nb = std::min(b, kmax - i0), ml = m - i0;
        Geqr2Args a{A + i0 + (size_t)i0 * lda, lda, ml, nb, b, tau + i0, (double *)(ws + w.part), bar};
        const bool resident = geqr2_resident_fits(ml, nb);   // also leaves Y^T Y in gram
        double *gram = Ti + (size_t)kTB * kTB;
        err = resident ? launch_geqr2_resident(ml, nb, a.A, lda, a.tau, gram, kTB, (double *)(ws + w.res), bar,
                                                                  &bars, st)
                                          : launch_coop((const void *)k_geqr2, grid, &a, st);
        if (err != cudaSuccess) return err;
        if (i0 + nb < n) {
            const int cols = n - i0 - nb;
            const Reflectors f{A + i0 + (size_t)i0 * lda, 1, lda, ml, nb};
            const TForm tf{gram, Ti, tau + i0, kTB, 1, 1, nb, 0, 0, 0};
            err = resident ? launch_tform(&tf, 1, 1, st)
                           : form_t(f, tau + i0, Ti, st);
            if (err != cudaSuccess) return err;
            if (panel_split(ml, cols, std::max(m, n))) {
                if ((err = apply_panel(f, Ti, ml, cols, A + i0 + (size_t)(i0 + nb) * lda, lda, Z, sw, st)) !=
                    cudaSuccess)
                    return err;
                continue;
            }
            const long long cnt = (long long)ml * nb;
            launch_pdl(k_form_y, (unsigned)((cnt + 255) / 256), 256, 0, st, Y, ml, nb, A + i0 + (size_t)i0 * lda, 1, lda);
            if ((err = cudaGetLastError()) != cudaSuccess) return err;
            if ((err = apply_block(1, 1, ml, n - i0 - nb, Y, nb, Ti, A + i0 + (size_t)(i0 + nb) * lda, lda, Z, st)) !=
                cudaSuccess)
                return err;
        }
    }
    return cudaSuccess;
}

// the n columns of Q = H_1 ... H_n in place of A (Eq. orgqr-q): the
// panels from the last to the first, each panel's reflectors copied to Y
// before its columns are reset to the identity's
cudaError_t dense_orgqr(int m, int n, double *A, int lda, const double *tau, char *ws, cudaStream_t st) {
    const DenseWs w = ws_orgqr(m, n);
    constexpr int b = kApplyBlock;
    const int k = n;
    SplitScope split_scope(ws, w);
    double *Y = (double *)(ws + w.Y), *Ti = (double *)(ws + w.Ti), *Z = (double *)(ws + w.Z);
    cudaError_t err = cudaSuccess;
    if (use_wide(k, m, n)) {
        const SplitWs sw = split_ws(ws, w);
        const Reflectors f{A, 1, lda, m, k};
        const WideJob job{f, tau, 1, n, A, lda, sw};
        if ((err = form_v(&job, 1, st)) != cudaSuccess) return err;
        for (int i0 = (k - 1) / kWide * kWide; i0 >= 0; i0 -= kWide) {
            const int nb = std::min(kWide, k - i0), ml = m - i0;
            const long long cnt = (long long)ml * nb, c2 = (long long)m * nb;
            launch_pdl(k_form_y, (unsigned)((cnt + 255) / 256), 256, 0, st, Y, ml, nb, A + i0 + (size_t)i0 * lda, 1, lda);
            if ((err = cudaGetLastError()) != cudaSuccess) return err;
            // the block's own columns, E of the identity: E - V Y^T E = (E - V) -
            // V (Y's first nb rows without the unit entries)^T; the ones would
            // set the slices' scale
            const double *V = sw.V + (size_t)i0 * m;
            launch_pdl(k_identity_less, (unsigned)((c2 + 255) / 256), 256, 0, st, A + (size_t)i0 * lda, m, nb, lda, i0, V, m);
            if ((err = cudaGetLastError()) != cudaSuccess) return err;
            const Reflectors fy{Y, 1, ml, ml, nb};
            SplitProd own{};
            own.a = SplitSide{V, 0, m, 1, ml, 1, 0, 0, 0};
            own.b = y_rows(fy, 0, nb, 3);
            own.C = A + i0 + (size_t)i0 * lda;
            own.ldc = lda;
            own.K = nb;
            own.sub = 1;
            err = apply_wide(1, ml, n - i0 - nb, [&](int k0) { return y_vectors(fy, 0, nb, k0); }, nb, V, m,
                             A + i0 + (size_t)(i0 + nb) * lda, lda, sw, st, &own);
            if (err != cudaSuccess) return err;
        }
        return cudaSuccess;
    }
    if ((err = form_t(Reflectors{A, 1, lda, m, k}, tau, Ti, st)) != cudaSuccess) return err;
    const int last = ((k - 1) / b) * b;
    for (int i0 = last; i0 >= 0; i0 -= b) {
        const int nb = std::min(b, k - i0), ml = m - i0;
        const long long cnt = (long long)ml * nb;
        launch_pdl(k_form_y, (unsigned)((cnt + 255) / 256), 256, 0, st, Y, ml, nb, A + i0 + (size_t)i0 * lda, 1, lda);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
        // the panel's columns become identity columns (rows i0.., zero above)
        const long long c2 = (long long)m * nb;
        k_fill<<<(unsigned)((c2 + 255) / 256), 256, 0, st>>>(A + (size_t)i0 * lda, m, nb, lda, 0.0);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
        k_fill<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(A + i0 + (size_t)i0 * lda, ml, nb, lda, 1.0);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
        if ((err = apply_block(1, 0, ml, n - i0, Y, nb, Ti + (size_t)i0 * kTB, A + i0 + (size_t)i0 * lda, lda, Z, st)) !=
            cudaSuccess)
            return err;
    }
    return cudaSuccess;
}

// back-transformation (Sec. 4.3): vect 0: C (m x cols) := Q1 C with the
// column reflectors of gebrd (A m x n, tauq); vect 1: C (rows x n) := C P1^T
// with the row reflectors (taup).  Panels from the last to the first.
cudaError_t dense_ormbr(int vect, int m, int n, const double *A, int lda, const double *tau, double *C, int ldc,
                        int cdim, char *ws, cudaStream_t st) {
    const DenseWs w = ws_ormbr(vect, m, n, cdim);
    constexpr int b = kApplyBlock;
    SplitScope split_scope(ws, w);
    double *Y = (double *)(ws + w.Y), *Ti = (double *)(ws + w.Ti), *Z = (double *)(ws + w.Z);
    cudaError_t err = cudaSuccess;
    const int refl = vect == 0 ? n : n - 1;
    if (use_wide(refl, vect == 0 ? m : n - 1, cdim)) {
        const SplitWs sw = split_ws(ws, w);
        return apply_job(vect == 0 ? WideJob{{A, 1, lda, m, n}, tau, 1, cdim, C, ldc, sw}
                                   : WideJob{{A + lda, lda, 1, n - 1, n - 1}, tau, 0, cdim, C + ldc, ldc, sw}, st);
    }
    if (vect == 0) {
        if ((err = form_t(Reflectors{A, 1, lda, m, n}, tau, Ti, st)) != cudaSuccess) return err;
        const int last = ((n - 1) / b) * b;
        for (int i0 = last; i0 >= 0; i0 -= b) {
            const int nb = std::min(b, n - i0), ml = m - i0;
            const long long cnt = (long long)ml * nb;
            launch_pdl(k_form_y, (unsigned)((cnt + 255) / 256), 256, 0, st, Y, ml, nb, A + i0 + (size_t)i0 * lda, 1, lda);
            if ((err = cudaGetLastError()) != cudaSuccess) return err;
            if ((err = apply_block(1, 0, ml, cdim, Y, nb, Ti + (size_t)i0 * kTB, C + i0, ldc, Z, st)) != cudaSuccess)
                return err;
        }
        return cudaSuccess;
    }
    if (n < 2) return cudaSuccess;
    const int nr = n - 1;   // row reflectors G_0 .. G_{n-2}, acting on columns 1..n-1
    if ((err = form_t(Reflectors{A + lda, lda, 1, n - 1, nr}, tau, Ti, st)) != cudaSuccess) return err;
    const int last = ((nr - 1) / b) * b;
    for (int i0 = last; i0 >= 0; i0 -= b) {
        const int nb = std::min(b, nr - i0), ny = n - 1 - i0;
        const long long cnt = (long long)ny * nb;
        // Y[r][j] = u_{i0+j} at column i0 + 1 + r: row i0 + j of A from column i0 + 1
        launch_pdl(k_form_y, (unsigned)((cnt + 255) / 256), 256, 0, st, Y, ny, nb, A + i0 + (size_t)(i0 + 1) * lda, lda, 1);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
        if ((err = apply_block(0, 1, cdim, ny, Y, nb, Ti + (size_t)i0 * kTB, C + (size_t)(i0 + 1) * ldc, ldc, Z, st)) !=
            cudaSuccess)
            return err;
    }
    return cudaSuccess;
}

// U := Q1 U (m x n) and VT := VT P1^T (n x n) with the reflectors of gebrd
cudaError_t dense_ormbr_both(int m, int n, const double *A, int lda, const double *tauq, const double *taup, double *U,
                             int ldu, double *VT, int ldvt, char *ws, cudaStream_t st) {
    if (both_at_once(m, n)) {
        const DenseWs w = ws_both(m, n);
        const WideJob j[kPair] = {{{A, 1, lda, m, n}, tauq, 1, n, U, ldu, split_ws(ws, w)},
                                  {{A + lda, lda, 1, n - 1, n - 1}, taup, 0, n, VT + ldvt, ldvt, split_ws(ws, w, 1)}};
        return apply_pair(j, st);
    }
    if (cudaError_t e = dense_ormbr(0, m, n, A, lda, tauq, U, ldu, n, ws, st)) return e;
    return dense_ormbr(1, m, n, A, lda, taup, VT, ldvt, n, ws, st);
}

size_t gebrd_bytes(int m, int n) { return ws_gebrd(m, n).total; }
size_t geqrf_bytes(int m, int n) { return std::max(ws_geqrf(m, n).total, apply_bytes(1, m, std::min(m, n), std::min(m, n), 1)); }
size_t ormbr_bytes(int m, int n, int cdim) {
    return std::max(apply_bytes(1, m, n, cdim, 0), apply_bytes(0, n - 1, n - 1, cdim, 0));
}
size_t gesvd_bytes(int m, int n) {
    size_t most = std::max(gebrd_bytes(m, n), ormbr_bytes(m, n, n));
    const int mp = std::min(m, kPairMost), np = std::min(n, kPairMost), nq = std::min(n, (int)(m / kQrRatio));
    if (both_at_once(mp, np)) most = std::max(most, ws_both(mp, np).total);
    if (nq > 0) most = std::max({most, geqrf_bytes(m, nq), ws_product(m, std::min(nq, kSplitMostK)).total});
    return most;
}
// (a kernel, not a memset: overlapped launches may follow it directly)
cudaError_t dense_clear_err(char *ws, cudaStream_t st) {
    k_clear_bar<<<1, 1, 0, st>>>((GridBar *)(ws + DenseWs().bar));
    return cudaGetLastError();
}
cudaError_t dense_read_err(char *ws, int *info, cudaStream_t st) {
    k_read_err<<<1, 1, 0, st>>>((const GridBar *)(ws + DenseWs().bar), info);
    return cudaGetLastError();
}
cudaError_t dense_poison(char *ws, double *C, int rows, int cols, int ld, cudaStream_t st) {
    k_poison<<<1, 1024, 0, st>>>(&((const GridBar *)(ws + DenseWs().bar))->err, C, rows, cols, ld);
    return cudaGetLastError();
}
cudaError_t dense_copy_upper(const double *A, int lda, double *R, int ldr, int n, cudaStream_t st) {
    const long long cnt = (long long)n * n;
    k_copy_upper<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(A, lda, R, ldr, n);
    return cudaGetLastError();
}
cudaError_t dense_zero_rows(double *X, int ld, int r0, int r1, int cols, cudaStream_t st) {
    const long long cnt = (long long)(r1 - r0) * cols;
    if (cnt <= 0) return cudaSuccess;
    k_zero_rows<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(X, ld, r0, r1, cols);
    return cudaGetLastError();
}
// C (m x n) = A (m x n, lda) B (n x n, ld n), in row slabs that fit the slices
cudaError_t dense_product(int m, int n, const double *A, int lda, const double *B, double *C, int ldc, char *ws,
                          cudaStream_t st) {
    const DenseWs w = ws_product(m, n);
    const SplitWs sw = split_ws(ws, w);
    auto fits = [&](int r) {
        return split_scratch(r, n, n, (long long)((r + 127) / 128) * ((n + 127) / 128)) <= sw.slice_bytes;
    };
    int slab = std::min(m, kSplitMostRows);
    while (slab > 128 && !fits(slab)) slab = (slab / 2 + 127) / 128 * 128;
    if (n < 64 || n > kSplitMostK || !fits(slab))
        return dgemm(0, 0, m, n, n, 1.0, A, lda, B, n, 0.0, C, ldc, st);
    for (int r0 = 0; r0 < m; r0 += slab) {
        SplitProd p{};
        p.a = SplitSide{A + r0, 0, lda, 1, std::min(slab, m - r0), 1, 0, 0, 0};
        p.b = SplitSide{B, 0, n, 0, n, 1, 0, 0, 0};
        p.C = C + r0;
        p.ldc = ldc;
        p.K = n;
        if (cudaError_t e = split_products(&p, 1, sw.slices, sw.slice_bytes, sw.err, st)) return e;
    }
    return cudaSuccess;
}

}  // namespace bdc

// ------------------------------------------------------------- C ABI
using namespace bdc;

namespace {

char *align_ws(void *work) { return (char *)(((uintptr_t)work + 255) & ~(uintptr_t)255); }

int note_cuda(cudaError_t e) { return e == cudaSuccess ? 0 : BDC_ERR_CUDA; }

struct GesvdWs {
    size_t dense, vecs, R, UR, bdc, total;
};
GesvdWs gesvd_layout(int m, int n, const bdc_opts *o) {
    GesvdWs w{};
    size_t off = 0;
    const bool qr = m >= kQrRatio * n;
    w.dense = off; off += al256(gesvd_bytes(m, n));
    w.vecs = off; off += al256(sizeof(double) * 4 * (size_t)n + 64);
    w.R = off; off += qr ? al256(sizeof(double) * (size_t)n * n) : 0;
    w.UR = off; off += qr ? al256(sizeof(double) * (size_t)n * n) : 0;
    w.bdc = off; off += al256(bdc_svd_workspace(n, o));
    w.total = off + 512;
    return w;
}

}  // namespace

extern "C" {

size_t bdc_gebrd_workspace(int m, int n) {
    if (m < n || n < 0) return 0;
    return gebrd_bytes(m, n) + 512;
}

int bdc_gebrd(int m, int n, double *A, int lda, double *d, double *e, double *tauq, double *taup, void *work,
              size_t lwork, int *d_info, bdc_stream_t stream) {
    if (n < 0) return -2;
    if (m < n) return -1;
    if (n > 0 && !A) return -3;
    if (lda < std::max(1, m)) return -4;
    if (n > 0 && (!d || !tauq || !taup || (n > 1 && !e))) return -5;
    if (!d_info) return -12;
    cudaStream_t st = (cudaStream_t)stream;
    const OverlapScope overlapped(st);
    if (int r = note_cuda(cudaMemsetAsync(d_info, 0, sizeof(int), st))) return r;
    if (n == 0) return 0;
    if (!work) return -10;
    if (lwork < bdc_gebrd_workspace(m, n)) return -11;
    char *ws = align_ws(work);
    if (int r = note_cuda(dense_clear_err(ws, st))) return r;
    if (int r = note_cuda(cudaMemsetAsync(taup, 0, sizeof(double) * n, st))) return r;
    if (int r = note_cuda(dense_gebrd(m, n, A, lda, d, e, tauq, taup, ws, st))) return r;
    return note_cuda(dense_read_err(ws, d_info, st));
}

int bdc_ormbr(int vect, int m, int n, const double *A, int lda, const double *tau, double *C, int ldc, int cdim,
              void *work, size_t lwork, bdc_stream_t stream) {
    if (vect < 0 || vect > 1) return -1;
    if (m < n || n < 0) return -2;
    if (n > 0 && !A) return -4;
    if (lda < std::max(1, m)) return -5;
    if (n > 0 && !tau) return -6;
    if (cdim < 0) return -9;
    if (cdim > 0 && n > 0 && !C) return -7;
    if (ldc < std::max(1, vect == 0 ? m : cdim)) return -8;
    if (n == 0 || cdim == 0) return 0;
    if (!work) return -10;
    if (lwork < bdc_ormbr_workspace(m, n, cdim)) return -11;
    cudaStream_t st = (cudaStream_t)stream;
    const OverlapScope overlapped(st);
    char *ws = align_ws(work);
    if (int r = note_cuda(dense_clear_err(ws, st))) return r;
    if (int r = note_cuda(dense_ormbr(vect, m, n, A, lda, tau, C, ldc, cdim, ws, st))) return r;
    return note_cuda(dense_poison(ws, C, vect == 0 ? m : cdim, vect == 0 ? cdim : n, ldc, st));
}

size_t bdc_ormbr_workspace(int m, int n, int cdim) {
    if (m < n || n < 0 || cdim < 0) return 0;
    return ormbr_bytes(m, n, cdim) + 512;
}

size_t bdc_geqrf_workspace(int m, int n) {
    if (m < 0 || n < 0) return 0;
    return geqrf_bytes(std::max(m, 1), std::max(n, 1)) + 512;
}

int bdc_geqrf(int m, int n, double *A, int lda, double *tau, void *work, size_t lwork, int *d_info,
              bdc_stream_t stream) {
    if (m < 0) return -1;
    if (n < 0) return -2;
    if (m > 0 && n > 0 && !A) return -3;
    if (lda < std::max(1, m)) return -4;
    if (std::min(m, n) > 0 && !tau) return -5;
    if (!d_info) return -9;
    cudaStream_t st = (cudaStream_t)stream;
    const OverlapScope overlapped(st);
    if (int r = note_cuda(cudaMemsetAsync(d_info, 0, sizeof(int), st))) return r;
    if (std::min(m, n) == 0) return 0;
    if (!work) return -6;
    if (lwork < bdc_geqrf_workspace(m, n)) return -7;
    char *ws = align_ws(work);
    if (int r = note_cuda(dense_clear_err(ws, st))) return r;
    if (int r = note_cuda(dense_geqrf(m, n, A, lda, tau, ws, st))) return r;
    return note_cuda(dense_read_err(ws, d_info, st));
}

int bdc_orgqr(int m, int n, double *A, int lda, const double *tau, void *work, size_t lwork, bdc_stream_t stream) {
    if (m < 0) return -1;
    if (n < 0 || n > m) return -2;
    if (n > 0 && !A) return -3;
    if (lda < std::max(1, m)) return -4;
    if (n > 0 && !tau) return -5;
    if (n == 0) return 0;
    if (!work) return -6;
    if (lwork < bdc_geqrf_workspace(m, n)) return -7;
    cudaStream_t st = (cudaStream_t)stream;
    const OverlapScope overlapped(st);
    char *ws = align_ws(work);
    if (int r = note_cuda(dense_clear_err(ws, st))) return r;
    if (int r = note_cuda(dense_orgqr(m, n, A, lda, tau, ws, st))) return r;
    return note_cuda(dense_poison(ws, A, m, n, lda, st));
}

size_t bdc_gesvd_workspace(int m, int n, const bdc_opts *o) {
    if (m < n || n < 0) return 0;
    return gesvd_layout(m, std::max(n, 1), o).total;
}

int bdc_gesvd(int m, int n, double *A, int lda, double *S, double *U, int ldu, double *VT, int ldvt,
              const bdc_opts *o, void *work, size_t lwork, int *d_info, bdc_stream_t stream) {
    if (n < 0) return -2;
    if (m < n) return -1;
    if (n > 0 && !A) return -3;
    if (lda < std::max(1, m)) return -4;
    if (n > 0 && (!S || !U || !VT)) return -5;
    if (ldu < std::max(1, m)) return -7;
    if (ldvt < std::max(1, n)) return -9;
    if (!d_info) return -13;
    cudaStream_t st = (cudaStream_t)stream;
    const OverlapScope overlapped(st);
    if (int r = note_cuda(cudaMemsetAsync(d_info, 0, sizeof(int), st))) return r;
    if (n == 0) return 0;
    if (o && o->vectors != BDC_VEC_BOTH) return -10;
    if (!work) return -11;
    const GesvdWs L = gesvd_layout(m, n, o);
    if (lwork < L.total) return -12;
    char *ws = align_ws(work);
    char *dws = ws + L.dense;
    double *d = (double *)(ws + L.vecs), *e = d + n, *tq = e + n, *tp = tq + n;
    if (int r = note_cuda(dense_clear_err(dws, st))) return r;
    if (int r = note_cuda(cudaMemsetAsync(tp, 0, sizeof(double) * n, st))) return r;
    const size_t lwb = bdc_svd_workspace(n, o);
    int rc = 0;
    if (m >= kQrRatio * n) {
        // tall and skinny: A = Q R, the SVD of R, U = Q U_R (Sec. 4.3)
        double *R = (double *)(ws + L.R), *UR = (double *)(ws + L.UR);
        if ((rc = note_cuda(dense_geqrf(m, n, A, lda, tq, dws, st)))) return rc;
        if ((rc = note_cuda(dense_copy_upper(A, lda, R, n, n, st)))) return rc;
        if ((rc = note_cuda(dense_orgqr(m, n, A, lda, tq, dws, st)))) return rc;
        if ((rc = note_cuda(cudaMemsetAsync(tq, 0, sizeof(double) * n, st)))) return rc;
        if ((rc = note_cuda(dense_gebrd(n, n, R, n, d, e, tq, tp, dws, st)))) return rc;
        if ((rc = bdc_svd_ex(n, d, e, UR, S, VT, n, ldvt, o, ws + L.bdc, lwb, d_info, stream))) return rc;
        if ((rc = note_cuda(dense_ormbr_both(n, n, R, n, tq, tp, UR, n, VT, ldvt, dws, st)))) return rc;
        if ((rc = note_cuda(dense_product(m, n, A, lda, UR, U, ldu, dws, st)))) return rc;
    } else {
        if ((rc = note_cuda(dense_gebrd(m, n, A, lda, d, e, tq, tp, dws, st)))) return rc;
        if ((rc = bdc_svd_ex(n, d, e, U, S, VT, ldu, ldvt, o, ws + L.bdc, lwb, d_info, stream))) return rc;
        if ((rc = note_cuda(dense_zero_rows(U, ldu, n, m, n, st)))) return rc;
        if ((rc = note_cuda(dense_ormbr_both(m, n, A, lda, tq, tp, U, ldu, VT, ldvt, dws, st)))) return rc;
    }
    return note_cuda(dense_read_err(dws, d_info, st));
}

}  // extern "C"
