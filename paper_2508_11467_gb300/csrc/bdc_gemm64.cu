// Merge products of Eq. (bdc-Mv2Bv-u-vt) in the working precision: C = A * B,
// all column-major, a batch of independent problems per launch (four per
// merge node: the top and bottom blocks of W~ U_M and Q~ V_M).
//
// FP32 build: CUDA-core FP32 FMA in packed pairs, CTA tiles 64 x 32 or
// 32 x 32 (launch_gemm64), 8 x 4 outputs a thread, operands staged k-major in
// two padded shared buffers (float4 reads, one barrier a K step), the next K
// step prefetched into registers.
//
// FP64 build: tensor-core FP64 (DMMA, mma.sync.m8n8k4.f64).  CTA tile 64 x 64
// (32 x 32, 32 x 64 or 64 x 32 for small problems), K step 16, warps of
// 32 x 32 (4 x 4 fragments of 8 x 8).  Shared tiles are padded
// so that the fragment loads of a warp hit every bank exactly twice (the
// minimum for 32 doubles).  The next K step is prefetched into registers while
// the current one is multiplied.  Problems whose actual size (known only on
// the device after deflation) is smaller than the launch grid exit early.
#include "bdc_internal.cuh"

namespace BDC_NS {

namespace {

#ifdef BDC_FP32
// acc(lo, hi) += a(lo, hi) * b: two FP32 fused multiply-adds, each rounded as
// fmaf rounds
__device__ __forceinline__ void ffma2(unsigned long long &acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pair2(float lo, float hi) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}

// RT x CT threads of 8 rows x 4 columns each.  Bound by latency (global loads
// of a step, shared reads) and by padding of the many small blocks, not by the
// FMA rate: the tiles are small, the registers capped (MINB) so that ~28 warps
// an SM are in flight, and BK = 8 halves the staging registers and shared
// memory.  Both operands of two FMAs ride in one packed instruction.  512
// matrices of order 32..1024 (whole solve): 64 x 64 tiles of 256 threads and
// single FMAs 4236 us; 64 x 64 tiles of 128 threads, packed, 3739; 64 x 32
// 3633; K step 8 and 70 registers 3489 (130 registers: 4008, 64: 3544).
// 64 x 64 with 8 x 8 outputs a thread: 3793.
template <int RT, int CT, int BK, int MINB>
__global__ void __launch_bounds__(RT * CT, MINB) k_gemm32(const GemmProb *__restrict__ probs, int tilesN) {
    constexpr int BM = 8 * RT, BN = 4 * CT, T = RT * CT;
    constexpr int SA = BM + 4, SB = BN + 4;          // padded row strides (floats)
    constexpr int LA = BM * BK / T, LB = BN * BK / T;
    __shared__ __align__(16) float As[2][BK * SA];   // As[.][k][m]
    __shared__ __align__(16) float Bs[2][BK * SB];   // Bs[.][k][n]
    const GemmProb pr = probs[blockIdx.y];
    const int m0 = (blockIdx.x / tilesN) * BM, n0 = (blockIdx.x % tilesN) * BN;
    if (m0 >= pr.M || n0 >= pr.N) return;
    const int tid = threadIdx.x;
    const int tm = (tid / CT) * 8, tn = (tid % CT) * 4;
    const float *__restrict__ A = pr.A;
    const float *__restrict__ B = pr.B;
    const int M = pr.M, N = pr.N, K = pr.K, lda = pr.lda, ldb = pr.ldb;
    unsigned long long acc[4][4];                   // rows 2 i, 2 i + 1
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    float ra[LA], rb[LB];
    auto load = [&](int k0) {
#pragma unroll
        for (int r = 0; r < LA; ++r) {
            const int idx = tid + r * T, gm = m0 + idx % BM, gk = k0 + idx / BM;
            ra[r] = (gm < M && gk < K) ? A[(size_t)gk * lda + gm] : 0.f;
        }
#pragma unroll
        for (int r = 0; r < LB; ++r) {
            const int idx = tid + r * T, gk = k0 + idx % BK, gn = n0 + idx / BK;
            rb[r] = (gn < N && gk < K) ? B[(size_t)gn * ldb + gk] : 0.f;
        }
    };
    load(0);
    for (int k0 = 0, buf = 0; k0 < K; k0 += BK, buf ^= 1) {
        // one barrier a step: the buffer written here was last read two steps
        // ago, before the barrier of the step between
#pragma unroll
        for (int r = 0; r < LA; ++r) {
            const int idx = tid + r * T;
            As[buf][(idx / BM) * SA + idx % BM] = ra[r];
        }
#pragma unroll
        for (int r = 0; r < LB; ++r) {
            const int idx = tid + r * T;
            Bs[buf][(idx % BK) * SB + idx / BK] = rb[r];
        }
        __syncthreads();
        if (k0 + BK < K) load(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(&As[buf][kk * SA + tm]);
            const ulonglong2 a1 = *reinterpret_cast<const ulonglong2 *>(&As[buf][kk * SA + tm + 4]);
            const unsigned long long av[4] = {a0.x, a0.y, a1.x, a1.y};
            const float4 b = *reinterpret_cast<const float4 *>(&Bs[buf][kk * SB + tn]);
            const unsigned long long bv[4] = {pair2(b.x, b.x), pair2(b.y, b.y), pair2(b.z, b.z), pair2(b.w, b.w)};
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) ffma2(acc[i][j], av[i], bv[j]);
        }
    }
    float *__restrict__ C = pr.C;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int gn = n0 + tn + j;
        if (gn >= N) continue;
        float *__restrict__ Cc = C + gemm_col(pr, gn);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int gm = m0 + tm + 2 * i;
            if (gm < M) Cc[gm] = __uint_as_float((unsigned)acc[i][j]);
            if (gm + 1 < M) Cc[gm + 1] = __uint_as_float((unsigned)(acc[i][j] >> 32));
        }
    }
}

template <int RT, int CT, int BK, int MINB>
cudaError_t gemm32(const GemmProb *probs, int nprobs, int rows, int cols, cudaStream_t st) {
    const int tm = (rows + 8 * RT - 1) / (8 * RT), tn = (cols + 4 * CT - 1) / (4 * CT);
    for (int p0 = 0; p0 < nprobs; p0 += 65535) {
        const int np = (nprobs - p0 < 65535) ? nprobs - p0 : 65535;
        k_gemm32<RT, CT, BK, MINB><<<dim3((unsigned)tm * tn, np), RT * CT, 0, st>>>(probs + p0, tn);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
#else
constexpr int BK = 16;

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
                 : "+d"(c[0]), "+d"(c[1])
                 : "d"(a), "d"(b));
}

// CTA tile (32 WM) x (32 WN): WM x WN warps of 32 x 32 each, registers
// capped so that twelve warps fit an SM (three 2 x 2 CTAs; measured: two
// CTAs of 206 registers 29.7 ms of FP64 products at n = 16384, three 29.0,
// four with spills 29.2); the small
// tiles serve merges whose blocks are a few dozen rows (a 64 x 64 tile
// there multiplies mostly zeros at GB300's modest FP64 tensor rate)
template <int WM, int WN>
__global__ void __launch_bounds__(32 * WM * WN, 3 * 4 / (WM * WN)) k_gemm64(const GemmProb *__restrict__ probs, int tilesN) {
    constexpr int BM = 32 * WM, BN = 32 * WN, T = 32 * WM * WN;
    constexpr int SA = BM + 8;   // As[k][m] row stride (doubles)
    constexpr int SB = BK + 4;   // Bs[n][k] row stride
    constexpr int LA = BM * BK / T, LB = BN * BK / T;   // elements per thread
    __shared__ double As[BK * SA];
    __shared__ double Bs[BN * SB];
    const GemmProb pr = probs[blockIdx.y];
    const int m0 = (blockIdx.x / tilesN) * BM, n0 = (blockIdx.x % tilesN) * BN;
    if (m0 >= pr.M || n0 >= pr.N) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = (warp / WN) * 32, wn = (warp % WN) * 32;
    const int g = lane >> 2, tg = lane & 3;
    const double *__restrict__ A = pr.A;
    const double *__restrict__ B = pr.B;
    const int M = pr.M, N = pr.N, K = pr.K, lda = pr.lda, ldb = pr.ldb;

    double acc[4][4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;

    // global -> register staging: A tile (BM m x BK k), B tile (BK k x BN n)
    double ra[LA], rb[LB];
    auto load = [&](int k0) {
#pragma unroll
        for (int r = 0; r < LA; ++r) {
            const int idx = tid + r * T;
            const int am = idx % BM, ak = idx / BM;
            const int gm = m0 + am, gk = k0 + ak;
            ra[r] = (gm < M && gk < K) ? A[(size_t)gk * lda + gm] : 0.0;
        }
#pragma unroll
        for (int r = 0; r < LB; ++r) {
            const int idx = tid + r * T;
            const int bk = idx % BK, bn = idx / BK;
            const int gn = n0 + bn, gk = k0 + bk;
            rb[r] = (gn < N && gk < K) ? B[(size_t)gn * ldb + gk] : 0.0;
        }
    };
    auto store = [&]() {
#pragma unroll
        for (int r = 0; r < LA; ++r) {
            const int idx = tid + r * T;
            As[(idx / BM) * SA + (idx % BM)] = ra[r];
        }
#pragma unroll
        for (int r = 0; r < LB; ++r) {
            const int idx = tid + r * T;
            Bs[(idx / BK) * SB + (idx % BK)] = rb[r];
        }
    };
    load(0);
    for (int k0 = 0; k0 < K; k0 += BK) {
        __syncthreads();
        store();
        __syncthreads();
        if (k0 + BK < K) load(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; kk += 4) {
            if (k0 + kk >= K) break;               // zero padding of the last K block
            double af[4], bf[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) af[i] = As[(kk + tg) * SA + wm + i * 8 + g];
#pragma unroll
            for (int j = 0; j < 4; ++j) bf[j] = Bs[(wn + j * 8 + g) * SB + kk + tg];
            // 8 x 8 fragments wholly outside M x N are skipped (warp-uniform):
            // a merge of order 16 has blocks of about 8 x 16 in a 32 x 32 tile
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (m0 + wm + i * 8 < M && n0 + wn + j * 8 < N) dmma(acc[i][j], af[i], bf[j]);
        }
    }
    // fragment (g, 2 tg + {0,1}) of each 8 x 8 tile
    double *__restrict__ C = pr.C;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int gm = m0 + wm + i * 8 + g;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int gn = n0 + wn + j * 8 + 2 * tg;
            if (gn < N) C[gemm_col(pr, gn) + gm] = acc[i][j][0];
            if (gn + 1 < N) C[gemm_col(pr, gn + 1) + gm] = acc[i][j][1];
        }
    }
}

// Small blocks: one warp per tile of F x F fragments (8 x 8 each), four
// independent tiles (of any problems) per CTA.  The fragments are loaded
// straight from global memory (L1/L2), one K step of 4 ahead of the MMAs, so
// a tile costs its loads' latency once instead of a shared-memory round trip
// per K block, and the warp's register budget (<= 128) keeps four CTAs of
// four warps per SM in flight.  Fragments wholly outside the block are
// neither loaded nor multiplied (warp-uniform).  An FP64 MMA holds its SM
// sub-partition for 615 cycles (1.67 multiply-adds a clock and SM, measured),
// so a tile's time is its MMAs: with fewer tiles than sub-partitions smaller
// ones are faster (the four products of one order-100 merge: 45.9 us at F = 4,
// 9.7 us at F = 1).  Every output sums its K steps in the same order at any F.
constexpr int SW_WARPS = 4;
// Largest blocks they serve once the chip is full: one half of a merge's rows
// by all its columns.  512 matrices of order 32..1024 (whole solve) with blocks
// of 35..64 x 65..128 here 21343 us, by the 64 x 64 tiles 21520 us.
constexpr int kSmallRows = 64, kSmallCols = 128;

template <int F>
__global__ void __launch_bounds__(32 * SW_WARPS, 4) k_gemm64_warp(const GemmProb *__restrict__ probs, int nprobs,
                                                                   int tilesM, int tilesN) {
    const int lane = threadIdx.x & 31;
    const long long gw = (long long)blockIdx.x * SW_WARPS + (threadIdx.x >> 5);
    const int tiles = tilesM * tilesN;
    const long long p = gw / tiles;
    if (p >= nprobs) return;
    const GemmProb pr = probs[p];
    const int t = (int)(gw % tiles);
    const int m0 = (t / tilesN) * (8 * F), n0 = (t % tilesN) * (8 * F);
    const int M = pr.M, N = pr.N, K = pr.K, lda = pr.lda, ldb = pr.ldb;
    if (m0 >= M || n0 >= N) return;
    const int fi = min(F, (M - m0 + 7) >> 3), fj = min(F, (N - n0 + 7) >> 3);   // live fragment rows / columns
    const int g = lane >> 2, tg = lane & 3;
    const double *__restrict__ A = pr.A;
    const double *__restrict__ B = pr.B;
    double acc[F][F][2];
#pragma unroll
    for (int i = 0; i < F; ++i)
#pragma unroll
        for (int j = 0; j < F; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
    // fragments of K step k: A (row m0 + 8 i + g, column k + tg), B (row k + tg, column n0 + 8 j + g)
    auto ldf = [&](int k, double (&af)[F], double (&bf)[F]) {
        const int kk = k + tg;
        const bool kok = kk < K;
#pragma unroll
        for (int i = 0; i < F; ++i) {
            const int row = m0 + 8 * i + g;
            af[i] = (i < fi && kok && row < M) ? A[(size_t)kk * lda + row] : 0.0;
        }
#pragma unroll
        for (int j = 0; j < F; ++j) {
            const int col = n0 + 8 * j + g;
            bf[j] = (j < fj && kok && col < N) ? B[(size_t)col * ldb + kk] : 0.0;
        }
    };
    auto mul = [&](const double (&af)[F], const double (&bf)[F]) {
#pragma unroll
        for (int i = 0; i < F; ++i)
#pragma unroll
            for (int j = 0; j < F; ++j)
                if (i < fi && j < fj) dmma(acc[i][j], af[i], bf[j]);
    };
    if constexpr (F == 4) {
        double a0[F], b0[F], a1[F], b1[F];
        ldf(0, a0, b0);
        for (int k = 0; k < K; k += 8) {
            if (k + 4 < K) ldf(k + 4, a1, b1);
            mul(a0, b0);
            if (k + 4 >= K) break;
            if (k + 8 < K) ldf(k + 8, a0, b0);
            mul(a1, b1);
        }
    } else {
        // four K steps ahead: few warps, so the loads' latency shows
        constexpr int P = 4;
        double a[P][F], b[P][F];
#pragma unroll
        for (int q = 0; q < P; ++q) ldf(4 * q, a[q], b[q]);
        for (int k = 0; k < K; k += 4 * P) {
#pragma unroll
            for (int q = 0; q < P; ++q) {
                if (k + 4 * q < K) mul(a[q], b[q]);
                ldf(k + 4 * q + 4 * P, a[q], b[q]);
            }
        }
    }
    // fragment (g, 2 tg + {0,1}) of each 8 x 8 tile; output columns through the column map
    double *__restrict__ C = pr.C;
    size_t col0[F], col1[F];
#pragma unroll
    for (int j = 0; j < F; ++j) {
        const int gn = n0 + 8 * j + 2 * tg;
        col0[j] = (j < fj && gn < N) ? gemm_col(pr, gn) : 0;
        col1[j] = (j < fj && gn + 1 < N) ? gemm_col(pr, gn + 1) : 0;
    }
#pragma unroll
    for (int i = 0; i < F; ++i) {
        const int gm = m0 + 8 * i + g;
        if (i >= fi || gm >= M) continue;
#pragma unroll
        for (int j = 0; j < F; ++j) {
            const int gn = n0 + 8 * j + 2 * tg;
            if (j >= fj) continue;
            if (gn < N) C[col0[j] + gm] = acc[i][j][0];
            if (gn + 1 < N) C[col1[j] + gm] = acc[i][j][1];
        }
    }
}

template <int F>
cudaError_t gemm64_warp(const GemmProb *probs, int nprobs, int rows, int cols, cudaStream_t st) {
    const int tm = (rows + 8 * F - 1) / (8 * F), tn = (cols + 8 * F - 1) / (8 * F);
    const long long ctas = ((long long)nprobs * tm * tn + SW_WARPS - 1) / SW_WARPS;
    k_gemm64_warp<F><<<(unsigned)ctas, 32 * SW_WARPS, 0, st>>>(probs, nprobs, tm, tn);
    return cudaGetLastError();
}

#endif  // BDC_FP32

}  // namespace

cudaError_t launch_gemm64(const GemmProb *probs, int nprobs, int mmax_rows, int nmax_cols, cudaStream_t st) {
    if (nprobs <= 0 || mmax_rows <= 0 || nmax_cols <= 0) return cudaSuccess;
#ifdef BDC_FP32
    // the fewest, longest-running tiles lose to smaller ones while the chip is
    // not full (four matrices of order 1000, whole solve: 494 us with 64 x 64
    // tiles, 482 us with 32 x 32 and K step 16), and up to 36 columns anything
    // wider is mostly padding (2000 matrices of order 24..80: 1005 us with
    // 32 x 64, 967 us with 32 x 32); elsewhere 64 x 32 (above)
    const long long tiles = (long long)nprobs * ((mmax_rows + 63) / 64) * ((nmax_cols + 63) / 64);
    if (tiles < 4 * 152) return gemm32<4, 8, 16, 12>(probs, nprobs, mmax_rows, nmax_cols, st);
    if (nmax_cols <= 36) return gemm32<4, 8, 8, 20>(probs, nprobs, mmax_rows, nmax_cols, st);
    return gemm32<8, 8, 8, 14>(probs, nprobs, mmax_rows, nmax_cols, st);
#else
    // tiles of one, four or sixteen fragments: the largest that still give
    // every SM sub-partition (4 x 152) four of them (by the host's
    // bounds; deflation leaves fewer)
    constexpr long long kFill = 4 * 152 * 4;
    const long long frags = (long long)nprobs * ((mmax_rows + 7) / 8) * ((nmax_cols + 7) / 8);
    if (frags <= 4 * kFill) return gemm64_warp<1>(probs, nprobs, mmax_rows, nmax_cols, st);
    if (frags <= 16 * kFill) return gemm64_warp<2>(probs, nprobs, mmax_rows, nmax_cols, st);
    if (mmax_rows <= kSmallRows && nmax_cols <= kSmallCols) return gemm64_warp<4>(probs, nprobs, mmax_rows, nmax_cols, st);
    // 32-row / 32-column tiles when the problems are that small
    const int wm = mmax_rows <= 32 ? 1 : 2, wn = nmax_cols <= 32 ? 1 : 2;
    const int bm = 32 * wm, bn = 32 * wn;
    const int tilesN = (nmax_cols + bn - 1) / bn, tilesM = (mmax_rows + bm - 1) / bm;
    for (int p0 = 0; p0 < nprobs; p0 += 65535) {
        const int np = (nprobs - p0 < 65535) ? nprobs - p0 : 65535;
        dim3 grid((unsigned)tilesN * tilesM, np);
        if (wm == 1 && wn == 1) k_gemm64<1, 1><<<grid, 32, 0, st>>>(probs + p0, tilesN);
        else if (wm == 1) k_gemm64<1, 2><<<grid, 64, 0, st>>>(probs + p0, tilesN);
        else if (wn == 1) k_gemm64<2, 1><<<grid, 64, 0, st>>>(probs + p0, tilesN);
        else k_gemm64<2, 2><<<grid, 128, 0, st>>>(probs + p0, tilesN);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
#endif
}

}  // namespace BDC_NS
