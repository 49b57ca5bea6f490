// Bidiagonalization of a matrix held on chip (Sec. 4.1, FP64), and the QR
// panels (Sec. 4.3).
//
// The blocked reduction (bdc_dense.cu) passes over the trailing matrix twice
// per column step and separates its phases by grid barriers.  When the matrix
// fits the SMs' shared memory (about 30 MB on 152 SMs) k_gebd2_resident loads
// it once, keeps a set of rows per CTA, applies every reflector pair at once
// (no panels V, X, Y, U, no trailing product) and needs two barriers a step.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "bdc_dense.cuh"

namespace bdc {

namespace {

// All CTAs of a cooperative launch wait until `target` arrivals have been
// counted (a counter that only grows: no reset, no generation); one thread
// arrives and polls.  ORDERED: what any thread of the grid wrote before is
// visible after (the arrival releases, the poll acquires, and the CTA's
// barriers carry both to its other threads).  Not ORDERED: only a hint that
// the other CTAs have got here, for readers of slots (below).  152 CTAs of
// 128 threads: 2480 cycles ordered, 1620 as a hint, 3260 with full fences
// around it; one thread polling per CTA matters: a flag per CTA polled by as
// many threads took 5000 to 14000.  The wait is bounded (kBarNs); false when
// it gave up here or elsewhere.
// meanwhile() runs on warp 0, thread LEAD arrives and polls.
template <bool ORDERED, int LEAD, typename F>
__device__ __forceinline__ bool grid_wait(GridBar *gb, unsigned target, F meanwhile) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x < 32) meanwhile();
    if (threadIdx.x == LEAD) {
        unsigned v;
        int ok = 1;
        auto poll = [&] {
            if (ORDERED) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&gb->mono) : "memory");
            else asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&gb->mono) : "memory");
        };
        if (ORDERED) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&gb->mono) : "memory");
        else asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(&gb->mono) : "memory");
        poll();
        if ((int)(v - target) < 0) {
            const unsigned long long t0 = gtime();
            unsigned spins = 0;
            do {
                poll();
                if ((++spins & 255u) == 0) {
                    if (*(volatile int *)&gb->err) { ok = 0; break; }
                    if (gtime() - t0 > kBarNs) {
                        atomicExch(&gb->err, 1);
                        ok = 0;
                        break;
                    }
                }
            } while ((int)(v - target) < 0);
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}
template <bool ORDERED = true>
__device__ __forceinline__ bool grid_wait(GridBar *gb, unsigned target) {
    return grid_wait<ORDERED, 0>(gb, target, [] {});
}

// Householder reflector from alpha and ||x_2..||^2 = sig2 (LAPACK's sign
// convention): beta = -sign(alpha) ||x||, tau = (beta - alpha) / beta, the
// vector's tail scaled by 1 / (alpha - beta); sig2 = 0 gives tau = 0 (H = I).
// On the critical path of every step, and every FP64 instruction of a warp
// takes 64 cycles here: 17 of them instead of the about 40 of a library
// square root and two divisions (a step at n = 64: 2 x 2300 -> 2 x 1450 cycles
// in this part).  With y the hardware estimate of 1 / sqrt(s) and r = 1 - s
// y^2 (at most 2^-19.0 measured over [1, 4)), the binomial series sqrt(s) = s y
// (1 - r)^(-1/2) = s y (1 + r/2 + 3 r^2/8 + 5 r^3/16 ...) leaves 2^-58 and a
// Newton step on nrm^2 = s the rounding of the last bit; the quotients are
// quot()'s (geometric series).  Outside 2^-900..2^900 the library calls.
__device__ __forceinline__ double reflector_fast(double alpha, double sig2, double &tau, double &beta) {
    if (__double_as_longlong(sig2) == 0) {
        tau = 0.0;
        beta = alpha;
        return 0.0;
    }
    const double s = fma(alpha, alpha, sig2);
    const long long sb = __double_as_longlong(s);
    const bool neg = __double_as_longlong(alpha) > (long long)0x8000000000000000ull &&
                     __double_as_longlong(alpha) < 0;       // (alpha = -0 counts as positive, as in k_geqr2)
    if (sb < (123ll << 52) || sb > (1923ll << 52)) {       // also NaN, infinity
        const double nrm = sqrt(s);
        beta = neg ? nrm : -nrm;
        tau = (beta - alpha) / beta;
        return 1.0 / (alpha - beta);
    }
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(s));
    const double g = s * y;
    const double r = fma(-g, y, 1.0);
    const double q = fma(0.375, r, 0.5) * r;
    double nrm = fma(g, q, g);
    nrm = fma(fma(-nrm, nrm, s), 0.5 * y, nrm);             // one residual step: the last bit
    beta = neg ? nrm : -nrm;
    const double D = alpha - beta;                          // no cancellation: the signs differ
    tau = quot(fabs(D), nrm);
    double z;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(z) : "d"(D));
    const double e = fma(-D, z, 1.0);
    return fma(z, fma(e, e, e), z);
}

// ---- exchange between CTAs without fences
// A slot is 16 bytes: the two halves of a double, each beside the step
// number that wrote it, so that a reader knows from the slot itself whether
// the value is there.  The CTAs wait for one another by an unordered
// grid_wait and then read: the rare slot that is still on its way is read
// again.  (Polling the slots alone, without that wait, kept L2 busy with 128
// threads a CTA: a 333 x 333 step took 18000 cycles, 16400 with the wait.)
// Each 8-byte half is written and read as one access.
typedef ulonglong2 Slot;

__device__ __forceinline__ void slot_put(Slot *p, double v, unsigned tag) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"((b & 0xffffffffull) | t),
                 "l"((b >> 32) | t)
                 : "memory");
}

__device__ __forceinline__ Slot slot_load(const Slot *p) {
    Slot s;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(s.x), "=l"(s.y) : "l"(p) : "memory");
    return s;
}

// K slots at once (all loads in flight together), polled
// until each carries `tag`.  Bounded: after kBarNs, or when another wait of
// the grid gave up, sets the error word and *s_err and returns.
// A null p[k] is skipped (v[k] = 0).
template <int K>
__device__ __forceinline__ void slot_get(const Slot *(&p)[K], unsigned tag, double (&v)[K], GridBar *gb,
                                         int *s_err) {
    const unsigned long long want = (unsigned long long)tag << 32;
    unsigned spins = 0;
    unsigned long long t0 = 0;
    for (;;) {
        Slot s[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            s[k] = Slot{want, want};
            if (p[k]) s[k] = slot_load(p[k]);
        }
        bool ok = true;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            ok = ok && (unsigned)(s[k].x >> 32) == tag && (unsigned)(s[k].y >> 32) == tag;
            v[k] = __longlong_as_double((long long)((s[k].x & 0xffffffffull) | (s[k].y << 32)));
        }
        if (ok) return;
        if ((++spins & 127u) == 0) {
            if (t0 == 0) t0 = gtime();
            if (*(volatile int *)&gb->err || gtime() - t0 > kBarNs) {
                atomicExch(&gb->err, 1);
                *(volatile int *)s_err = 1;
                return;
            }
        }
    }
}

constexpr int NT = 128;            // threads per CTA: one warp per SM sub-partition
constexpr int kRedLd = NT + 8;     // row stride of the reduction buffer
constexpr int LR = 12;             // rows of a CTA handled together at most (1500 x 1100: 17.3 ms at 8, 16.5 at 12)

// f(integral_constant<K>) for K = k in 1..LR: straight-line code per row
// count, so that the loads, FMAs and stores of all rows are scheduled
// together (one warp per scheduler: nothing else hides a latency; with a
// test per row the passes ran at a third of this rate)
template <int LR, typename F>
__device__ __forceinline__ void rows_dispatch(int k, F f) {
    if constexpr (LR >= 1) {
        if (k == LR) f(std::integral_constant<int, LR>{});
        else rows_dispatch<LR - 1>(k, f);
    }
}

// A -= v y^T on K rows and this thread's columns i + 1.., red[q][t] = this
// thread's part of A r over the columns i + 2..
template <int K>
__device__ __forceinline__ void pass_left(double *W, int ldw, const double *vv, const double *sy, const double *sr,
                                          int i, int n, int t, double *red) {
    double acc[K], v[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        acc[q] = 0.0;
        v[q] = -vv[q];
    }
    int c = i + 1 + t;
    if constexpr (K <= 4) {     // two columns at once
        for (; c + NT < n; c += 2 * NT) {
            const double y0 = sy[c], y1 = sy[c + NT], r0 = (c > i + 1) ? sr[c] : 0.0, r1 = sr[c + NT];
            double x[K], z[K];
#pragma unroll
            for (int q = 0; q < K; ++q) {
                x[q] = W[(size_t)q * ldw + c];
                z[q] = W[(size_t)q * ldw + c + NT];
            }
#pragma unroll
            for (int q = 0; q < K; ++q) {
                x[q] = fma(v[q], y0, x[q]);
                z[q] = fma(v[q], y1, z[q]);
            }
#pragma unroll
            for (int q = 0; q < K; ++q) acc[q] = fma(x[q], r0, acc[q]);
#pragma unroll
            for (int q = 0; q < K; ++q) {
                W[(size_t)q * ldw + c] = x[q];
                W[(size_t)q * ldw + c + NT] = z[q];
            }
#pragma unroll
            for (int q = 0; q < K; ++q) acc[q] = fma(z[q], r1, acc[q]);
        }
    }
    for (; c < n; c += NT) {
        const double y0 = sy[c], r0 = (c > i + 1) ? sr[c] : 0.0;
        double x[K];
#pragma unroll
        for (int q = 0; q < K; ++q) x[q] = W[(size_t)q * ldw + c];
#pragma unroll
        for (int q = 0; q < K; ++q) x[q] = fma(v[q], y0, x[q]);
#pragma unroll
        for (int q = 0; q < K; ++q) {
            W[(size_t)q * ldw + c] = x[q];
            acc[q] = fma(x[q], r0, acc[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < K; ++q) red[q * kRedLd + t] = acc[q];
}

// A -= x u^T on K rows and this thread's columns, su[c] = u_c; sums of A^T a
// over the rows: from 0 (first) or sum[c], into sum[c] or (gp) the slots
template <int K>
__device__ __forceinline__ void pass_right(double *W, int ldw, const double *xv, const double *av, const double *su,
                                           double *sum, bool first, Slot *gp, int i, int n, int t,
                                           unsigned tag) {
    double xr[K], ar[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        xr[q] = -xv[q];
        ar[q] = av[q];
    }
    int c = i + 1 + t;
    if constexpr (K <= 4) {
        for (; c + NT < n; c += 2 * NT) {
            const double u0 = su[c], u1 = su[c + NT];
            double x[K], z[K];
            double s0 = first ? 0.0 : sum[c], s1 = first ? 0.0 : sum[c + NT];
#pragma unroll
            for (int q = 0; q < K; ++q) {
                x[q] = W[(size_t)q * ldw + c];
                z[q] = W[(size_t)q * ldw + c + NT];
            }
#pragma unroll
            for (int q = 0; q < K; ++q) {
                x[q] = fma(xr[q], u0, x[q]);
                z[q] = fma(xr[q], u1, z[q]);
            }
#pragma unroll
            for (int q = 0; q < K; ++q) {
                s0 = fma(ar[q], x[q], s0);
                s1 = fma(ar[q], z[q], s1);
            }
#pragma unroll
            for (int q = 0; q < K; ++q) {
                W[(size_t)q * ldw + c] = x[q];
                W[(size_t)q * ldw + c + NT] = z[q];
            }
            if (gp) {
                slot_put(gp + c, s0, tag);
                slot_put(gp + c + NT, s1, tag);
            } else {
                sum[c] = s0;
                sum[c + NT] = s1;
            }
        }
    }
    for (; c < n; c += NT) {
        const double u0 = su[c];
        double x[K];
        double s0 = first ? 0.0 : sum[c];
#pragma unroll
        for (int q = 0; q < K; ++q) x[q] = W[(size_t)q * ldw + c];
#pragma unroll
        for (int q = 0; q < K; ++q) x[q] = fma(xr[q], u0, x[q]);
#pragma unroll
        for (int q = 0; q < K; ++q) {
            W[(size_t)q * ldw + c] = x[q];
            s0 = fma(ar[q], x[q], s0);
        }
        if (gp) slot_put(gp + c, s0, tag);
        else sum[c] = s0;
    }
}

struct Gebd2Args {
    double *A;
    int lda, m, n;
    double *d, *e, *tauq, *taup;
    Slot *gp;                      // [grid][n]: per-CTA partial sums of A^T a (column i: of a^T a)
    Slot *row, *gs;                // [2][n] top row, by the step's parity; [n] sums of g over the CTAs
    GridBar *bar;
    unsigned base;                 // arrivals before this launch
};

// CTA g holds rows g, g + G, g + 2G, ... (cyclic: the rows that drop out
// step by step leave every CTA with the same share) in shared memory, row
// major.  With a = column i of the current matrix, step i is
//   Y phase (a block of columns per CTA): g_c = sum over CTAs of A[:, c]^T a
//     (tail rows), sig2 = the same for a itself -> H_i's scalars (every CTA
//     forms them, while the sums g travel)
//   X phase (own rows): y_c = A[i, c] + sc g_c, row i: r_c = A[i, c] - tau
//     y_c (every CTA, all columns); v = tau sc a; one pass A -= v y^T with h =
//     A r; block reduction of h and ||r||^2 -> G_i's scalars; x = pi A u with u
//     = [1; scr r]; next column a' = A[:, i+1] - x; one pass A -= x u^T with the
//     partial sums of A^T a' and a'^T a' for step i + 1, and the next top row
// The products are taken with the unscaled a and r, so that no phase waits
// for a norm.  Four FMAs per entry and step; FP64 runs at two lanes per
// clock and SM, so four warps fill the pipe and the block reduction (one add
// per thread and row) is kept small by them.  The phases exchange their
// vectors through slots (above).  One buffer of the sums is enough: a CTA
// writes its sums of step i + 1 after it has the g of every column of step i,
// which their owners sent after reading all sums of step i (of column i, which
// all read, no later sum is written); and an owner sends step i + 1's g after
// the sums of every CTA, which each sent after reading all of step i's g.  The
// top row has two: all read step i's in the X phase, where its next owner
// writes step i + 1's, over that of step i - 1, which all have read before
// they arrived in the Y phase of step i.
// What bounds it: the two exchanges (about 3500 cycles each) and the
// dependent FP64 chains of a step (64 cycles an operation), above n ~ 1000
// the FP64 pipe.  333 x 333: 18.9 ms (blocked panels, seven barriers a step)
// -> 2.6 ms; 1100 x 1100: 13.9 ms; 1500 x 1100: 82 -> 15.7 ms.  Sending y and
// r from the owners of the columns, each after its own H_i scalars, put those
// (1450 cycles) in front of the exchange instead of beside it: 2.8, 14.6 and
// 16.3 ms.
__global__ void __launch_bounds__(NT, 1) k_gebd2_resident(Gebd2Args a) {
    extern __shared__ double smem[];
    __shared__ int s_err;
    __shared__ double s_alpha, s_sc, s_tau;
    const int G = gridDim.x, g = blockIdx.x, t = threadIdx.x;
    const int m = a.m, n = a.n, ldw = a.n;
    const int lr = (m - g + G - 1) / G;             // own rows (g < G <= m)
    const int lrmax = (m + G - 1) / G;
    double *W = smem;                               // [lr][ldw]
    double *sy = W + (size_t)lrmax * ldw;           // this thread's columns of y, r (written and read by one thread)
    double *sr = sy + ldw;
    double *red = sr + ldw;                         // [LR + 1][kRedLd]
    double *av = red + (LR + 1) * kRedLd;           // [lrmax] a, x, v of the own rows; h sums
    double *xv = av + lrmax, *vv = xv + lrmax, *hs = vv + lrmax;
    double *A = a.A;
    const size_t lda = a.lda;

    if (t == 0) s_err = 0;
    for (int c = t; c < n; c += NT)
        for (int l = 0; l < lr; ++l) W[(size_t)l * ldw + c] = A[(size_t)c * lda + g + (size_t)G * l];
    // clear the slots' step numbers
    const Slot zero = {0ull, 0ull};
    for (int c = t; c < n; c += NT) a.gp[(size_t)g * ldw + c] = zero;
    for (int c = g * NT + t; c < n; c += G * NT) a.row[c] = a.row[n + c] = a.gs[c] = zero;
    unsigned target = a.base + G;
    if (!grid_wait(a.bar, target)) return;
    for (int l = t; l < lr; l += NT) av[l] = W[(size_t)l * ldw];
    __syncthreads();
    for (int c = t; c < n; c += NT) {               // sums of step 0
        double s = 0.0;
        for (int l = (g == 0); l < lr; ++l) s = fma(av[l], W[(size_t)l * ldw + c], s);
        if (g == 0) slot_put(a.row + c, W[c], 1u);
        slot_put(a.gp + (size_t)g * ldw + c, s, 1u);
    }
    if (!grid_wait<false>(a.bar, target += G)) return;

    for (int i = 0; i < n; ++i) {
        const unsigned tag = (unsigned)i + 1u;
        // ---- Y phase
        const int ncol = n - 1 - i, cb = (ncol + G - 1) / G;
        const int c0 = i + 1 + g * cb, nc = max(0, min(cb, n - c0));
        const Slot *row = a.row + (size_t)(i & 1) * n;
        // sums over the CTAs of nc columns and of column i (slot nc); every
        // CTA sums column i, in the same order (the cut follows cb, not nc)
        int sp = 1;
        while (sp < cb + 1) sp <<= 1;               // slots per pass (power of two, at most 32)
        if (sp > 32) sp = 32;
        const bool one = cb + 1 <= sp;
        {
            const int slots = nc + 1;
            const int sub = t / sp, subs = NT / sp;
            for (int s0 = 0; s0 < slots; s0 += sp) {
                const int s = s0 + (t & (sp - 1));
                double v0 = 0.0;
                // eight CTAs' slots per round (one round for most sizes), and
                // alpha
                const Slot *p = a.gp + (s < nc ? c0 + s : i);
                for (int k = sub; k < G; k += 8 * subs) {
                    const Slot *q[9];
                    double v[9];
#pragma unroll
                    for (int j = 0; j < 8; ++j) q[j] = k + j * subs < G && s < slots ? p + (size_t)(k + j * subs) * ldw : nullptr;
                    q[8] = t == 0 ? row + i : nullptr;
                    slot_get<9>(q, tag, v, a.bar, &s_err);
                    if (t == 0) s_alpha = v[8];
                    v0 += v[0];
#pragma unroll
                    for (int j = 1; j < 8; ++j)
                        if (k + j * subs < G) v0 += v[j];
                }
                for (int o = sp; o < 32; o <<= 1) v0 += __shfl_xor_sync(0xffffffffu, v0, o);
                if (s0 > 0) __syncthreads();
                if ((t & 31) < sp) red[(t >> 5) * 32 + (t & 31)] = v0;
                __syncthreads();
                if (t < sp && s0 + t < slots) {
                    const double gs = (red[t] + red[32 + t]) + (red[64 + t] + red[96 + t]);
                    if (s0 + t < nc) slot_put(a.gs + c0 + s0 + t, gs, tag);
                    else if (!one) sy[0] = gs;
                }
            }
        }
        // H_i's scalars while the other CTAs' sums are on their way
        if (!grid_wait<false, 32>(a.bar, target += G, [&] {
                const double sig2 = one ? (red[nc] + red[32 + nc]) + (red[64 + nc] + red[96 + nc]) : sy[0];
                double tau, beta;
                const double sc = reflector_fast(s_alpha, sig2, tau, beta);
                if (t == 0) {
                    s_sc = sc;
                    s_tau = tau;
                    if (g == 0) {
                        a.d[i] = beta;
                        a.tauq[i] = tau;
                        A[(size_t)i * lda + i] = beta;
                    }
                }
            }))
            return;
        const double sc = s_sc, tau = s_tau;
        // ---- X phase
        const int l0 = (i < g) ? 0 : (i - g) / G + 1;   // first own row below i
        const bool more = i + 1 < n;
        for (int c = i + 1 + t; c < n; c += 4 * NT) {
            // four columns of g and row i per round
            const Slot *q[8];
            double v[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                q[2 * j] = c + j * NT < n ? a.gs + c + j * NT : nullptr;
                q[2 * j + 1] = c + j * NT < n ? row + c + j * NT : nullptr;
            }
            slot_get<8>(q, tag, v, a.bar, &s_err);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c + j * NT < n) {
                    const double y = fma(sc, v[2 * j], v[2 * j + 1]);
                    sy[c + j * NT] = y;
                    sr[c + j * NT] = fma(-tau, y, v[2 * j + 1]);
                }
        }
        for (int l = l0 + t; l < lr; l += NT) {
            const double v = sc * av[l];
            vv[l] = tau * v;
            A[(size_t)i * lda + g + (size_t)G * l] = v;
        }
        __syncthreads();
        if (s_err || !more) return;                 // a wait gave up (uniform: read after the barrier), or done
        // A -= v y^T with the products h = A r (the tail of row i: columns
        // i + 2...) in chunks of LR rows; slot LR of the last chunk: ||r||^2
        double pi, betr;
        // equal chunks of at most LR rows
        const int chunks = max(1, (lr - l0 + LR - 1) / LR), rows0 = (lr - l0 + chunks - 1) / chunks;
        for (int b0 = l0;; b0 += rows0) {
            const int nq = max(0, min(rows0, lr - b0));   // rows of this chunk
            const bool lastc = b0 + rows0 >= lr;
            double nrm = 0.0;                           // slot nq of the reduction: ||r||^2 (last chunk)
            if (lastc)
                for (int c = i + 1 + t; c < n; c += NT) {
                    const double rt = (c > i + 1) ? sr[c] : 0.0;
                    nrm = fma(rt, rt, nrm);
                }
            red[nq * kRedLd + t] = nrm;
            rows_dispatch<LR>(nq, [&](auto K) {
                pass_left<decltype(K)::value>(W + (size_t)b0 * ldw, ldw, vv + b0, sy, sr, i, n, t, red);
            });
            __syncthreads();
            // block reduction: P lanes per row (all the rows at once)
            const int rows = nq + 1;
            const int P = rows <= 4 ? 32 : rows <= 8 ? 16 : 8;
            {
                const int q = t / P, p = t & (P - 1);
                double s0 = 0.0;
                if (q < rows) {
                    s0 = red[q * kRedLd + p];
                    for (int k = p + P; k < NT; k += P) s0 += red[q * kRedLd + k];
                }
                for (int o = P >> 1; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
                if (q < rows && p == 0) hs[q == nq ? lrmax : b0 + q] = s0;
            }
            __syncthreads();
            if (lastc) break;
        }
        const double scr = reflector_fast(sr[i + 1], hs[lrmax], pi, betr);
        for (int l = l0 + t; l < lr; l += NT) {
            const double w = W[(size_t)l * ldw + i + 1];
            const double x = pi * fma(scr, hs[l], w);
            xv[l] = x;
            av[l] = w - x;
        }
        if (g == 0 && t == 0) {
            a.e[i] = betr;
            a.taup[i] = pi;
            A[(size_t)(i + 1) * lda + i] = betr;
        }
        __syncthreads();
        // A -= x u^T, the partial sums of the next step, its top row
        const bool topmine = l0 < lr && g + G * l0 == i + 1;
        const int l1 = l0 + (topmine ? 1 : 0);
        double *ug = g == i % G ? A + i : nullptr;       // this CTA stores row i's reflector
        const double xt = topmine ? xv[l0] : 0.0;
        for (int c = i + 1 + t; c < n; c += NT) {
            const double u = (c == i + 1) ? 1.0 : scr * sr[c];
            if (ug && c > i + 1) ug[(size_t)c * lda] = u;
            if (topmine) slot_put(a.row + (size_t)((i + 1) & 1) * n + c, fma(-xt, u, W[(size_t)l0 * ldw + c]), tag + 1u);
            sr[c] = u;
            if (l1 >= lr) slot_put(a.gp + (size_t)g * ldw + c, 0.0, tag + 1u);
        }
        const int chunks1 = max(1, (lr - l1 + LR - 1) / LR), rows1 = max(1, (lr - l1 + chunks1 - 1) / chunks1);
        for (int b0 = l1; b0 < lr; b0 += rows1) {
            const int nq = min(rows1, lr - b0);
            Slot *gp = b0 + rows1 >= lr ? a.gp + (size_t)g * ldw : nullptr;
            rows_dispatch<LR>(nq, [&](auto K) {
                pass_right<decltype(K)::value>(W + (size_t)b0 * ldw, ldw, xv + b0, av + b0, sr, sy, b0 == l1, gp, i, n,
                                               t, tag + 1u);
            });
        }
        if (!grid_wait<false>(a.bar, target += G)) return;
    }
}

// shared memory of a grid of G CTAs (bytes)
size_t res_smem(int m, int n, int G) {
    const size_t lr = (m + G - 1) / G, ldw = n;
    return sizeof(double) * (lr * ldw + 2 * ldw + (size_t)(LR + 1) * kRedLd + 4 * lr + 2);
}

struct DevInfo {
    int sms = 0, smem = 0;
};
DevInfo dev_info() {
    static std::mutex mu;
    static DevInfo cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return {};
    std::lock_guard<std::mutex> lk(mu);
    DevInfo &d = cache[dev];
    if (d.sms == 0) {
        cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&d.smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        d.smem -= 128;   // the kernels' static shared memory
    }
    return d;
}

// ------------------------------------------------------ blocked panel
// Panel of Algorithm 1 (labrd) on the m x n trailing matrix A, for matrices
// that do not fit on chip: nb column and row reflectors, the corrections of
// the not yet updated trailing matrix kept in V, X (m x b, ld m) and Y, U (n x
// b, ld n).  Four phases a step, separated by grid_wait:
//   P1  own rows: x_{i-1} (the products with r_{i-1} are sums of partial
//       products), column i: a_i
//   P2  a_i^T A over the trailing columns, V^T a_i, X^T a_i, a_i^T a_i
//   P3  own columns: y_i, row i: r_i; the scaled reflector v_i
//   P4  A r_i over the trailing rows, Y^T r_i, U^T r_i, r_i^T r_i
// The products take the unscaled a and r, so that no phase waits for a norm,
// and each norm is one more dot product.  P2 and P4 cut the flattened
// (columns x rows) space evenly over the grid's warps (a warp's range may
// span several columns; partial sums, at most kParts per result, are added by
// their reader), 16 warps an SM with 20 loads in flight a lane.
// What bounds it: P2 and P4 at the FP64 pipe and L2 (16 bytes a clock and SM
// at the pipe's two lanes): 65000 cycles each at n = 4096, of which
// 55000 are the FMAs at two a clock.  P1 and P3 are chains of FP64 operations and L2 trips,
// 10600 and 8500 cycles, and a barrier 3100.  FP64 instructions of a CTA's
// warps queue at the pipe (64 cycles each), so the scalars are one warp's and
// the short sums are cut so that few warps hold full ones.  4096 x 4096: 126 us
// a step behind seven barriers -> 84 at the first panel, 31 at order 1900;
// whole reduction 533 -> 178 ms.
constexpr int kLT = 512, kLW = kLT / 32, kParts = 32, kLb = 32;

struct Labrd2Args {
    double *A;
    int lda, m, n, nb;
    double *d, *e, *tauq, *taup;
    double *V, *X, *Y, *U;
    double *av, *rv;               // a_i (m), r_i (n)
    double *cpart, *hpart, *tpart; // partial sums: P2 (n + 2b + 1) x kParts, P4 rows ceil(m/32) x kParts x 32, P4 dots
    GridBar *bar;
    unsigned base;
};

// How `groups` results of `blocks` blocks each are cut over nw warps: every
// result in `parts` equal ranges of `size` blocks, so that readers know the
// count of partial sums; the count (a lane tries each) that leaves the warps
// with the fewest blocks, a range's start counted as two.
struct Cut {
    int parts, size;
};
__device__ __forceinline__ Cut cut_of(int groups, int blocks, int nw) {
    const int s = (threadIdx.x & 31) + 1, size = (blocks + s - 1) / s;
    const unsigned rounds = (unsigned)(groups * s + nw - 1) / (unsigned)nw;
    const unsigned cost = s <= blocks ? min(rounds * (unsigned)(size + 2), 0x3ffffffu) : 0x3ffffffu;
    const int parts = (int)(__reduce_min_sync(0xffffffffu, cost << 6 | (unsigned)s) & 63u);
    return Cut{parts, (blocks + parts - 1) / parts};
}
static_assert(kParts == 32, "a lane per count");

// x over four columns p[0..3] against y, entries [r0, r1) in lane steps of 32:
// four accumulators reduced together; lane 8 c ends with column c's sum
__device__ __forceinline__ double dot4(const double *const (&p)[4], const double *y, int r0, int r1, int lane) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    int r = r0 + lane;
    for (; r + 96 < r1; r += 128) {
        double yv[4], x[4][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) yv[k] = __ldcg(y + r + 32 * k);
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int k = 0; k < 4; ++k) x[c][k] = __ldcg(p[c] + r + 32 * k);
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int c = 0; c < 4; ++c) s[c] = fma(x[c][k], yv[k], s[c]);
    }
    for (; r < r1; r += 32) {
        const double yv = __ldcg(y + r);
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] = fma(__ldcg(p[c] + r), yv, s[c]);
    }
    // halves exchange two columns, quarters one: six adds instead of twenty
    const bool hi = lane & 16;
    double a0 = hi ? s[2] : s[0], a1 = hi ? s[3] : s[1];
    a0 += __shfl_xor_sync(0xffffffffu, hi ? s[0] : s[2], 16);
    a1 += __shfl_xor_sync(0xffffffffu, hi ? s[1] : s[3], 16);
    const bool q = lane & 8;
    double b = q ? a1 : a0;
    b += __shfl_xor_sync(0xffffffffu, q ? a0 : a1, 8);
    for (int o = 4; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
    return b;                      // lanes 8 c .. 8 c + 7: column (c >> 1) * 2 + (c & 1)
}

// the dot products of `count` vectors (ptr(k)) with y over [r0, r1), cut over
// the grid's warps; partial sums at part[k kParts + p]
template <typename F>
__device__ __forceinline__ void dots(int count, F ptr, const double *y, int r0, int r1, double *part, int gwarp, int nw,
                                     int lane) {
    const int groups = (count + 3) / 4, blocks = (r1 - r0 + 31) / 32;
    if (blocks <= 0) return;
    const Cut cut = cut_of(groups, blocks, nw);
    for (int u = gwarp; u < groups * cut.parts; u += nw) {
        const int g = u / cut.parts, q = u - g * cut.parts;
        const int b0 = q * cut.size, b1 = min(blocks, b0 + cut.size);
        const double *p[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) p[c] = ptr(min(4 * g + c, count - 1));
        const double s = dot4(p, y, r0 + 32 * b0, min(r1, r0 + 32 * b1), lane);   // (0 for an empty range)
        const int c = 4 * g + (lane >> 3);
        if ((lane & 7) == 0 && c < count) __stcg(part + (size_t)c * kParts + q, s);
    }
}
// the sums of results first .. first + count - 1 of dots(total, ..) into out,
// eight lanes each
__device__ __forceinline__ void dot_sums(const double *part, int total, int r0, int r1, int nw, int first, int count,
                                         double *out) {
    const int groups = (total + 3) / 4, blocks = (r1 - r0 + 31) / 32;
    const Cut cut = blocks > 0 ? cut_of(groups, blocks, nw) : Cut{0, 0};
    const int l = threadIdx.x & 7;
    for (int k0 = 0; k0 < count; k0 += kLT / 8) {
        const int k = k0 + threadIdx.x / 8;
        if (k0 + (int)(threadIdx.x >> 5) * 4 >= count) break;   // whole warps
        double v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = k < count && l + 8 * q < cut.parts ? __ldcg(part + (size_t)(first + k) * kParts + l + 8 * q) : 0.0;
        double s = v[0];
#pragma unroll
        for (int q = 1; q < 4; ++q)
            if (8 * q < cut.parts) s += v[q];
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (l == 0 && k < count) out[k] = s;
    }
}

// A panel phase's own 32 rows (or columns) r, a lane each: sums over the
// panel's earlier columns j of P[r, j] f1[j] + Q[r, j] f2[j] and of P[r, j]
// f3[j] + Q[r, j] f4[j], P's cp and Q's cq columns split over eight warps
// (loaded before the factors are known); the partial sums of a product over
// four more warps.
struct Rows {
    double p[4], q[4], h[8];
    __device__ __forceinline__ void load(const double *P, int cp, const double *Q, int cq, int ld, int r, bool ok,
                                         const double *hp, size_t hstride, int parts, int warp) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int j = warp + 8 * k;
            p[k] = ok && warp < 8 && j < cp ? __ldcg(P + (size_t)j * ld + r) : 0.0;
            q[k] = ok && warp < 8 && j < cq ? __ldcg(Q + (size_t)j * ld + r) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int z = warp - 8 + 4 * k;
            h[k] = ok && warp >= 8 && warp < 12 && z < parts ? __ldcg(hp + z * hstride) : 0.0;
        }
    }
    __device__ __forceinline__ void sum(int cp, int cq, const double *f1, const double *f2, const double *f3,
                                        const double *f4, int parts, double (*red)[2][32], int warp, int lane) {
        if (warp < 8) {
            double s0 = 0.0, s1 = 0.0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = warp + 8 * k;
                if (j < cp) { s0 = fma(p[k], f1[j], s0); s1 = fma(p[k], f3[j], s1); }
                if (j < cq) { s0 = fma(q[k], f2[j], s0); s1 = fma(q[k], f4[j], s1); }
            }
            red[warp][0][lane] = s0;
            red[warp][1][lane] = s1;
        } else if (warp < 12) {
            double s = h[0];
#pragma unroll
            for (int k = 1; k < 8; ++k)
                if (warp - 8 + 4 * k < parts) s += h[k];
            red[warp][0][lane] = s;
        }
    }
};
__device__ __forceinline__ double red8(const double (*red)[2][32], int k, int lane) {
    return ((red[0][k][lane] + red[1][k][lane]) + (red[2][k][lane] + red[3][k][lane])) +
           ((red[4][k][lane] + red[5][k][lane]) + (red[6][k][lane] + red[7][k][lane]));
}
__device__ __forceinline__ double red4(const double (*red)[2][32], int lane) {
    return (red[8][0][lane] + red[9][0][lane]) + (red[10][0][lane] + red[11][0][lane]);
}

__global__ void __launch_bounds__(kLT, 1) k_labrd_panel(Labrd2Args a) {
    __shared__ double s_t[2 * kLb + 2], s_1[kLb], s_2[kLb], s_3[kLb], s_4[kLb];
    __shared__ double s_red[12][2][32], s_x[32], s_c[2];
    const int G = gridDim.x, g = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int m = a.m, n = a.n, nw = G * kLW, gwarp = warp * G + g;   // consecutive ranges on different SMs
    double *A = a.A, *V = a.V, *X = a.X, *Y = a.Y, *U = a.U;
    const size_t lda = a.lda;
    unsigned target = a.base;

    for (int i = 0;; ++i) {
        const bool last = i == a.nb;
        // ---- P1
        {
            const int rb = (m - i + G - 1) / G, ra = i + g * rb, rz = min(m, ra + rb);
            const int cblocks = i > 0 ? (n - i - 1 + 15) / 16 : 0;           // P4's cut of step i - 1
            const Cut hc = cblocks > 0 ? cut_of((m - i + 31) / 32, cblocks, nw) : Cut{0, 0};
            const int cp = i, cq = max(0, i - 1);
            Rows rows;
            double a0 = 0.0;
            auto load = [&](int r0) {
                const int r = r0 + lane, rg = (r - i) >> 5, rl = (r - i) & 31;
                rows.load(V, cp, X, cq, m, r, r < rz, a.hpart + (size_t)rg * kParts * 32 + rl, 32, hc.parts, warp);
                if (warp < 2 && r < rz) a0 = __ldcg(A + (size_t)min(i, n - 1) * lda + r);
            };
            load(ra);
            double pi = 0.0, scr = 0.0, betr = 0.0;
            if (i > 0) {
                const int nd = 2 * i;
                const double alr = __ldcg(a.rv + i);
                if (t >= 384 && t < 384 + i) s_3[t - 384] = __ldcg(Y + (size_t)(t - 384) * n + i);
                if (t >= 448 && t < 448 + i - 1) s_4[t - 448] = __ldcg(U + (size_t)(t - 448) * n + i);
                dot_sums(a.tpart, nd, i + 1, n, nw, 0, nd, s_t);
                __syncthreads();
                if (warp == 0) {   // one warp: each further one would take its turn at the FP64 pipe
                    scr = reflector_fast(alr, s_t[nd - 1], pi, betr);
                    if (lane < i) s_1[lane] = fma(scr, s_t[lane], s_3[lane]);
                    if (lane < i - 1) s_2[lane] = fma(scr, s_t[i + lane], s_4[lane]);
                    if (lane == 0) { s_c[0] = scr; s_c[1] = betr; }
                }
            }
            for (int r0 = ra; r0 < rz; r0 += 32) {
                const int r = r0 + lane;
                if (r0 > ra) load(r0);
                __syncthreads();   // s_1 .. s_4, s_c; s_red, s_x of the previous rows
                if (i > 0) rows.sum(cp, cq, s_1, s_2, s_3, s_4, hc.parts, s_red, warp, lane);
                __syncthreads();
                double sa = 0.0;
                if (i > 0 && warp == 0) {
                    const double x = pi * (fma(scr, red4(s_red, lane), a0) - red8(s_red, 0, lane));
                    s_x[lane] = x;
                    if (r < rz) __stcg(X + (size_t)(i - 1) * m + r, x);
                } else if (i > 0 && warp == 1) {
                    sa = red8(s_red, 1, lane);
                }
                __syncthreads();
                if (warp == 1 && r < rz && !last) __stcg(a.av + r, i > 0 ? (a0 - sa) - s_x[lane] : a0);
            }
            // the row reflector i - 1
            if (i > 0) {
                if (ra >= rz) __syncthreads();   // s_c
                scr = s_c[0];
                betr = s_c[1];
                const int cb = (n - i + G - 1) / G, c0 = i + g * cb;
                for (int c = c0 + t - 64; c < min(n, c0 + cb); c += kLT - 64) {
                    if (c < c0) continue;
                    const double u = c == i ? 1.0 : scr * __ldcg(a.rv + c);
                    __stcg(U + (size_t)(i - 1) * n + c, u);
                    A[(size_t)c * lda + i - 1] = c == i ? betr : u;
                }
                if (g == 0 && t == 0) {
                    a.e[i - 1] = betr;
                    a.taup[i - 1] = pi;
                }
            }
        }
        if (last) return;
        if (!grid_wait(a.bar, target += G)) return;
        // ---- P2
        const int nc = n - 1 - i, n2 = nc + 2 * i + 1;
        dots(n2, [&](int k) {
                return (const double *)(k < nc ? A + (size_t)(i + 1 + k) * lda
                                        : k < nc + i ? V + (size_t)(k - nc) * m
                                        : k < nc + 2 * i ? X + (size_t)(k - nc - i) * m : a.av);
            }, a.av, i + 1, m, a.cpart, gwarp, nw, lane);
        if (!grid_wait(a.bar, target += G)) return;
        // ---- P3
        {
            const int nd = 2 * i + 1, blocks = (m - i - 1 + 31) / 32;
            const int cb = (nc + G - 1) / G, ca = i + 1 + g * cb, cz = min(n, ca + cb);
            const Cut gc = blocks > 0 ? cut_of((n2 + 3) / 4, blocks, nw) : Cut{0, 0};
            Rows rows;
            double a0 = 0.0;
            auto load = [&](int c0) {
                const int c = c0 + lane;
                rows.load(Y, i, U, i, n, c, c < cz, a.cpart + (size_t)(c - i - 1) * kParts, 1, gc.parts, warp);
                if (warp < 2 && c < cz) a0 = __ldcg(A + (size_t)c * lda + i);
            };
            load(ca);
            const double alpha = __ldcg(a.av + i);
            if (t >= 384 && t < 384 + i) s_3[t - 384] = __ldcg(V + (size_t)(t - 384) * m + i);
            if (t >= 448 && t < 448 + i) s_4[t - 448] = __ldcg(X + (size_t)(t - 448) * m + i);
            dot_sums(a.cpart, n2, i + 1, m, nw, nc, nd, s_t);
            __syncthreads();
            double tau = 0.0, beta = 0.0, sc = 0.0;
            if (warp == 0) {
                sc = reflector_fast(alpha, s_t[2 * i], tau, beta);
                if (lane < i) {
                    s_1[lane] = fma(sc, s_t[lane], s_3[lane]);
                    s_2[lane] = fma(sc, s_t[i + lane], s_4[lane]);
                }
                if (lane == 0) s_c[0] = sc;
            }
            for (int c0 = ca; c0 < cz; c0 += 32) {
                const int c = c0 + lane;
                if (c0 > ca) load(c0);
                __syncthreads();
                rows.sum(i, i, s_1, s_2, s_3, s_4, gc.parts, s_red, warp, lane);
                __syncthreads();
                double sr = 0.0;
                if (warp == 0) {
                    const double y = tau * (fma(sc, red4(s_red, lane), a0) - red8(s_red, 0, lane));
                    s_x[lane] = y;
                    if (c < cz) __stcg(Y + (size_t)i * n + c, y);
                } else if (warp == 1) {
                    sr = red8(s_red, 1, lane);
                }
                __syncthreads();
                if (warp == 1 && c < cz) __stcg(a.rv + c, (a0 - sr) - s_x[lane]);
            }
            // the column reflector i
            if (ca >= cz) __syncthreads();   // s_c
            sc = s_c[0];
            const int rb = (m - i - 1 + G - 1) / G, ra = i + 1 + g * rb;
            for (int r = ra + t - 64; r < min(m, ra + rb); r += kLT - 64) {
                if (r < ra) continue;
                const double v = sc * __ldcg(a.av + r);
                __stcg(V + (size_t)i * m + r, v);
                A[(size_t)i * lda + r] = v;
            }
            if (g == 0 && t == 0) {
                a.d[i] = beta;
                a.tauq[i] = tau;
                A[(size_t)i * lda + i] = beta;
            }
            if (nc == 0) return;   // the last column of the matrix: no row reflector
        }
        if (!grid_wait(a.bar, target += G)) return;
        // ---- P4: rows i + 1 .. by groups of 32 (a row per lane), columns i + 2 .. by 16
        {
            const int groups = (m - i - 1 + 31) / 32, cblocks = (n - i - 2 + 15) / 16;
            if (groups > 0 && cblocks > 0) {
                const Cut cut = cut_of(groups, cblocks, nw);
                for (int u = gwarp; u < groups * cut.parts; u += nw) {
                    const int rg = u / cut.parts, q = u - rg * cut.parts;
                    const int b0 = q * cut.size, b1 = min(cblocks, b0 + cut.size);
                    const int r = i + 1 + 32 * rg + lane, ce = min(n, i + 2 + 16 * b1);
                    const double *p = A + min(r, m - 1);
                    double s0 = 0.0, s1 = 0.0;
                    for (int c = i + 2 + 16 * b0; c < ce; c += 16) {
                        const double rr = c + (lane & 15) < ce ? __ldcg(a.rv + c + (lane & 15)) : 0.0;
                        double x[16];
#pragma unroll
                        for (int k = 0; k < 16; ++k) x[k] = __ldcg(p + (size_t)min(c + k, ce - 1) * lda);
#pragma unroll
                        for (int k = 0; k < 16; k += 2) {
                            s0 = fma(x[k], __shfl_sync(0xffffffffu, rr, k), s0);
                            s1 = fma(x[k + 1], __shfl_sync(0xffffffffu, rr, k + 1), s1);
                        }
                    }
                    __stcg(a.hpart + ((size_t)rg * kParts + q) * 32 + lane, s0 + s1);
                }
            }
            dots(2 * i + 2, [&](int k) {
                    return (const double *)(k <= i ? Y + (size_t)k * n : k <= 2 * i ? U + (size_t)(k - i - 1) * n : a.rv);
                }, a.rv, i + 2, n, a.tpart, nw - 1 - gwarp, nw, lane);
        }
        if (!grid_wait(a.bar, target += G)) return;
    }
}

// -------------------------------------------------------------- QR panel
constexpr int kQld = kQp + 1;      // row stride in shared memory

struct Geqr2ResArgs {
    double *A;
    int lda, m, nb;
    double *tau, *gram;            // gram[c ldg + i]: v_c^T v_i, c < i (what T is formed from)
    int ldg;
    Slot *gp;                      // [grid][32]: per-CTA partial sums a^T A[:, c] (column i: a^T a)
    Slot *row, *sv;                // [2][32] top row, by the step's parity; [32] sums over the CTAs
    GridBar *bar;
    unsigned base;
};

// Householder QR of an m x nb panel (Sec. 4.3, step 1) held on chip: a block
// of rows per CTA in shared memory (row major), a column per lane, the rows
// over four warps.  With a = column i (unscaled; v = sc a, v_i = 1):
//   owners  column c != i is owned by one warp of the grid: g_c = sum over CTAs
//           of a^T A[:, c] (tail rows), sent to every CTA; a warp of every CTA
//           sums sig2 = a^T a and forms H_i's scalars while these travel.  The
//           finished columns (c < i) give v_c^T v_i: their lanes would idle,
//           and T needs those products (a separate pass over a 10000 x 32
//           panel for them measured 335 us, this kernel 200).
//   rows    s_c = tau (A[i, c] + sc g_c), R[i, c] = A[i, c] - s_c is final;
//           one pass A[r, c] -= a_r (sc s_c) with the partial sums of the next
//           column a' = A[:, i + 1] (a lane broadcast) against all columns
// Two slot exchanges per column (buffers reused as in k_gebd2_resident)
// instead of three grid barriers with the panel read from L2.  What bounds
// it: the exchanges; two FP64 operations per row and column are about 2000
// cycles of a column at 66 rows a CTA.  geqrf of 10000 x 32, 10000 x 600 and
// 2048 x 2048: 355, 8449 and 29191 us with the scalars formed by the owners
// before they sent their results, 301, 7442 and 27524 us now.
__global__ void __launch_bounds__(NT) k_geqr2_resident(Geqr2ResArgs a) {
    extern __shared__ double smem[];
    __shared__ int s_err;
    __shared__ double s_red[4][kQp], s_fac[kQp], s_sc[kQp], s_alpha, s_sig2, s_tau;
    const int G = gridDim.x, g = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int m = a.m, nb = a.nb;
    const int rb = (m + G - 1) / G, r0 = min(m, g * rb), nr = min(m, r0 + rb) - r0;
    double *W = smem;              // [nr][kQld]
    double *A = a.A;
    const size_t lda = a.lda;
    if (t == 0) s_err = 0;
    for (int c = warp; c < kQp; c += 4)
        for (int r = lane; r < nr; r += 32) W[r * kQld + c] = c < nb ? A[(size_t)c * lda + r0 + r] : 0.0;
    const Slot zero = {0ull, 0ull};
    if (t < kQp) a.gp[g * kQp + t] = zero;
    if (g == 0 && t < kQp) a.row[t] = a.row[kQp + t] = a.sv[t] = zero;
    unsigned target = a.base + G;
    if (!grid_wait(a.bar, target)) return;

    auto publish = [&](double acc, unsigned tag) {
        s_red[warp][lane] = acc;
        __syncthreads();
        if (warp == 0 && lane < nb)
            slot_put(a.gp + g * kQp + lane, (s_red[0][lane] + s_red[1][lane]) + (s_red[2][lane] + s_red[3][lane]), tag);
    };
    {
        double acc = 0.0;
        for (int r = warp; r < nr; r += 4) {
            const double x = W[r * kQld + lane], y = W[r * kQld];
            if (r0 + r == 0) {
                if (lane < nb) slot_put(a.row + lane, x, 1u);
            } else {
                acc = fma(y, x, acc);
            }
        }
        publish(acc, 1u);
    }
    for (int i = 0; i < nb; ++i) {
        const unsigned tag = (unsigned)i + 1u;
        if (!grid_wait<false>(a.bar, target += G)) return;
        const Slot *row = a.row + (i & 1) * kQp;
        // ---- warps 1-3: the k-th column other than i; warp 0: column i itself
        {
            const int k = g + G * (warp - 1), c = warp == 0 ? i : k < i ? k : k + 1;
            if (c < nb) {
                double s = 0.0;
                for (int q0 = lane; q0 < G; q0 += 160) {
                    const Slot *q[6];
                    double v[6];
#pragma unroll
                    for (int j = 0; j < 5; ++j) q[j] = q0 + 32 * j < G ? a.gp + (q0 + 32 * j) * kQp + c : nullptr;
                    q[5] = warp == 0 ? row + i : nullptr;
                    slot_get<6>(q, tag, v, a.bar, &s_err);
                    if (t == 0) s_alpha = v[5];
                    s += v[0];
#pragma unroll
                    for (int j = 1; j < 5; ++j)
                        if (q0 + 32 * j < G) s += v[j];
                }
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) {
                    if (warp == 0) s_sig2 = s;
                    else slot_put(a.sv + c, s, tag);
                }
            }
        }
        // the scalars of H_i while the other columns' sums are on their way
        if (!grid_wait<false, 32>(a.bar, target += G, [&] {
                double tau, beta;
                const double sc = reflector_fast(s_alpha, s_sig2, tau, beta);
                if (t == 0) {
                    s_sc[i] = sc;
                    s_tau = tau;
                    if (g == 0) {
                        a.tau[i] = tau;
                        A[(size_t)i * lda + i] = beta;
                    }
                }
            }))
            return;
        // ---- rows
        if (warp == 0) {
            const bool on = lane != i && lane < nb;
            const Slot *q[2] = {on ? a.sv + lane : nullptr, on ? row + lane : nullptr};
            double v[2];
            slot_get<2>(q, tag, v, a.bar, &s_err);
            const double sc = s_sc[i], w = fma(sc, v[0], v[1]), sfac = s_tau * w;
            s_fac[lane] = lane > i && lane < nb ? -(sc * sfac) : 0.0;
            if (g == 0 && on) {
                if (lane < i) a.gram[(size_t)lane * a.ldg + i] = s_sc[lane] * w;
                else A[(size_t)lane * lda + i] = v[1] - sfac;
            }
        }
        __syncthreads();
        if (s_err) return;         // uniform: read after the barrier
        if (i + 1 == nb) break;
        const double f = s_fac[lane];
        const int rl = max(0, i + 1 - r0);              // own rows below i
        double acc = 0.0;
        int r = rl + warp;
        if (r0 + rl == i + 1 && rl < nr && warp == 0) { // the next top row
            const double x = fma(W[r * kQld + i], f, W[r * kQld + lane]);
            if (lane < nb) slot_put(a.row + ((i + 1) & 1) * kQp + lane, x, tag + 1u);
            r += 4;
        }
        for (; r + 12 < nr; r += 16) {
            double x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] = W[(r + 4 * j) * kQld + lane];
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] = fma(W[(r + 4 * j) * kQld + i], f, x[j]);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc = fma(__shfl_sync(0xffffffffu, x[j], i + 1), x[j], acc);
#pragma unroll
            for (int j = 0; j < 4; ++j) W[(r + 4 * j) * kQld + lane] = x[j];   // (lanes <= i: unchanged, f = 0)
        }
        for (; r < nr; r += 4) {
            const double x = fma(W[r * kQld + i], f, W[r * kQld + lane]);
            acc = fma(__shfl_sync(0xffffffffu, x, i + 1), x, acc);
            W[r * kQld + lane] = x;
        }
        publish(acc, tag + 1u);
    }
    // the reflectors' entries, scaled
    for (int c = warp; c < nb; c += 4)
        for (int r = lane; r < nr; r += 32)
            if (r0 + r > c) A[(size_t)c * lda + r0 + r] = s_sc[c] * W[r * kQld + c];
}

}  // namespace

size_t resident_scratch_doubles(int n) {
    // a matrix with m >= n that fits has n^2 doubles in kResGrid SMs of 227 KB
    const size_t nn = std::max(std::min(n, 2200), kQp);   // (at least a QR panel's slots)
    return 2 * ((size_t)kResGrid * nn + 3 * nn + 8);
}

size_t labrd_scratch_doubles(int m, int n) {
    return (size_t)m + n + 64 + (size_t)kParts * ((size_t)n + 2 * kLb + 8) + (size_t)kParts * 32 * ((m + 31) / 32 + 1) +
           (size_t)kParts * (2 * kLb + 8);
}

cudaError_t launch_labrd_panel(int m, int n, int nb, double *A, int lda, double *d, double *e, double *tauq,
                               double *taup, double *PW, double *QW, double *scratch, GridBar *bar, unsigned *bars,
                               cudaStream_t st) {
    if (nb > kLb) return cudaErrorInvalidValue;
    const int G = std::max(1, dev_info().sms);
    double *av = scratch, *rv = av + m, *cp = rv + n + 32, *hp = cp + (size_t)kParts * (n + 2 * kLb + 8);
    double *tp = hp + (size_t)kParts * 32 * ((m + 31) / 32 + 1);
    Labrd2Args a{A, lda, m, n, nb, d, e, tauq, taup, PW, PW + (size_t)kLb * m, QW, QW + (size_t)kLb * n, av, rv, cp, hp,
                 tp, bar, *bars};
    // four waits a step; the matrix's last column (no row reflector) ends after two
    *bars += (unsigned)G * (nb == n ? 4u * (unsigned)(nb - 1) + 2u : 4u * (unsigned)nb);
    void *params[] = {&a};
    return cudaLaunchCooperativeKernel((const void *)k_labrd_panel, dim3(G), dim3(kLT), params, 0, st);
}

// rows of a QR panel's CTA: about 64, at least 11 CTAs (the owners of 31
// columns are a warp each, three a CTA), as many as there are SMs
static int qr_grid(int m) {
    const DevInfo d = dev_info();
    return std::max(11, std::min({(m + 63) / 64, d.sms, kResGrid}));
}
static size_t qr_smem(int m, int G) { return sizeof(double) * (size_t)((m + G - 1) / G) * kQld + 64; }

bool geqr2_resident_fits(int m, int nb) {
    const DevInfo d = dev_info();
    return d.sms >= 11 && nb >= 1 && nb <= kQp && m >= nb && qr_smem(m, qr_grid(m)) <= (size_t)d.smem - 4096;
}

cudaError_t launch_geqr2_resident(int m, int nb, double *A, int lda, double *tau, double *gram, int ldg,
                                  double *scratch, GridBar *bar, unsigned *bars, cudaStream_t st) {
    const int G = qr_grid(m);
    Slot *gp = (Slot *)scratch, *row = gp + (size_t)kResGrid * kQp, *sv = row + 2 * kQp;
    Geqr2ResArgs a{A, lda, m, nb, tau, gram, ldg, gp, row, sv, bar, *bars};
    *bars += (unsigned)G * (1u + 2u * (unsigned)nb);
    cudaError_t err =
        cudaFuncSetAttribute(k_geqr2_resident, cudaFuncAttributeMaxDynamicSharedMemorySize, dev_info().smem - 4096);
    if (err != cudaSuccess) return err;
    void *params[] = {&a};
    return cudaLaunchCooperativeKernel((const void *)k_geqr2_resident, dim3(G), dim3(NT), params, qr_smem(m, G), st);
}

int res_grid(int m) {
    const DevInfo d = dev_info();
    return std::max(1, std::min(std::min(d.sms, kResGrid), m));
}

bool resident_fits(int m, int n) {
    const DevInfo d = dev_info();
    if (d.sms <= 0 || n < 1 || n > 2200) return false;
    const int G = res_grid(m);
    return res_smem(m, n, G) <= (size_t)d.smem;
}

cudaError_t launch_gebd2_resident(int m, int n, double *A, int lda, double *d, double *e, double *tauq, double *taup,
                                  double *scratch, GridBar *bar, unsigned *bars, cudaStream_t st) {
    const int G = res_grid(m);
    const size_t smem = res_smem(m, n, G);
    Slot *gp = (Slot *)scratch, *row = gp + (size_t)kResGrid * n, *gs = row + 2 * n;
    Gebd2Args a{A, lda, m, n, d, e, tauq, taup, gp, row, gs, bar, *bars};
    *bars += (unsigned)G * (1u + 2u * (unsigned)n);   // load, first sums, n Y phases, n - 1 X phases
    // the device's maximum, not this launch's size: another thread may be
    // between its own call and its launch
    cudaError_t err =
        cudaFuncSetAttribute(k_gebd2_resident, cudaFuncAttributeMaxDynamicSharedMemorySize, dev_info().smem);
    if (err != cudaSuccess) return err;
    void *params[] = {&a};
    return cudaLaunchCooperativeKernel((const void *)k_gebd2_resident, dim3(G), dim3(NT), params, smem, st);
}

}  // namespace bdc
