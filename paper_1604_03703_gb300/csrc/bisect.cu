// bisect.cu -- eigenvalues of the final symmetric tridiagonal by Sturm-count
// bisection (the last step of Algorithm 4.3, which returns the tridiagonal's
// eigenvalues as the result), plus the
// small copy kernels between dense, packed-band and tridiagonal storage.
//
// The bisection runs on T scaled by an exact power of two 2^-s that brings
// its Gershgorin bound into [0.5, 1).  The Sturm count at x is the number of
// sign changes of the leading principal minors of T - xI (Sturm's theorem),
//   p_1 = d_0 - x,  p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1},
// the division-free form of the LDL^T pivot count: per step one FMA on the
// dependence chain (instead of a ~1000-cycle FP64 division), the pair
// (p_{i-1}, p_i) rescaled by a power of two when |p_i| leaves
// [2^-256, 2^256], a zero minor counted as a sign change, the recurrence begun
// anew after two of them in a row (T splits behind a singular block).  Every FP64
// operation is written with an explicit round-to-nearest intrinsic so no
// multiply-add is contracted: the result is the exact IEEE evaluation of the
// recurrence in the order written.
#include <atomic>

#include "sturm.cuh"

namespace sev {

// ------------------------------------------------------------ storage copies
template <typename T>
__global__ void band_from_dense_kernel(int n, const T *__restrict__ A, int lda, int b, T *__restrict__ AB, int ldab) {
    const long total = (long)ldab * n;
    for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int d = (int)(idx % ldab);
        const int j = (int)(idx / ldab);
        T v = 0;
        if (d <= b && j + d < n) v = A[(size_t)(j + d) + (size_t)j * lda];
        AB[idx] = v;
    }
}

template <typename T>
int launch_band_from_dense(sev_ctx *h, int n, const T *A, int lda, int b, T *AB, int ldab) {
    if (n <= 0) return SEV_OK;
    const long total = (long)ldab * n;
    int grid = (int)((total + kThreads - 1) / kThreads);
    if (grid > h->sm_count * 16) grid = h->sm_count * 16;
    SEV_LAUNCH(h, K_BAND_FROM_DENSE, band_from_dense_kernel<T>, grid, kThreads, 0, n, A, lda, b, AB, ldab);
    return SEV_OK;
}

template <typename T>
__global__ void tridiag_extract_kernel(int n, const T *__restrict__ AB, int ldab, double *__restrict__ d,
                                       double *__restrict__ e) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        d[j] = (double)AB[(size_t)j * ldab];
        if (j + 1 < n) e[j] = (double)AB[1 + (size_t)j * ldab];
    }
}

template <typename T>
int launch_tridiag_extract(sev_ctx *h, int n, const T *AB, int ldab, double *d, double *e) {
    if (n <= 0) return SEV_OK;
    int grid = (n + kThreads - 1) / kThreads;
    if (grid > h->sm_count * 4) grid = h->sm_count * 4;
    SEV_LAUNCH(h, K_TRIDIAG_EXTRACT, tridiag_extract_kernel<T>, grid, kThreads, 0, n, AB, ldab, d, e);
    return SEV_OK;
}

// Non-finite scan of the lower triangle (diagonal included): CTA c takes
// columns c, c + grid, ...; its threads read down a column (coalesced).  With
// dst the triangle is copied to it on the way (leading dimension ldd).
template <typename T>
__global__ void check_finite_kernel(int n, const T *__restrict__ A, int lda, int *__restrict__ flag, int *err,
                                    T *__restrict__ dst, int ldd) {
    bool bad = false;
    for (int j = blockIdx.x; j < n; j += gridDim.x)
        for (int i = j + threadIdx.x; i < n; i += blockDim.x) {
            const T v = A[(size_t)i + (size_t)j * lda];
            bad |= !isfinite(v);
            if (dst) dst[(size_t)i + (size_t)j * ldd] = v;
        }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) {
        latch_error(err, SEV_ERR_NONFINITE);
        if (flag) atomicExch(flag, 1);
    }
}

template <typename T>
int launch_check_finite(sev_ctx *h, int n, const T *A, int lda, int *flag, T *dst, int ldd) {
    if (n <= 0) return SEV_OK;
    int grid = n < h->sm_count * 8 ? n : h->sm_count * 8;
    SEV_LAUNCH(h, K_CHECK_FINITE, check_finite_kernel<T>, grid, kThreads, 0, n, A, lda, flag, h->d_err, dst, ldd);
    return SEV_OK;
}

// The lower triangle of A from the packed band (half-bandwidth b): the band's
// entries and exact zeros below them.
template <typename T>
__global__ void dense_from_band_kernel(int n, T *__restrict__ A, int lda, int b, const T *__restrict__ AB, int ldab) {
    for (int j = blockIdx.x; j < n; j += gridDim.x)
        for (int i = j + threadIdx.x; i < n; i += blockDim.x)
            A[(size_t)i + (size_t)j * lda] = i - j <= b ? AB[(i - j) + (size_t)j * ldab] : T(0);
}

template <typename T>
int launch_dense_from_band(sev_ctx *h, int n, T *A, int lda, int b, const T *AB, int ldab) {
    if (n <= 0) return SEV_OK;
    int grid = n < h->sm_count * 8 ? n : h->sm_count * 8;
    SEV_LAUNCH(h, K_BAND_FROM_DENSE, dense_from_band_kernel<T>, grid, kThreads, 0, n, A, lda, b, AB, ldab);
    return SEV_OK;
}

template int launch_dense_from_band<float>(sev_ctx *, int, float *, int, int, const float *, int);
template int launch_dense_from_band<double>(sev_ctx *, int, double *, int, int, const double *, int);
template int launch_check_finite<float>(sev_ctx *, int, const float *, int, int *, float *, int);
template int launch_check_finite<double>(sev_ctx *, int, const double *, int, int *, double *, int);
template int launch_band_from_dense<float>(sev_ctx *, int, const float *, int, int, float *, int);
template int launch_band_from_dense<double>(sev_ctx *, int, const double *, int, int, double *, int);
template int launch_tridiag_extract<float>(sev_ctx *, int, const float *, int, double *, double *);
template int launch_tridiag_extract<double>(sev_ctx *, int, const double *, int, double *, double *);

// ----------------------------------------------------------------- bisection
// par[0] = gl, par[1] = gu (scaled, widened Gershgorin interval), par[2] = sc
// = 2^-s, par[3] = tnorm (scaled max |end| of the unwidened interval),
// par[4] = 2^s, par[5] = 1 if T = 0 (a zero Gershgorin bound), par[6] = 1 if
// the caller's skip flag was set (non-finite input) or, with such a flag, a
// wait has run out in the reductions (no bisection, NaN eigenvalues), par[7] =
// 1 if some e2s is nonzero but below 2^-322.  e2s[i] = (e_i 2^-s)^2.
__global__ void bisect_prep_kernel(int n, const double *__restrict__ d, const double *__restrict__ e,
                                   double *__restrict__ e2s, double *__restrict__ par, const int *skip,
                                   const int *status) {
    __shared__ double red[32];
    __shared__ double s_sc;
    __shared__ int s_tiny;
    if (threadIdx.x == 0) s_tiny = 0;
    double lo = INFINITY, hi = -INFINITY;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double r = 0.0;
        if (i > 0) r = __dadd_rn(r, fabs(e[i - 1]));
        if (i + 1 < n) r = __dadd_rn(r, fabs(e[i]));
        lo = fmin(lo, __dsub_rn(d[i], r));
        hi = fmax(hi, __dadd_rn(d[i], r));
    }
    lo = -block_max(-lo, red);
    hi = block_max(hi, red);
    if (threadIdx.x == 0) {
        double tnorm = fmax(fabs(lo), fabs(hi));
        int s = 0;
        if (tnorm > 0.0) (void)frexp(tnorm, &s);  // tnorm = m 2^s, m in [0.5, 1)
        const double sc = pow2_exact(-s);
        lo = __dmul_rn(lo, sc);
        hi = __dmul_rn(hi, sc);
        tnorm = __dmul_rn(tnorm, sc);
        const double pad = __dadd_rn(__dmul_rn(__dmul_rn(__dmul_rn(2.0, (double)n), DBL_EPSILON), tnorm), 0x1p-1000);
        par[0] = __dsub_rn(lo, pad);
        par[1] = __dadd_rn(hi, pad);
        par[2] = sc;
        par[3] = tnorm;
        par[4] = pow2_exact(s);
        par[5] = tnorm == 0.0 ? 1.0 : 0.0;
        par[6] = (skip && (*skip || any_gave_up(status))) ? 1.0 : 0.0;
        s_sc = sc;
    }
    __syncthreads();
    const double sc = s_sc;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        if (i + 1 < n) {
            const double es = __dmul_rn(e[i], sc), e2 = __dmul_rn(es, es);
            e2s[i] = e2;
            if (es != 0.0 && e2 < 0x1p-322) s_tiny = 1;
        } else {
            e2s[i] = 0.0;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) par[7] = s_tiny ? 1.0 : 0.0;
}

__device__ __forceinline__ int sturm_count(int n, const double *__restrict__ d, const double *__restrict__ e2s,
                                           double x, double sc, bool plain) {
    return sturm_count_blocks<8>(
        n, [&](int i) { return __ldg(d + i); }, [&](int i) { return __ldg(e2s + i); }, x, sc, plain);
}

// One thread per eigenvalue index k (the (k+1)-th smallest).
__global__ void bisect_kernel(int n, const double *__restrict__ d, const double *__restrict__ e2s,
                              const double *__restrict__ par, double rtol, int maxit, double *__restrict__ eigs,
                              int *err) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    if (n == 1) {
        eigs[0] = d[0];
        return;
    }
    if (par[5] != 0.0) {
        eigs[k] = 0.0;
        return;
    }
    const double sc = par[2];
    const bool plain = par[7] == 0.0;
    const double atol = __dmul_rn(rtol, par[3]);
    double lo = par[0], hi = par[1];
    int it = 0;
    for (;;) {
        const double w = __dsub_rn(hi, lo);
        const double mag = fmax(fabs(lo), fabs(hi));
        double tol = __dmul_rn(rtol, mag);
        if (atol > tol) tol = atol;
        if (w <= tol) break;
        if (it >= maxit) {
            latch_error(err, SEV_ERR_NOCONV);
            break;
        }
        const double mid = __dmul_rn(0.5, __dadd_rn(lo, hi));
        if (mid <= lo || mid >= hi) break;
        if (sturm_count(n, d, e2s, mid, sc, plain) >= k + 1)
            hi = mid;
        else
            lo = mid;
        ++it;
    }
    eigs[k] = __dmul_rn(__dmul_rn(0.5, __dadd_rn(lo, hi)), par[4]);
}

// ------------------------------------------------- shared-interval rounds
// The per-eigenvalue bisection above visits, for index k, the path of
// intervals that the counts at its midpoints dictate.  Indices whose
// intervals coincide take identical steps (same midpoint, same count, same
// stopping test), and by monotonicity of the count they form contiguous
// runs of k.  bisect_rounds_kernel exploits both facts without changing a
// single rounding: every round (1) lists the distinct active intervals
// (leaders), (2) evaluates, for each leader, the counts at all midpoints of
// its subtree of depth d -- the midpoints its next d bisection steps can
// reach, computed by the same IEEE operations -- with d as deep as the
// thread budget allows, and (3) lets every index walk d steps down its
// leader's subtree using those counts.  The result is bitwise the one of
// bisect_kernel; the chain of dependent Sturm counts per index shrinks from
// one per level to one per round (the early levels, where few intervals are
// distinct, are resolved many at a time).
//
// The kernel is persistent and cooperative (all CTAs resident); the three
// phases of a round are separated by a grid barrier with a capped wait.
struct BisCtl {
    int bar;    // monotone arrival counter of the grid barrier
    int D;      // leaders this round
    int depth;  // subtree depth this round
    int done;   // no active index left
    int abort;  // a wait hit its cap
    int rounds;       // rounds run (diagnostics)
    long long items;  // subtree midpoints evaluated (diagnostics)
};

// Grid barrier number `seq` (1, 2, ...): returns false if the wait hit its cap
// or another CTA gave up.
__device__ bool bis_barrier(BisCtl *ctl, int seq, long long cap, int *err) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&ctl->bar, 1);
        const int target = seq * (int)gridDim.x;
        const int ok = wait_flag(&ctl->bar, target, cap, err, [&] { return *(volatile int *)&ctl->abort != 0; }) >= 0;
        if (!ok) *(volatile int *)&ctl->abort = 1;
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// The stopping test of one bisection step on [lo, hi] (same operations and
// order as bisect_kernel).  Returns 0 to continue with mid, 1 when converged
// or mid no longer splits, 2 when the step cap is reached.
__device__ __forceinline__ int bis_step_test(double lo, double hi, int it, double rtol, double atol, int maxit,
                                             double &mid) {
    const double w = __dsub_rn(hi, lo);
    const double mag = fmax(fabs(lo), fabs(hi));
    double tol = __dmul_rn(rtol, mag);
    if (atol > tol) tol = atol;
    if (w <= tol) return 1;
    if (it >= maxit) return 2;
    mid = __dmul_rn(0.5, __dadd_rn(lo, hi));
    if (mid <= lo || mid >= hi) return 1;
    return 0;
}

struct BisWs {
    double *lo, *hi;
    int *it, *st;        // steps taken; state: 0 active, 1 finished
    int *lead, *leadof;  // leader list; leader slot of each index
    int *cnt;            // counts of the round's subtree midpoints
    BisCtl *ctl;
};

#ifndef SEV_BIS_CHAINS_PER_SM
#define SEV_BIS_CHAINS_PER_SM 128
#endif
constexpr int kBisThreads = 512;  // 128 registers a thread for the Sturm blocks
constexpr int kBisMaxItems = 131072;

// Depth of a round's subtrees for D distinct intervals: fewest rounds per
// level, counting a round as one chain latency while its items fit the budget
// of chains the GPU keeps in flight, and proportionally longer beyond it.
__device__ __forceinline__ int bis_depth(int D, int budget, int most) {
    int dep = 1;
    float best = 2.f;
    for (int t = 1; t <= 24; ++t) {
        const long items = (long)D * ((1L << t) - 1);
        if (items > most) break;
        const float cost = fmaxf(1.f, (float)items / (float)budget) / (float)t;
        if (cost < best) {
            best = cost;
            dep = t;
        }
    }
    return dep;
}

// Count at midpoint m (heap order) of the subtree under [lo, hi]; -1 when the
// bisection ends before it.
__device__ __forceinline__ int bis_item(int n, const double *__restrict__ d, const double *__restrict__ e2, double lo,
                                        double hi, int it, int m, double rtol, double atol, int maxit, double sc,
                                        bool plain) {
    // node m: its depth is floor(log2(m + 1)); the bits of m + 1 below the
    // leading one, top first, are the turns (1 = right)
    const int path = m + 1;
    double mid = 0.0;
    for (int l = 30 - __clz(path); l >= 0; --l) {
        if (bis_step_test(lo, hi, it, rtol, atol, maxit, mid) != 0) return -1;
        if ((path >> l) & 1)
            lo = mid;
        else
            hi = mid;
        ++it;
    }
    if (bis_step_test(lo, hi, it, rtol, atol, maxit, mid) != 0) return -1;
    return sturm_count(n, d, e2, mid, sc, plain);
}

// Index k walks at most dep steps down its subtree: cnt(node) >= k + 1 turns
// left.  Returns the stopping test's state after the last step.
template <typename F>
__device__ __forceinline__ int bis_walk(int k, int dep, double &lo, double &hi, int &it, double rtol, double atol,
                                        int maxit, F cnt) {
    double mid = 0.0;
    int node = 0;
    for (int l = 0; l < dep; ++l) {
        const int r = bis_step_test(lo, hi, it, rtol, atol, maxit, mid);
        if (r != 0) return r;
        if (cnt(node) >= k + 1) {
            hi = mid;
            node = 2 * node + 1;
        } else {
            lo = mid;
            node = 2 * node + 2;
        }
        ++it;
    }
    return bis_step_test(lo, hi, it, rtol, atol, maxit, mid);
}

// Small orders: the same rounds with every CTA keeping ALL indices' intervals
// in shared memory and running the leader list and the walk for itself, so
// that only the counts travel and a round has one grid barrier instead of
// three (at these orders a round's chain is shorter than its barriers:
// n = 100 217 -> 111 us with the faster Sturm
// loop, n = 2048 3.07 -> 2.10 ms).  The counts of alternate rounds go to
// alternate halves of W.cnt: a CTA writes round r + 2 only after barrier
// r + 1, which every CTA reaches after it has read round r.
constexpr int kBisSmallN = 2048;
constexpr int kBisStage = 16384;  // counts of a round held in shared memory (16 bits each)
constexpr int kBisSmallItems = kBisMaxItems / 2;
__host__ __device__ constexpr size_t bis_small_smem(int n) { return (size_t)n * 24 + 64 + kBisStage * 2; }

__global__ void __launch_bounds__(kBisThreads)
    bisect_small_kernel(int n, const double *__restrict__ d, const double *__restrict__ e2,
                        const double *__restrict__ par, double rtol, int maxit, int budget, double *__restrict__ eigs,
                        int *cnt, BisCtl *ctl, int *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    double *lo = (double *)smem, *hi = lo + n;
    short *lead = (short *)(hi + n), *leadof = lead + n, *it = leadof + n, *st = it + n;
    short *stage = st + n;
    __shared__ int s_warp[32];
    const long long cap = wait_cap(err);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (par[6] != 0.0) {  // no tridiagonal to bisect (every CTA reads the same flag: no barrier is entered)
        if (blockIdx.x == 0)
            for (int k = tid; k < n; k += kBisThreads) eigs[k] = __longlong_as_double(0x7ff8000000000000LL);
        return;
    }
    const double sc = par[2], atol = __dmul_rn(rtol, par[3]);
    const bool plain = par[7] == 0.0;
    const int zero = par[5] != 0.0;  // T = 0: every eigenvalue is exactly 0
    for (int k = tid; k < n; k += kBisThreads) {
        lo[k] = zero ? 0.0 : par[0];
        hi[k] = zero ? 0.0 : par[1];
        it[k] = 0;
        st[k] = (short)zero;
    }
    __syncthreads();
    constexpr int kPer = kBisSmallN / kBisThreads;  // indices per thread, consecutive
    for (int round = 0;; ++round) {
        // ---- leaders: the first index of every distinct active interval
        bool is[kPer];
        int mine = 0;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int k = tid * kPer + u;
            is[u] = k < n && st[k] == 0 && (k == 0 || st[k - 1] != 0 || lo[k] != lo[k - 1] || hi[k] != hi[k - 1]);
            mine += is[u];
        }
        int pos = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, pos, o);
            if (lane >= o) pos += v;
        }
        if (lane == 31) s_warp[warp] = pos;
        __syncthreads();
        int before = 0, D = 0;
#pragma unroll
        for (int w = 0; w < kBisThreads / 32; ++w) {
            const int v = s_warp[w];
            before += w < warp ? v : 0;
            D += v;
        }
        if (D == 0) break;
        pos += before - mine;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int k = tid * kPer + u;
            if (is[u]) lead[pos++] = (short)k;
            if (k < n) leadof[k] = (short)(pos - 1);
        }
        __syncthreads();
        // ---- counts of this CTA's share of the round's midpoints
        const int dep = bis_depth(D, budget, kBisSmallItems);
        const int M = (1 << dep) - 1, items = D * M;
        int *cr = cnt + (round & 1) * kBisSmallItems;
        for (int w = blockIdx.x + tid * gridDim.x; w < items; w += gridDim.x * kBisThreads) {
            const int k = lead[w / M];
            __stcg(cr + w, bis_item(n, d, e2, lo[k], hi[k], it[k], w % M, rtol, atol, maxit, sc, plain));
        }
        if (!bis_barrier(ctl, round + 1, cap, err)) return;
        const bool staged = items <= kBisStage;
        if (staged) {
            for (int w = tid; w < items; w += kBisThreads) stage[w] = (short)__ldcg(cr + w);
            __syncthreads();
        }
        // ---- every active index walks down its leader's subtree
        for (int k = tid; k < n; k += kBisThreads) {
            if (st[k] != 0) continue;
            const int j0 = (int)leadof[k] * M;
            double l = lo[k], h = hi[k];
            int i = it[k];
            const int state = bis_walk(k, dep, l, h, i, rtol, atol, maxit, [&](int node) {
                return staged ? (int)stage[j0 + node] : __ldcg(cr + j0 + node);
            });
            if (state == 2) latch_error(err, SEV_ERR_NOCONV);
            lo[k] = l;
            hi[k] = h;
            it[k] = (short)i;
            st[k] = state != 0;
        }
        __syncthreads();
    }
    const double up = par[4];
    if (blockIdx.x == 0)
        for (int k = tid; k < n; k += kBisThreads) eigs[k] = __dmul_rn(__dmul_rn(0.5, __dadd_rn(lo[k], hi[k])), up);
}

__global__ void __launch_bounds__(kBisThreads) bisect_rounds_kernel(int n, const double *__restrict__ d,
                                                                    const double *__restrict__ e2,
                                                                    const double *__restrict__ par, double rtol,
                                                                    int maxit, int budget, double *__restrict__ eigs,
                                                                    BisWs W, int *err) {
    __shared__ int s_scan[kBisThreads];
    const long long cap = wait_cap(err);
    const double sc = par[2];
    const bool plain = par[7] == 0.0;
    const double atol = __dmul_rn(rtol, par[3]);
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    const int gthreads = gridDim.x * blockDim.x;
    if (par[6] != 0.0) {  // no tridiagonal to bisect (every CTA reads the same flag: no barrier is entered)
        for (int k = gtid; k < n; k += gthreads) eigs[k] = __longlong_as_double(0x7ff8000000000000LL);
        return;
    }
    const int zero = par[5] != 0.0;  // T = 0: every eigenvalue is exactly 0 (lo = hi = 0, finished)
    for (int k = gtid; k < n; k += gthreads) {
        W.lo[k] = zero ? 0.0 : par[0];
        W.hi[k] = zero ? 0.0 : par[1];
        W.it[k] = 0;
        W.st[k] = zero;
    }
    int seq = 0;
    if (!bis_barrier(W.ctl, ++seq, cap, err)) return;
    for (;;) {
        // ---- (1) leaders: CTA 0 compacts the distinct active intervals
        if (blockIdx.x == 0) {
            const int chunk = (n + kBisThreads - 1) / kBisThreads;
            const int k0 = threadIdx.x * chunk, k1 = min(n, k0 + chunk);
            int mine = 0;
            for (int k = k0; k < k1; ++k)
                if (W.st[k] == 0 && (k == 0 || W.st[k - 1] != 0 || W.lo[k] != W.lo[k - 1] || W.hi[k] != W.hi[k - 1]))
                    ++mine;
            s_scan[threadIdx.x] = mine;
            __syncthreads();
            for (int off = 1; off < kBisThreads; off <<= 1) {  // inclusive scan
                const int v = threadIdx.x >= off ? s_scan[threadIdx.x - off] : 0;
                __syncthreads();
                s_scan[threadIdx.x] += v;
                __syncthreads();
            }
            int pos = s_scan[threadIdx.x] - mine;  // leaders before this chunk
            for (int k = k0; k < k1; ++k) {
                if (W.st[k] != 0) continue;
                if (k == 0 || W.st[k - 1] != 0 || W.lo[k] != W.lo[k - 1] || W.hi[k] != W.hi[k - 1]) W.lead[pos++] = k;
                W.leadof[k] = pos - 1;
            }
            if (threadIdx.x == kBisThreads - 1) {
                // depth: fewest rounds per level, counting a round as one
                // chain latency while its items fit the budget of chains the
                // GPU keeps in flight, and proportionally longer beyond it
                const int D = s_scan[kBisThreads - 1];
                const int dep = bis_depth(D, budget, n > kBisMaxItems ? n : kBisMaxItems);
                W.ctl->D = D;
                W.ctl->depth = dep;
                W.ctl->done = D == 0;
                if (D > 0) {
                    W.ctl->rounds += 1;
                    W.ctl->items += (long long)D * ((1L << dep) - 1);
                }
            }
        }
        if (!bis_barrier(W.ctl, ++seq, cap, err)) return;
        if (*(volatile int *)&W.ctl->done) break;
        const int D = *(volatile int *)&W.ctl->D;
        const int dep = *(volatile int *)&W.ctl->depth;
        const int M = (1 << dep) - 1;
        // ---- (2) counts at every midpoint of every leader's subtree
        const long items = (long)D * M;
        // items are dealt round-robin over the CTAs so every SM gets its share
        for (long w = blockIdx.x + (long)threadIdx.x * gridDim.x; w < items; w += gthreads) {
            const int j = (int)(w / M), m = (int)(w % M);
            const int k = W.lead[j];
            W.cnt[w] = bis_item(n, d, e2, W.lo[k], W.hi[k], W.it[k], m, rtol, atol, maxit, sc, plain);
        }
        if (!bis_barrier(W.ctl, ++seq, cap, err)) return;
        // ---- (3) every active index walks dep steps down its leader's subtree
        for (int k = gtid; k < n; k += gthreads) {
            if (W.st[k] != 0) continue;
            const int *cj = W.cnt + (long)W.leadof[k] * M;
            double lo = W.lo[k], hi = W.hi[k];
            int it = W.it[k];
            const int state = bis_walk(k, dep, lo, hi, it, rtol, atol, maxit, [&](int node) { return cj[node]; });
            if (state == 2) latch_error(err, SEV_ERR_NOCONV);
            W.lo[k] = lo;
            W.hi[k] = hi;
            W.it[k] = it;
            W.st[k] = state != 0;
        }
        if (!bis_barrier(W.ctl, ++seq, cap, err)) return;
    }
    const double up = par[4];
    for (int k = gtid; k < n; k += gthreads) eigs[k] = __dmul_rn(__dmul_rn(0.5, __dadd_rn(W.lo[k], W.hi[k])), up);
}

size_t bisect_workspace(int n) {
    Carver c(nullptr);
    c.take<double>((size_t)n + 1);
    c.take<double>(8);
    c.take<double>((size_t)n);
    c.take<double>((size_t)n);
    for (int a = 0; a < 4; ++a) c.take<int>((size_t)n);
    c.take<int>((size_t)(n > kBisMaxItems ? n : kBisMaxItems));
    c.take<BisCtl>(1);
    return c.bytes();
}

int launch_bisect(sev_ctx *h, int n, const double *d, const double *e, double rtol, double *eigs, void *ws,
                  size_t ws_bytes, const int *skip) {
    if (n <= 0) return SEV_OK;
    if (ws_bytes < bisect_workspace(n)) return SEV_ERR_WORKSPACE;
    Carver c(ws);
    double *e2 = c.take<double>((size_t)n + 1);
    double *par = c.take<double>(8);
    BisWs W;
    W.lo = c.take<double>((size_t)n);
    W.hi = c.take<double>((size_t)n);
    W.it = c.take<int>((size_t)n);
    W.st = c.take<int>((size_t)n);
    W.lead = c.take<int>((size_t)n);
    W.leadof = c.take<int>((size_t)n);
    W.cnt = c.take<int>((size_t)(n > kBisMaxItems ? n : kBisMaxItems));
    W.ctl = c.take<BisCtl>(1);
    SEV_LAUNCH(h, K_BISECT_PREP, bisect_prep_kernel, 1, 1024, 0, n, d, e, e2, par, skip, h->d_err);
    if (n == 1) {
        SEV_CUDA(cudaMemcpyAsync(eigs, d, sizeof(double), cudaMemcpyDeviceToDevice, h->stream));
        return SEV_OK;
    }
    SEV_CUDA(cudaMemsetAsync(W.ctl, 0, sizeof(BisCtl), h->stream));
    // One chain a scheduler and lane (128 chains per SM) keeps the FP64 pipe
    // ~75 % busy; a round with more items takes proportionally longer.
    const int grid = h->sm_count;  // one CTA per SM, all resident for the grid barrier
    int budget = grid * SEV_BIS_CHAINS_PER_SM;
    int maxit = 200;
    const bool small = n <= kBisSmallN;
    const void *kern = small ? (const void *)bisect_small_kernel : (const void *)bisect_rounds_kernel;
    const size_t smem = small ? bis_small_smem(n) : 0;
    if (small)
        SEV_CUDA(allow_smem(h, (const void *)kern));
    int per_sm = 0;
    SEV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kBisThreads, smem));
    if (per_sm < 1) return SEV_ERR_UNSUPPORTED;
    void *args[] = {(void *)&n, (void *)&d, (void *)&e2, (void *)&par, (void *)&rtol, (void *)&maxit,
                    (void *)&budget, (void *)&eigs, (void *)&W, (void *)&h->d_err};
    void *args_small[] = {(void *)&n, (void *)&d, (void *)&e2, (void *)&par, (void *)&rtol, (void *)&maxit,
                          (void *)&budget, (void *)&eigs, (void *)&W.cnt, (void *)&W.ctl, (void *)&h->d_err};
    timing_begin(h, K_BISECT);
    SEV_CUDA(cudaLaunchCooperativeKernel(kern, grid, kBisThreads, small ? args_small : args, smem, h->stream));
    timing_end(h, K_BISECT);
    return SEV_OK;
}

}  // namespace sev

// ------------------------------------------------- allocation-free variant
// sev_tridiag_bisect_static runs bisect_prep_kernel (the kernel
// sev_tridiag_bisect also starts with) and then bisect_kernel, one thread per
// eigenvalue index.  The handle path runs the cooperative bisect_rounds_kernel
// instead; for every index that kernel takes the same IEEE operations in the
// same order as bisect_kernel (the shared-interval rounds only change which
// thread evaluates a count, never its value), so both give the same bits.
// The scratch -- the squared scaled off-diagonal, the scaling and Gershgorin
// parameters and the status word -- lives in this file-scope device array
// instead of handle workspace, so a call allocates nothing.  The array is
// (kStaticMaxN + 16) doubles (~512 KiB) on every device that loads the
// library, held until the process exits.
namespace sev {
constexpr int kStaticMaxN = 65536;
constexpr int kStaticPar = kStaticMaxN + 1;     // 8 doubles of bisection parameters
constexpr int kStaticStatus = kStaticMaxN + 9;  // status word (a DevStatus-sized slot)
static __device__ __align__(256) double g_bisect_scratch[kStaticMaxN + 16];

// The array's device address and the SM count, per device ordinal.  They are
// looked up again by every call made outside stream capture (so a
// cudaDeviceReset, which reloads the module at a new address, is picked up)
// and published atomically (concurrent first calls from several host
// threads store the same values).
struct StaticScratch {
    std::atomic<double *> ptr{nullptr};
    std::atomic<int> sm_count{0};
};
static StaticScratch g_static_dev[128];
}  // namespace sev

extern "C" int sev_tridiag_bisect_static(int n, const double *d, const double *e, double rtol, double *eigs,
                                         void *stream) {
    using namespace sev;
    if (n < 0 || n > kStaticMaxN) return -1;
    if (n > 0 && !d) return -2;
    if (n > 1 && !e) return -3;
    if (!(rtol >= 1e-16) || !(rtol < 1.0)) return -4;
    if (n > 0 && !eigs) return -5;
    if (n == 0) return SEV_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return SEV_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) return SEV_ERR_CUDA;
    StaticScratch &S = g_static_dev[dev];
    double *ptr = S.ptr.load(std::memory_order_acquire);
    if (cap == cudaStreamCaptureStatusNone || !ptr) {
        // with the device current: the array's device address (in host code
        // the array's name is only a stand-in for it)
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_bisect_scratch) != cudaSuccess) return SEV_ERR_CUDA;
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return SEV_ERR_CUDA;
        S.sm_count.store(sms, std::memory_order_relaxed);
        ptr = (double *)p;
        S.ptr.store(ptr, std::memory_order_release);
    }
    const int sm_count = S.sm_count.load(std::memory_order_relaxed);
    double *e2 = ptr;                  // n + 1 doubles
    double *par = ptr + kStaticPar;    // 8 doubles
    int *status = (int *)(ptr + kStaticStatus);
    if (cudaMemsetAsync(status, 0, sizeof(int), st) != cudaSuccess) return SEV_ERR_CUDA;
    bisect_prep_kernel<<<1, 1024, 0, st>>>(n, d, n > 1 ? e : d, e2, par, nullptr, status);
    if (cudaGetLastError() != cudaSuccess) return SEV_ERR_CUDA;
    int bs = 64;
    while (bs > 32 && (n + bs - 1) / bs < sm_count) bs >>= 1;
    bisect_kernel<<<(n + bs - 1) / bs, bs, 0, st>>>(n, d, e2, par, rtol, 200, eigs, status);
    return cudaGetLastError() == cudaSuccess ? SEV_OK : SEV_ERR_CUDA;
}
