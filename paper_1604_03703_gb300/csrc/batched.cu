// batched.cu -- eigenvalues of many independent small symmetric matrices in
// one persistent launch.  The paper treats one matrix; batching is this
// library's addition for workloads of many small uneven matrices (a
// sequence of SCF-style eigenproblems).  Each matrix runs the paper's path
// unchanged, inside one CTA:
//
//   full-to-band (Algorithm 4.1) -- per panel the Householder QR of the
//     N x b panel (the tree of Algorithm 3.2 with a single leaf: the panel
//     fits in shared memory), the compact-WY factor T (Cor. 3.7's form
//     Q = I - U T U^T) and the two-sided update A22 += U V^T + V U^T with
//     V = U (T^T U^T A22 U T) / 2 - A22 U T (Eq. 4.1);
//   b -> 1 band reduction (Algorithm 4.2 with h = 1) on the whole band held
//     in shared memory: every warp owns one sweep at a time, and step (i, j)
//     of band_tri.cu starts once sweep i - 1 has finished step j + 1;
//   Sturm bisection of the tridiagonal (the final step of Algorithm 4.3).
//
// CTAs take matrices from a global queue (the host orders it largest
// first), so the launch load-balances uneven sizes by itself.  The matrix
// is overwritten (both triangles: the kernel first mirrors the lower
// triangle).
//
// What bounds it: 4096 FP32 matrices of order 32..512 (b = 16) 147.7 -> 85.6 ms,
// 60% of it the bisection's FP64 recurrence; 500 FP64 ones (b = 8) 136 -> 95.5 ms, the
// FP64 pipes (2 FMA per cycle and SM) in every phase and the largest matrices'
// own time.  Nothing is allocated and nothing waits on the host, so the
// launch can be captured in a CUDA graph.
#include "band_step.cuh"
#include "sturm.cuh"
#include "tri_step.cuh"

namespace sev {

constexpr int kBatchThreads = 256;
constexpr int kBatchWarps = kBatchThreads / 32;
constexpr int kDone = 2047;  // chase counter value of a finished sweep

struct BatchMat {
    void *A;
    double *eigs;
    int n;
    int lda;
};

template <typename T, int B>
struct BatchLayout {
    // columns of the panel buffers: a multiple of 4 for 16-byte loads
    static __host__ __device__ int ldp(int nmax) { return (nmax + 3) & ~3; }
    // partial sums of U^T Y: one share per warp, fewer where eight would
    // outgrow the bisection's arrays, whose place they take
    static constexpr int NS = B == 32 ? 2 : (B * sizeof(T) == 128 ? 4 : kBatchWarps);
    // full-to-band: U, Y (ldp x B each), T (B x B), tau (B); then the band:
    // nmax columns x 2B diagonals in the same place
    static __host__ __device__ size_t x_off(int nmax) {
        const size_t f = 2 * (size_t)ldp(nmax) * B + (size_t)B * B + B, b = (size_t)nmax * 2 * B;
        return (sizeof(T) * (f > b ? f : b) + 15) & ~(size_t)15;
    }
    // behind it, one after the other in the same place: G, Z and the shares
    // (B x B each); the vectors and counters of the warps' sweeps; d, e, e^2
    // (n doubles each), parameters and reduction scratch of the bisection
    static __host__ __device__ size_t bytes(int nmax) {
        const size_t f = sizeof(T) * (NS + 2) * (size_t)B * B;
        const size_t b = sizeof(T) * 3 * kBatchWarps * kTriVec + sizeof(int) * kBatchWarps;
        const size_t e = sizeof(double) * (3 * (size_t)nmax + 48);
        const size_t fb = f > b ? f : b;
        return x_off(nmax) + (fb > e ? fb : e);
    }
};

// ------------------------------------------------------------ full to band
// G = U^T Y (B x B) in NS shares of the rows: lanes hold the outputs (row
// lane mod B, columns dealt to the lane groups and, with fewer shares than
// warps, to the warps of a share), then the shares are added in order.  (One
// thread per 4 x 4 tile left all but (B/4)^2 threads idle through N steps.)
template <typename T, int B>
__device__ __forceinline__ void batch_uty(int N, const T *U, const T *Y, int ldp, T *share, T *G) {
    constexpr int NS = BatchLayout<T, B>::NS, W = kBatchWarps / NS;
    constexpr int LG = 32 / B < B ? 32 / B : B;  // lane groups (B = 4 leaves 16 lanes over)
    constexpr int CP = B / (LG * W);             // columns of a lane
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int a = lane % B, g = lane / B % LG + LG * (warp / NS), sh = warp % NS;
    T acc[CP];
#pragma unroll
    for (int q = 0; q < CP; ++q) acc[q] = T(0);
#pragma unroll 2
    for (int i = sh; i < N; i += NS) {
        const T u = U[i + (size_t)a * ldp];
#pragma unroll
        for (int q = 0; q < CP; ++q) acc[q] = fmat(u, Y[i + (size_t)(g + LG * W * q) * ldp], acc[q]);
    }
    if (lane < B * LG) {
#pragma unroll
        for (int q = 0; q < CP; ++q) share[sh * B * B + a + (g + LG * W * q) * B] = acc[q];
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < B * B; idx += kBatchThreads) {
        T s = share[idx];
#pragma unroll
        for (int w = 1; w < NS; ++w) s += share[w * B * B + idx];
        G[idx] = s;
    }
    __syncthreads();
}

// A22 += U V^T + V U^T, both triangles: the lower tiles are computed and
// written to both places.  A warp takes patches of 32 x 16 entries, its lanes
// 8 x 4 tiles of 4 x 4: one shared-memory wavefront feeds all lanes of an
// operand, and the lower and the mirrored entries both fill half of the
// sectors they touch (whole rows of tiles would leave one of the two
// scattered).  A thread's entries of A are on their way while it multiplies.
// Against two full products of 4 x 4 tiles that each read and write all of A22:
// 8.7 -> 1.4 s of CTA time over the 4096 FP32 matrices, 6.7 -> 3.4 s over the
// 500 FP64 ones (the FP64 pipe's floor).
template <typename T, int B>
__device__ __forceinline__ void batch_syr2k(int N, T *A, int lda, const T *U, const T *V, int ldp) {
    const int lane = threadIdx.x & 31;
    const int PR = (N + 31) >> 5, PC = (N + 15) >> 4;
    for (int p = threadIdx.x >> 5, R = 0; p < PR * (PR + 1); p += kBatchWarps) {
        while ((R + 1) * (R + 2) <= p) ++R;  // 2 R + 2 patches in patch row R
        const int C = p - R * (R + 1);
        const int m0 = 32 * R + 4 * (lane & 7), n0 = 16 * C + 4 * (lane >> 3);
        if (C >= PC || m0 >= N || m0 + 3 < n0) continue;
        T old[4][4], acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                old[i][j] = (m0 + i < N && m0 + i >= n0 + j) ? A[(m0 + i) + (size_t)(n0 + j) * lda] : T(0);
                acc[i][j] = T(0);
            }
#pragma unroll 4
        for (int k = 0; k < B; ++k) {
            T um[4], vm[4], un[4], vn[4];
            vec_ld<T, 4>(U + m0 + k * ldp, um);
            vec_ld<T, 4>(V + m0 + k * ldp, vm);
            vec_ld<T, 4>(U + n0 + k * ldp, un);
            vec_ld<T, 4>(V + n0 + k * ldp, vn);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmat(vm[i], un[j], fmat(um[i], vn[j], acc[i][j]));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int m = m0 + i, n = n0 + j;
                if (m < N && m >= n) {
                    const T v = old[i][j] + acc[i][j];
                    A[m + (size_t)n * lda] = v;
                    if (m > n) A[n + (size_t)m * lda] = v;
                }
            }
    }
}

template <typename T, int B>
__device__ void batch_full_to_band(T *A, int n, int lda, unsigned char *smem, int nmax) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int ldp = BatchLayout<T, B>::ldp(nmax);
    T *U = (T *)smem;
    T *Y = U + (size_t)ldp * B;
    T *Tm = Y + (size_t)ldp * B;
    T *tau = Tm + B * B;
    T *G = (T *)(smem + BatchLayout<T, B>::x_off(nmax));
    T *Z = G + B * B;
    T *share = Z + B * B;
    for (int c0 = 0; c0 + B < n; c0 += B) {
        const int r0 = c0 + B, N = n - r0;
        if (N < 2) break;
        T *A22 = A + r0 + (size_t)r0 * lda;
        batched_copy<T>(
            N * B, tid, nt, [&](int k) { return A[(r0 + k % N) + (size_t)(c0 + k / N) * lda]; },
            [&](int k, T v) { U[k % N + (size_t)(k / N) * ldp] = v; });
        __syncthreads();
        const int r = cta_qr(N, B, U, ldp, tau, nullptr);
        // the band block: R's upper triangle (rows r0.., columns c0..)
        for (int idx = tid; idx < B * B; idx += nt) {
            const int i = idx % B, j = idx / B;
            if (i <= j && i < N) A[(r0 + i) + (size_t)(c0 + j) * lda] = U[i + (size_t)j * ldp];
        }
        cta_form_t(N, r, U, ldp, tau, Tm, B, G, B);
        // explicit U (unit lower trapezoidal, zero columns r..B-1), T padded with zeros
        for (int idx = tid; idx < N * B; idx += nt) {
            const int i = idx % N, c = idx / N;
            const T v = U[i + (size_t)c * ldp];
            U[i + (size_t)c * ldp] = (c < r) ? (i < c ? T(0) : (i == c ? T(1) : v)) : T(0);
        }
        for (int idx = tid; idx < B * B; idx += nt) {
            const int a = idx % B, c = idx / B;
            if (a >= r || c >= r) Tm[idx] = T(0);
        }
        __syncthreads();
        // Y = A22 U;  G = U^T Y;  Z = G T;  G = T^T Z  (= T^T U^T A22 U T)
        cta_gemm<T, false, false>(N, B, N, T(1), A22, lda, U, ldp, T(0), Y, ldp);
        __syncthreads();
        batch_uty<T, B>(N, U, Y, ldp, share, G);
        cta_gemm<T, false, false>(B, B, B, T(1), G, B, Tm, B, T(0), Z, B);
        __syncthreads();
        cta_gemm<T, true, false>(B, B, B, T(0.5), Tm, B, Z, B, T(0), G, B);
        __syncthreads();
        // V = U G - Y T (G holds half), row by row in place of Y
        for (int i = tid; i < N; i += nt) {
            T y[B], u[B];
#pragma unroll
            for (int q = 0; q < B; ++q) {
                y[q] = Y[i + (size_t)q * ldp];
                u[q] = U[i + (size_t)q * ldp];
            }
#pragma unroll 4
            for (int c = 0; c < B; ++c) {
                T acc = 0;
#pragma unroll
                for (int k = 0; k < B; ++k) acc = fma(u[k], G[k + c * B], fma(-y[k], Tm[k + c * B], acc));
                Y[i + (size_t)c * ldp] = acc;
            }
        }
        __syncthreads();
        // both triangles: the next panel's product reads all of A22
        batch_syr2k<T, B>(N, A22, lda, U, Y, ldp);
        __syncthreads();
    }
}

// ------------------------------------------------------------- band to 1
// Returns false if a wait hit its cap.  (With the one-warp chase of blocks in
// registers, sweeps three chases apart: 9.6 s of CTA time over the 4096 FP32
// matrices; so 2.6 s.)
template <typename T, int B>
__device__ bool batch_band_to_tri(const T *A, int n, int lda, unsigned char *smem, int nmax, int *err) {
    constexpr int LDW = 2 * B;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31;
    T *band = (T *)smem;
    T *vb = (T *)(smem + BatchLayout<T, B>::x_off(nmax));  // per warp: v of this step and the next, scratch
    volatile int *sval = (volatile int *)(vb + 3 * kBatchWarps * kTriVec);
    __shared__ int s_fail;
    for (int idx = tid; idx < n * LDW; idx += nt) {
        const int c = idx / LDW, d = idx % LDW;
        band[idx] = (d <= B && c + d < n) ? A[(c + d) + (size_t)c * lda] : T(0);
    }
    if (tid < kBatchWarps) sval[tid] = 0;
    if (tid == 0) s_fail = 0;
    __syncthreads();
    constexpr int S = 1 << 30;  // no ring: the whole band lies in the window
    const int nsweeps = n >= 3 ? n - 2 : 0;
    const long long cap = wait_cap(err);
    T *const vw = vb + 3 * warp * kTriVec, *const wb = vw + 2 * kTriVec;
    for (int i = 1 + warp; i <= nsweeps; i += kBatchWarps) {
        const int Ji = tri_chases(n, B, i);
        const int Jp = i > 1 ? tri_chases(n, B, i - 1) : 0;
        T rv[TriLanes<B>::CPL], rtau = T(0);
#pragma unroll
        for (int q = 0; q < TriLanes<B>::CPL; ++q) rv[q] = T(0);
        for (int j = 0; j <= Ji; ++j) {
            if (i > 1) {
                const int need = (i - 1) * 2048 + (j + 1 <= Jp ? j + 1 : kDone);
                int ok = 1;
                if (lane == 0) {
                    const long long t0 = clock64();
                    while (sval[(i - 2) % kBatchWarps] < need) {
                        if (*(volatile int *)&s_fail || wait_expired(t0, cap)) {
                            ok = 0;
                            break;
                        }
                    }
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) {
                    if (lane == 0) {
                        latch_error(err, SEV_ERR_TIMEOUT);
                        s_fail = 1;
                    }
                    i = nsweeps + 1;  // leave both loops
                    break;
                }
                __threadfence_block();
            }
            const int o = i + (j - 1) * B;
            T *cur = vw + (j & 1) * kTriVec, *nxt = vw + ((j + 1) & 1) * kTriVec;
            if (j == 0) {
                tri_first<T, B, S>(band, n, i, nxt, rv, rtau);
            } else if (o + 2 * B <= n) {
                tri_diag<T, B, S, true, false>(band, n, o, cur, wb);
                tri_bulge<T, B, S, true, false>(band, n, o, rv, rtau, nxt);
            } else {
                tri_diag<T, B, S, false, false>(band, n, o, cur, wb);
                tri_bulge<T, B, S, false, false>(band, n, o, rv, rtau, nxt);
            }
            __threadfence_block();
            __syncwarp();
            if (lane == 0) sval[(i - 1) % kBatchWarps] = i * 2048 + (j == Ji ? kDone : j);
        }
    }
    __syncthreads();
    return s_fail == 0;
}

// A matrix that holds a NaN or an Inf has no eigenvalues to find: as in the
// single-matrix path the error is latched and they are NaN.
__device__ __forceinline__ void batch_nonfinite(int n, double *eigs, int *err) {
    if (threadIdx.x == 0) latch_error(err, SEV_ERR_NONFINITE);
    for (int k = threadIdx.x; k < n; k += blockDim.x) eigs[k] = __longlong_as_double(0x7ff8000000000000LL);
}

// -------------------------------------------------------------- bisection
// The same scaling, minors count, stopping rule and IEEE operations as
// bisect.cu, on shared-memory d and (e 2^-s)^2.  20.4 -> 15.8 s of CTA time over
// the 4096 FP32 matrices with the first levels shared.
template <typename T, int B>
__device__ void batch_bisect(int n, int nmax, unsigned char *smem, double rtol, double *eigs, int *err) {
    constexpr int LDW = 2 * B;
    const int tid = threadIdx.x, nt = blockDim.x;
    const T *band = (const T *)smem;
    double *d = (double *)(smem + BatchLayout<T, B>::x_off(nmax));
    double *e = d + nmax;
    double *e2s = e + nmax;
    double *par = e2s + nmax;  // gl, gu, sc, tnorm, 2^s, zero, no tiny e2s
    double *red = par + 8;     // 32
    for (int i = tid; i < n; i += nt) {
        d[i] = (double)band[(size_t)i * LDW];
        e[i] = i + 1 < n ? (double)band[(size_t)i * LDW + 1] : 0.0;
    }
    __syncthreads();
    double lo = INFINITY, hi = -INFINITY;
    bool bad = false;  // an entry that the reductions left non-finite (fmin and fmax would pass over a NaN)
    for (int i = tid; i < n; i += nt) {
        double r = 0.0;
        if (i > 0) r = __dadd_rn(r, fabs(e[i - 1]));
        if (i + 1 < n) r = __dadd_rn(r, fabs(e[i]));
        bad |= !isfinite(__dadd_rn(fabs(d[i]), r));
        lo = fmin(lo, __dsub_rn(d[i], r));
        hi = fmax(hi, __dadd_rn(d[i], r));
    }
    if (__syncthreads_or(bad)) {
        batch_nonfinite(n, eigs, err);
        return;
    }
    lo = -block_max(-lo, red);
    hi = block_max(hi, red);
    if (tid == 0) {
        double tnorm = fmax(fabs(lo), fabs(hi));
        int s = 0;
        if (tnorm > 0.0) (void)frexp(tnorm, &s);
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
        par[6] = 1.0;
    }
    __syncthreads();
    const double sc = par[2];
    for (int i = tid; i < n; i += nt) {
        if (i + 1 < n) {
            const double es = __dmul_rn(e[i], sc), e2 = __dmul_rn(es, es);
            e2s[i] = e2;
            if (es != 0.0 && e2 < 0x1p-322) par[6] = 0.0;
        } else {
            e2s[i] = 0.0;
        }
    }
    __syncthreads();
    const double atol = __dmul_rn(rtol, par[3]);
    const bool zero = par[5] != 0.0, plain = par[6] != 0.0;
    const double lo0 = par[0], hi0 = par[1];
    // One step of the bisection on [a, b] (the operations of bisect.cu):
    // 0 with the midpoint to count at, 1 converged, 2 step cap.
    auto step = [&](double a, double b, int it, double &mid) {
        const double w = __dsub_rn(b, a);
        const double mag = fmax(fabs(a), fabs(b));
        double tol = __dmul_rn(rtol, mag);
        if (atol > tol) tol = atol;
        if (w <= tol) return 1;
        if (it >= 200) return 2;
        mid = __dmul_rn(0.5, __dadd_rn(a, b));
        return mid <= a || mid >= b ? 1 : 0;
    };
    auto count = [&](double x) {
        return sturm_count_blocks<4>(
            n, [&](int i) { return d[i]; }, [&](int i) { return e2s[i]; }, x, sc, plain);
    };
    // All indices share the first levels: the counts at the midpoints of the
    // first L levels (a tree of 2^L - 1 <= n of them, one thread each) serve
    // every index, L counts less per index with the same operations -- at
    // 1e-9 about a quarter of the FP64 work, which bounds this phase.
    int L = 0;
    while (L < 8 && (2 << L) - 1 <= n) ++L;
    int *cnt = (int *)e;  // (e is not needed past e2s)
    if (!zero)
        for (int m = tid; m < (1 << L) - 1; m += nt) {
            // node m in heap order: the bits of m + 1 below the leading one are the turns
            double a = lo0, b = hi0, mid = 0.0;
            int it = 0, c = -1;
            bool live = true;
            for (int l = 30 - __clz(m + 1); l >= 0 && live; --l) {
                live = step(a, b, it, mid) == 0;
                if (((m + 1) >> l) & 1)
                    a = mid;
                else
                    b = mid;
                ++it;
            }
            if (live && step(a, b, it, mid) == 0) c = count(mid);
            cnt[m] = c;
        }
    __syncthreads();
    for (int k = tid; k < n; k += nt) {
        double a = lo0, b = hi0, mid = 0.0;
        int node = 0;
        for (int it = 0; !zero; ++it) {
            const int r = step(a, b, it, mid);
            if (r == 2) latch_error(err, SEV_ERR_NOCONV);
            if (r != 0) break;
            const int c = it < L ? cnt[node] : count(mid);
            if (c >= k + 1) {
                b = mid;
                node = 2 * node + 1;
            } else {
                a = mid;
                node = 2 * node + 2;
            }
        }
        eigs[k] = zero ? 0.0 : __dmul_rn(__dmul_rn(0.5, __dadd_rn(a, b)), par[4]);
    }
    __syncthreads();
}

// ----------------------------------------------------------------- kernel
template <typename T, int B>
__global__ void __launch_bounds__(kBatchThreads) batch_eig_kernel(int count, const BatchMat *__restrict__ mats,
                                                                   int *queue, int nmax, double rtol, int *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_idx;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_idx = atomicAdd(queue, 1);
        __syncthreads();
        const int q = s_idx;
        if (q >= count) return;
        const BatchMat m = mats[q];
        T *A = (T *)m.A;
        const int n = m.n, lda = m.lda;
        if (n <= 0) continue;
        if (n == 1) {
            if (threadIdx.x == 0) {
                m.eigs[0] = (double)A[0];
                if (!isfinite(A[0])) latch_error(err, SEV_ERR_NONFINITE);
            }
            continue;
        }
        // mirror the lower triangle: the panel products read all of A22
        bool bad = false;
        for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
            const int i = idx % n, j = idx / n;
            if (i <= j) {
                const T v = A[j + (size_t)i * lda];
                bad |= !isfinite(v);
                A[i + (size_t)j * lda] = v;
            }
        }
        if (__syncthreads_or(bad)) {
            batch_nonfinite(n, m.eigs, err);
            continue;
        }
        batch_full_to_band<T, B>(A, n, lda, smem, nmax);
        if (!batch_band_to_tri<T, B>(A, n, lda, smem, nmax, err)) return;
        batch_bisect<T, B>(n, nmax, smem, rtol, m.eigs, err);
    }
}

int batch_supported(int b, int elem) { return b == 4 || b == 8 || b == 16 || (b == 32 && elem == 4); }

template <typename T>
size_t batch_smem_bytes(int b, int nmax) {
    switch (b) {
        case 4: return BatchLayout<T, 4>::bytes(nmax);
        case 8: return BatchLayout<T, 8>::bytes(nmax);
        case 16: return BatchLayout<T, 16>::bytes(nmax);
        case 32: return BatchLayout<T, 32>::bytes(nmax);
        default: return 0;
    }
}

// Host preparation (outside any stream capture): opt in to the kernel's
// dynamic shared memory and size the persistent grid.
template <typename T, int B>
static int prepare_batch_b(sev_ctx *h, int count, int nmax, int *grid) {
    const size_t smem = BatchLayout<T, B>::bytes(nmax);
    if (smem > h->smem_optin) return SEV_ERR_UNSUPPORTED;
    auto kern = batch_eig_kernel<T, B>;
    SEV_CUDA(allow_smem(h, (const void *)kern));
    int per_sm = 0;
    SEV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kBatchThreads, smem));
    if (per_sm < 1) return SEV_ERR_UNSUPPORTED;
    int g = h->sm_count * per_sm;
    if (g > count) g = count;
    *grid = g;
    return SEV_OK;
}

template <typename T, int B>
static int launch_batch_b(sev_ctx *h, int count, const BatchMat *mats, int *queue, int nmax, double rtol, int grid) {
    const size_t smem = BatchLayout<T, B>::bytes(nmax);
    SEV_CUDA(cudaMemsetAsync(queue, 0, sizeof(int), h->stream));
    auto kern = batch_eig_kernel<T, B>;
    SEV_LAUNCH(h, K_BATCH, kern, grid, kBatchThreads, smem, count, mats, queue, nmax, rtol, h->d_err);
    return SEV_OK;
}

template <typename T>
int prepare_batch_small(sev_ctx *h, int count, int b, int nmax, int *grid) {
    switch (b) {
        case 4: return prepare_batch_b<T, 4>(h, count, nmax, grid);
        case 8: return prepare_batch_b<T, 8>(h, count, nmax, grid);
        case 16: return prepare_batch_b<T, 16>(h, count, nmax, grid);
        case 32:
            if constexpr (sizeof(T) == 4) return prepare_batch_b<T, 32>(h, count, nmax, grid);
            return SEV_ERR_UNSUPPORTED;
        default: return SEV_ERR_UNSUPPORTED;
    }
}

template <typename T>
int launch_batch_small(sev_ctx *h, int count, const void *mats, int *queue, int b, int nmax, double rtol, int grid) {
    if (count <= 0) return SEV_OK;
    const BatchMat *m = (const BatchMat *)mats;
    switch (b) {
        case 4: return launch_batch_b<T, 4>(h, count, m, queue, nmax, rtol, grid);
        case 8: return launch_batch_b<T, 8>(h, count, m, queue, nmax, rtol, grid);
        case 16: return launch_batch_b<T, 16>(h, count, m, queue, nmax, rtol, grid);
        case 32:
            if constexpr (sizeof(T) == 4) return launch_batch_b<T, 32>(h, count, m, queue, nmax, rtol, grid);
            return SEV_ERR_UNSUPPORTED;
        default: return SEV_ERR_UNSUPPORTED;
    }
}

size_t batch_mat_bytes() { return sizeof(BatchMat); }

void batch_pack_mat(void *dst, void *A, double *eigs, int n, int lda) {
    BatchMat m;
    m.A = A;
    m.eigs = eigs;
    m.n = n;
    m.lda = lda;
    *(BatchMat *)dst = m;
}


// ---------------------------------------------------------------- autotune
// Synthetic symmetric matrices for timing candidate band widths: the lower
// triangle gets uniform(-1, 1) entries from a counter-based hash (splitmix64
// of the matrix index and the entry index).
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

template <typename T>
__global__ void batch_fill_kernel(int count, const BatchMat *__restrict__ mats, unsigned long long seed) {
    for (int q = blockIdx.x; q < count; q += gridDim.x) {
        const BatchMat m = mats[q];
        T *A = (T *)m.A;
        for (int idx = threadIdx.x; idx < m.n * m.n; idx += blockDim.x) {
            const int i = idx % m.n, j = idx / m.n;
            if (i < j) continue;
            const unsigned long long r = splitmix64(seed ^ ((unsigned long long)q << 32) ^ (unsigned long long)idx);
            A[i + (size_t)j * m.lda] = (T)((double)(r >> 11) * 0x1.0p-52 - 1.0);
        }
    }
}

template <typename T>
int launch_batch_fill(sev_ctx *h, int count, const void *mats, unsigned long long seed) {
    if (count <= 0) return SEV_OK;
    SEV_LAUNCH(h, K_MISC, batch_fill_kernel<T>, count < 4096 ? count : 4096, 256, 0, count, (const BatchMat *)mats,
               seed);
    return SEV_OK;
}
template int launch_batch_fill<float>(sev_ctx *, int, const void *, unsigned long long);
template int launch_batch_fill<double>(sev_ctx *, int, const void *, unsigned long long);

template int launch_batch_small<float>(sev_ctx *, int, const void *, int *, int, int, double, int);
template int launch_batch_small<double>(sev_ctx *, int, const void *, int *, int, int, double, int);
template int prepare_batch_small<float>(sev_ctx *, int, int, int, int *);
template int prepare_batch_small<double>(sev_ctx *, int, int, int, int *);
template size_t batch_smem_bytes<float>(int, int);
template size_t batch_smem_bytes<double>(int, int);

}  // namespace sev
