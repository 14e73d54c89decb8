// band_step.cuh -- band-to-band reduction b -> h (Algorithm 4.2) for bands of up
// to 128 and targets of up to 64, as a chain of steps in which every block
// reflector is applied as soon as it exists.
//
// Step (i, j) of sweep i, with r = i h + (j - 1) b, n_r = min(n - r, b) and the
// block reflector H_j = I - U T U^T of rows [r, r + n_r):
//   D: the diagonal block X = B[r : r + n_r, same] gets H_j^T X H_j;
//   M: the block of rows [r + b, r + 2b) and columns [r, r + b) gets M H_j; the
//      QR of its first h columns (they become [R; 0]) is H_{j+1}, and the other
//      columns get H_{j+1}^T M.
// Step (i, 0) forms H_1 from columns [(i-1) h, i h).  (As printed, the QR and the
// product H_{j+1}^T M belong to chase j + 1; nothing reads these entries in
// between, so the matrix is the same and M is read and written once a sweep.)
//
// Order.  Step (i, j) works on columns [r, r + b); step (i - 1, j + 2) starts
// at column r + 2b - h >= r + b, so they run side by side, and sweep i trails
// sweep i - 1 by two steps (three when the QR of chase j + 1 is left to chase
// j + 1).  In detail, with C1 the first h columns of M and C2 the others, M of
// step (i, j) needs C1 and D of step (i - 1, j + 1) and C2 of step (i - 1, j);
// D needs D of (i - 1, j + 1) and C2 of (i - 1, j).
//
// Roles.  What bounds a stage is (n / h) times [the chain of one step + the time
// until a step's results are published]: the chain is W = M (U T), the update of
// C1 and its QR; D and C2 need not wait for it.  So three roles work on a sweep
// at the same time: role 0 the chain, role 1 D, roles 2 (and 3) C2 (half each).
//   Narrow FP32 bands (MULTI = false): one CTA per sweep, a role is four warps,
//     U and U T pass through shared memory.
//   Wide bands, and FP64 (whose products keep an SM's FP64 pipes busy for tens
//     of thousands of cycles): a role is a CTA of eight warps, U and U T pass
//     through a ring in global memory (they are off the chain there).
// The same arithmetic per entry in both.  Roles publish their progress per sweep
// with release stores; every wait is capped.  Each role takes sweeps from a
// counter of its own in order, so the smallest unfinished sweep is always held
// by running CTAs (MULTI: the launch is cooperative, all roles run).
//
// T is never formed: with G = U^T U (a by-product of the QR's dot products) the
// columns of U T follow from (U T) T^{-1} = U, T^{-1} = diag(1/tau) + striu(G),
// row by row in registers; T^T U^T X = (U T)^T X.
//
// QR (step_qr): four warps, lane = row, columns dealt to the warps; one barrier
// and one set of warp sums per column: with x the current column below its
// diagonal entry and v = e + x / (alpha - beta), every warp sums x^T a for its
// columns and x^T x at once, before the scalars are known.  ~0.9K cycles per
// column in FP32 (1.1K at b = 128; FP64 4.8K, its pipe) against ~2.8K for an owner
// warp that first updates its column, then forms the reflector, with T's
// recurrence in between.  A step of 128 -> 32: 45% of it the QR, then U T, M (U T)
// and the loads.
// Measured (GB300): 64 -> 16 at n = 8192, FP32: 48.1 -> 13.9 ms; 128 -> 32 and
// 32 -> 16 together at n = 16384: 200 -> 72 ms; 128 -> 64 at n = 6000 44 -> 21 ms;
// 32 -> 16 at n = 3001, FP64: 95.5 -> 19.8 ms; 32 -> 16 -> 8 -> 4 -> 2 at n = 512, FP64: 67.0
// -> 14.8 ms.
#pragma once
#include "regtile.cuh"

namespace sev {

// ------------------------------------------------------------ sizes, layout
__host__ __device__ __forceinline__ int step_num_steps(int n, int b, int h, int i) {
    return n - i * h < 2 ? 0 : (n - 2 - i * h) / b + 1;
}
__host__ __device__ __forceinline__ int step_num_sweeps(int n, int h) { return n >= 2 ? (n - 2) / h : 0; }

// Strides: columns of length b padded to ldb, rows of length h to ldu (both
// multiples of 4, and 4 mod 8: 16-byte accesses of 8 lanes spread over the banks).
struct StepDims {
    int b, h, b4, h4, ldb, ldu;
    __host__ __device__ StepDims(int b_, int h_) : b(b_), h(h_) {
        b4 = (b + 3) & ~3;
        h4 = (h + 3) & ~3;
        ldb = b4 + 4;
        ldu = h4 + 4;
    }
    // U (ldb x h4, columns), U T (the same), U T by rows (ldu x b4)
    __host__ __device__ int set_elems() const { return 2 * ldb * h4 + ldu * b4; }
};
constexpr int kStepSets = 4;     // sets of (U, U T) per sweep in flight
constexpr int kStepFlags = 8;    // flags per sweep: progress of roles 0-3, loads of roles 2, 3, sets
constexpr int kStepThreadsRole = 128, kStepThreadsMulti = 256;

template <typename T, int RT, int Q>
struct StepSmem {
    // elements: role 0: M, W, G, two column buffers, tau, scratch; role 1: X, W, Z;
    // role 2: M, and W, whose place Z takes
    static __host__ __device__ int role0(const StepDims &d) {
        return d.ldb * d.b4 + d.ldb * d.h4 + 4 * Q * (4 * Q + 4) + 2 * 32 * RT + 4 * Q + 16;
    }
    static __host__ __device__ int role1(const StepDims &d) { return d.ldb * d.b4 + d.ldb * d.h4 + d.ldu * d.h4; }
    static __host__ __device__ int role2(const StepDims &d) { return d.ldb * d.b4 + d.ldb * d.h4; }
    static __host__ __device__ size_t bytes(int b, int h, bool multi) {
        const StepDims d(b, h);
        const int m01 = role0(d) > role1(d) ? role0(d) : role1(d);
        const int m = m01 > role2(d) ? m01 : role2(d);
        const int e = multi ? m + d.set_elems() : role0(d) + role1(d) + role2(d) + kStepSets * d.set_elems();
        return sizeof(T) * (size_t)e;
    }
};

// ----------------------------------------------------- products of a group
template <typename T, int K>
__device__ __forceinline__ void vec_ld(const T *p, T (&v)[K]) {
    if constexpr (sizeof(T) == 4 && K == 4) {
        const float4 x = *reinterpret_cast<const float4 *>(p);
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
    } else if constexpr (sizeof(T) == 4 && K == 2) {
        const float2 x = *reinterpret_cast<const float2 *>(p);
        v[0] = x.x, v[1] = x.y;
    } else if constexpr (sizeof(T) == 8 && K % 2 == 0) {
#pragma unroll
        for (int i = 0; i < K; i += 2) {
            const double2 x = *reinterpret_cast<const double2 *>(p + i);
            v[i] = x.x, v[i + 1] = x.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) v[i] = p[i];
    }
}

// f(m, n, sum_k A1(m, k) B1(n, k) + sum_k A2(m, k) B2(n, k)) for m < M, n < N:
// A(m, k) = A[m + k lda], B(n, k) = B[n + k ldb] (m, n contiguous; the second
// pair only when TWO).  Threads tid of nt take TM x TN tiles; operands are read
// up to the tile edges (padded storage).  LOWER: only tiles that reach the
// diagonal or below.
template <typename T, int TM, int TN, bool TWO, bool LOWER, typename F>
__device__ __forceinline__ void grp_outer(int tid, int nt, int M, int N, int K, const T *A1, int lda1, const T *B1,
                                          int ldb1, const T *A2, int lda2, const T *B2, int ldb2, F f) {
    const int Mb = (M + TM - 1) / TM, Nb = (N + TN - 1) / TN;
    for (int blk = tid; blk < Mb * Nb; blk += nt) {
        const int m0 = (blk % Mb) * TM, n0 = (blk / Mb) * TN;
        if (LOWER && m0 + TM - 1 < n0) continue;
        T acc[TM][TN];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
        const T *pa = A1 + m0, *pb = B1 + n0;
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            T a[TM], bb[TN];
            vec_ld<T, TM>(pa + k * lda1, a);
            vec_ld<T, TN>(pb + k * ldb1, bb);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmat(a[i], bb[j], acc[i][j]);
        }
        if constexpr (TWO) {
            const T *qa = A2 + m0, *qb = B2 + n0;
#pragma unroll 4
            for (int k = 0; k < K; ++k) {
                T a[TM], bb[TN];
                vec_ld<T, TM>(qa + k * lda2, a);
                vec_ld<T, TN>(qb + k * ldb2, bb);
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) acc[i][j] = fmat(a[i], bb[j], acc[i][j]);
            }
        }
#pragma unroll
        for (int j = 0; j < TN; ++j)
#pragma unroll
            for (int i = 0; i < TM; ++i)
                if (m0 + i < M && n0 + j < N) f(m0 + i, n0 + j, acc[i][j]);
    }
}

// f(m, n, sum_k A(k, m) B(k, n)), A[k + m lda], B[k + n ldb] (k contiguous; K a
// multiple of 4, padded with zeros in A).  With N odd the last tile reads one
// column past B -- of the pad or of the buffer behind it -- and drops the result.
template <typename T, int TM, int TN, typename F>
__device__ __forceinline__ void grp_dot(int tid, int nt, int M, int N, int K, const T *A, int lda, const T *B, int ldb,
                                        F f) {
    const int Mb = (M + TM - 1) / TM, Nb = (N + TN - 1) / TN;
    for (int blk = tid; blk < Mb * Nb; blk += nt) {
        const int m0 = (blk % Mb) * TM, n0 = (blk / Mb) * TN;
        T acc[TM][TN];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
#pragma unroll 2
        for (int k = 0; k < K; k += 4) {
            T a[TM][4], bb[TN][4];
#pragma unroll
            for (int i = 0; i < TM; ++i) vec_ld<T, 4>(A + (m0 + i) * lda + k, a[i]);
#pragma unroll
            for (int j = 0; j < TN; ++j) vec_ld<T, 4>(B + (n0 + j) * ldb + k, bb[j]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) acc[i][j] = fmat(a[i][u], bb[j][u], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (m0 + i < M && n0 + j < N) f(m0 + i, n0 + j, acc[i][j]);
    }
}

__device__ __forceinline__ void step_bar(int id, int nt) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nt) : "memory"); }

// The same barrier, returning whether any of its threads passed a nonzero
// `stop`: every thread of the group takes the same decision to leave (a flag in
// memory could change between their reads, and a group that splits up would
// wait for itself at its next barrier).
__device__ __forceinline__ bool step_bar_or(int id, int nt, int stop) {
    int r;
    asm volatile(
        "{\n"
        " .reg .pred p, q;\n"
        " setp.ne.s32 p, %3, 0;\n"
        " bar.red.or.pred q, %1, %2, p;\n"
        " selp.s32 %0, 1, 0, q;\n"
        "}\n"
        : "=r"(r)
        : "r"(id), "r"(nt), "r"(stop)
        : "memory");
    return r != 0;
}

// ------------------------------------------------------------------- QR
// Householder QR of the m x h block held by four warps (warp w, lane l:
// a[q][t] = row l + 32 t of column w + 4 q; rows >= m and columns >= h zero), r =
// min(m - 1, h) reflectors.  On return column c holds R on and above the
// diagonal and v_c below it, tau[c] the scalars (zero for c >= r), G[c ldg + k] =
// v_c^T v_k for c < k < r.  Barrier `bar` is for these 128 threads.
template <typename T, int RT, int Q>
__device__ __forceinline__ int step_qr(int w, T (&a)[Q][RT], int m, int h, T *xs, T *G, T *tau, T *red, int bar) {
    constexpr int LDG = 4 * Q + 4;
    // two columns per FMA, selects on a column replaced by branches: fewer
    // instructions where they bound the step (128 -> 32 at n = 16384, FP32 49.0 -> 45.6
    // ms, 32 -> 16 at 8191 12.4 -> 11.6); 64 -> 16 and FP64 are 1% faster without
    constexpr bool PACK = sizeof(T) == 4 && RT != 2;
    const int lane = threadIdx.x & 31;
    const int r = m - 1 < h ? (m - 1 > 0 ? m - 1 : 0) : h;
    // the largest entry: the block is held times its power of two, so that no
    // square or product that matters over- or underflows.  (All of it, not x alone:
    // x may be 1e-140 of it, x^T a is multiplied by 1 / (alpha - beta) afterwards,
    // and with a at 1e-190 as it came x^T a had underflowed before.)
    T mx = T(0);
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int t = 0; t < RT; ++t) mx = max(mx, (T)fabs(a[q][t]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red[w] = mx;
    for (int c = (w * 32 + lane); c < 4 * Q; c += 128) tau[c] = T(0);
    step_bar(bar, 128);
    mx = max(max(red[0], red[1]), max(red[2], red[3]));
    T scale, unscale;
    if constexpr (sizeof(T) == 4) {
        int e = (int)((__float_as_uint((float)mx) >> 23) & 0xff) - 126;  // mx < 2^e
        if (mx == 0.f || e > 126) e = mx == 0.f ? 0 : 126;
        if (e < -125) e = -125;
        scale = __uint_as_float((unsigned)(127 - e) << 23);
        unscale = __uint_as_float((unsigned)(127 + e) << 23);
    } else {
        int e = (int)(((unsigned)__double2hiint((double)mx) >> 20) & 0x7ff) - 1022;
        if (mx == 0.0 || e > 1000) e = mx == 0.0 ? 0 : 1000;
        if (e < -1000) e = -1000;
        scale = pow2i(-e);
        unscale = pow2i(e);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int t = 0; t < RT; ++t) a[q][t] *= scale;
    if (w == 0) {
#pragma unroll
        for (int t = 0; t < RT; ++t) xs[lane + 32 * t] = a[0][t];
    }
    step_bar(bar, 128);
    for (int k = 0; k < r; ++k) {
        const T *xk = xs + (k & 1) * (32 * RT);
        const T alpha = xk[k];
        T xr[RT], d[Q];
#pragma unroll
        for (int t = 0; t < RT; ++t) {
            const T x = xk[lane + 32 * t];  // rows < k are zero
            xr[t] = lane + 32 * t == k ? T(0) : x;
        }
        if constexpr (PACK) {
            float2 dd[Q / 2];
#pragma unroll
            for (int p = 0; p < Q / 2; ++p) dd[p] = make_float2(0.f, 0.f);
#pragma unroll
            for (int t = 0; t < RT; ++t) {
                const float2 xx = make_float2(xr[t], xr[t]);
#pragma unroll
                for (int p = 0; p < Q / 2; ++p) dd[p] = ffma2(xx, make_float2(a[2 * p][t], a[2 * p + 1][t]), dd[p]);
            }
#pragma unroll
            for (int p = 0; p < Q / 2; ++p) {
                d[2 * p] = dd[p].x;
                d[2 * p + 1] = dd[p].y;
            }
        } else {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                d[q] = T(0);
#pragma unroll
                for (int t = 0; t < RT; ++t) d[q] = fmat(xr[t], a[q][t], d[q]);
            }
        }
        T tk = T(0), beta = T(0), inv = T(0), s[Q];
        if constexpr (sizeof(T) == 4) {
            F2 p = two_prod((float)xr[0], (float)xr[0]);
#pragma unroll
            for (int t = 1; t < RT; ++t) p = f2_add(p, two_prod((float)xr[t], (float)xr[t]));
            const T sd = warp_sums_t<T, Q>(d);
            const F2 ssq = warp_sum_f2(p);
#pragma unroll
            for (int q = 0; q < Q; ++q) s[q] = __shfl_sync(0xffffffffu, sd, q * (32 / Q));
            float tf = 0.f, bf = 0.f, vf = 0.f;
            // (a column 1e-16 times smaller than the block's largest entry counts as zero)
            if (fmaf((float)alpha, (float)alpha, ssq.hi) >= 1e-32f) house_scalars_f2((float)alpha, ssq, &tf, &bf, &vf);
            tk = (T)tf, beta = (T)bf, inv = (T)vf;
        } else {
            double p = (double)xr[0] * (double)xr[0];
#pragma unroll
            for (int t = 1; t < RT; ++t) p = fma((double)xr[t], (double)xr[t], p);
            const double ssq = warp_sum(p);
            const T sd = warp_sums_t<T, Q>(d);
#pragma unroll
            for (int q = 0; q < Q; ++q) s[q] = __shfl_sync(0xffffffffu, sd, q * (32 / Q));
            double td = 0.0, bd = 0.0, id = 0.0;
            if (fma((double)alpha, (double)alpha, ssq) >= 1e-280) house_scalars((double)alpha, ssq, &td, &bd, &id);
            tk = (T)td, beta = (T)bd, inv = (T)id;
        }
        T v[RT], ms[Q];
#pragma unroll
        for (int t = 0; t < RT; ++t) v[t] = lane + 32 * t == k ? T(1) : xr[t] * inv;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int c = w + 4 * q;
            const T rk = __shfl_sync(0xffffffffu, rsel<RT>(a[q], k >> 5), k & 31);
            s[q] = fmat(inv, s[q], rk);
            ms[q] = c > k ? -tk * s[q] : T(0);
            if (c < k && lane == 0) G[c * LDG + k] = s[q];
        }
        const int k1 = k + 1;
        if constexpr (PACK) {
#pragma unroll
            for (int t = 0; t < RT; ++t) {
                const float2 vv = make_float2(v[t], v[t]);
#pragma unroll
                for (int p = 0; p < Q / 2; ++p) {
                    const float2 u = ffma2(make_float2(ms[2 * p], ms[2 * p + 1]), vv, make_float2(a[2 * p][t], a[2 * p + 1][t]));
                    a[2 * p][t] = u.x;
                    a[2 * p + 1][t] = u.y;
                }
            }
            if (k1 < r && (k1 & 3) == w) {
                T *xn = xs + (k1 & 1) * (32 * RT);
                const unsigned pick = 1u << (k1 >> 2);
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if ((pick >> q) & 1) {
#pragma unroll
                        for (int t = 0; t < RT; ++t) xn[lane + 32 * t] = lane + 32 * t >= k1 ? a[q][t] : T(0);
                    }
            }
            if ((k & 3) == w) {
                const unsigned pick = 1u << (k >> 2);
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if ((pick >> q) & 1) {
#pragma unroll
                        for (int t = 0; t < RT; ++t) {
                            const int g = lane + 32 * t;
                            a[q][t] = g > k ? v[t] : (g == k && tk != T(0) ? beta : a[q][t]);
                        }
                    }
            }
        } else {
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int t = 0; t < RT; ++t) {
                    const int g = lane + 32 * t;
                    const T u = fmat(ms[q], v[t], a[q][t]);
                    a[q][t] = w + 4 * q == k ? (g > k ? v[t] : (g == k && tk != T(0) ? beta : a[q][t])) : u;
                }
            if (k1 < r && (k1 & 3) == w) {
                T *xn = xs + (k1 & 1) * (32 * RT);
                const unsigned pick = 1u << (k1 >> 2);
#pragma unroll
                for (int t = 0; t < RT; ++t) {
                    T x = a[0][t];
#pragma unroll
                    for (int q = 1; q < Q; ++q) x = (pick >> q) & 1 ? a[q][t] : x;
                    xn[lane + 32 * t] = lane + 32 * t >= k1 ? x : T(0);
                }
            }
        }
        if (w == 0 && lane == 0) tau[k] = tk;
        step_bar(bar, 128);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int t = 0; t < RT; ++t)
            if (lane + 32 * t <= w + 4 * q) a[q][t] *= unscale;
    return r;
}

// U explicit into set (rows >= m and columns >= r zero), then U T row by row:
// (U T)(., k) = tau_k (U(., k) - sum_{q < k} (U T)(., q) G(q, k)).
template <typename T, int RT, int Q>
__device__ __forceinline__ void step_make_set(int w, const T (&a)[Q][RT], int m, int r, const StepDims &D, T *set,
                                              const T *G, const T *tau, int bar) {
    constexpr int LDG = 4 * Q + 4, LPR = 4 / RT, HPL = 4 * Q / LPR;
    const int lane = threadIdx.x & 31;
    T *U = set, *UTc = U + D.ldb * D.h4, *UTt = UTc + D.ldb * D.h4;
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int t = 0; t < RT; ++t) {
            const int g = lane + 32 * t, c = w + 4 * q;
            if (g < D.b4 && c < D.h4)
                U[g + c * D.ldb] = c < r && g < m ? (g < c ? T(0) : (g == c ? T(1) : a[q][t])) : T(0);
        }
    step_bar(bar, 128);
    // LPR lanes share a row (row = this warp's share), columns dealt to them
    constexpr int RPW = 32 / LPR;
    const int row = w * RPW + lane % RPW, g = lane / RPW;
    T acc[HPL];
#pragma unroll
    for (int i = 0; i < HPL; ++i) {
        const int c = g + LPR * i;
        acc[i] = row < D.b4 && c < D.h4 ? U[row + c * D.ldb] : T(0);
    }
#pragma unroll
    for (int k = 0; k < 4 * Q; ++k) {
        if (k < r) {
            const T mine = tau[k] * acc[k / LPR];
            const T val = LPR == 1 ? mine : __shfl_sync(0xffffffffu, mine, lane % RPW + RPW * (k % LPR));
            if (g == k % LPR) acc[k / LPR] = val;
            // (columns c >= r take whatever G holds there; they are dropped below)
            if constexpr (LPR == 1) {
#pragma unroll
                for (int c4 = (k + 1) & ~3; c4 < HPL; c4 += 4) {
                    T gv[4];
                    vec_ld<T, 4>(G + k * LDG + c4, gv);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (c4 + u > k) acc[c4 + u] = fmat(-val, gv[u], acc[c4 + u]);
                }
            } else {
#pragma unroll
                for (int i = k / LPR; i < HPL; ++i) {
                    const int c = g + LPR * i;
                    if (c > k) acc[i] = fmat(-val, G[k * LDG + c], acc[i]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < HPL; ++i) {
        const int c = g + LPR * i;
        if (row < D.b4 && c < D.h4) {
            const T v = c < r ? acc[i] : T(0);
            UTc[row + c * D.ldb] = v;
            UTt[c + row * D.ldu] = v;
        }
    }
}

// --------------------------------------------------------------- the kernel
template <typename T>
struct StepArgs {
    int n, ldab, b, h, nsweeps, slots, sms;
    T *AB;
    int *flags;  // kStepFlags per sweep
    int *ctr;    // sweep counters of the roles
    T *ring;     // slots x kStepSets sets (MULTI)
    int *err;
};

// One group's view: its threads, its barrier, and the waits it makes.
struct StepGroup {
    int tid, nt, bar;
    long long cap;
    int *err;
    volatile int *abort;
    __device__ __forceinline__ void sync() const { step_bar(bar, nt); }
    // One thread's wait for *f >= need (need <= 0: none); true when it failed.
    __device__ __forceinline__ bool flag_failed(const int *f, int need) const {
        return need > 0 && wait_flag(f, need, cap, err, [&] { return any_gave_up(err) || *abort; }) < 0;
    }
    // One thread's wait for a counter in this CTA's shared memory; true when it failed.
    __device__ __forceinline__ bool local_failed(const volatile int *f, int need) const {
        const long long t0 = clock64();
        while (*f < need) {
            if (*abort) return true;
            if (wait_expired(t0, cap)) {
                latch_timeout(err);
                return true;
            }
        }
        __threadfence_block();
        return false;
    }
    // The group's barrier; false when any of its threads failed a wait.
    __device__ __forceinline__ bool sync_ok(bool failed) const {
        __syncwarp();
        if (!step_bar_or(bar, nt, failed)) return true;
        *abort = 1;
        return false;
    }
    // flags f[k] >= need[k] (k < 4), then the group's barrier
    __device__ __forceinline__ bool wait4(const int *f, int n0, int n1, int n2, int n3) const {
        bool failed = false;
        if (tid < 4) failed = flag_failed(f + tid, tid == 0 ? n0 : (tid == 1 ? n1 : (tid == 2 ? n2 : n3)));
        return sync_ok(failed);
    }
};

// Two CTAs per SM (more sweeps at once: 64 -> 16 at n = 8192 15.0 ms, with one 16.2)
// where the block in registers leaves room for it.
template <typename T, int RT, int Q, bool MULTI>
constexpr int step_min_blocks() {
    return MULTI ? (RT * Q * sizeof(T) <= 64 ? 2 : 1) : (RT == 1 ? 2 : 1);
}

template <typename T, int RT, int Q, bool MULTI>
__global__ void __launch_bounds__(MULTI ? kStepThreadsMulti : 3 * kStepThreadsRole, step_min_blocks<T, RT, Q, MULTI>())
    band_step_kernel(StepArgs<T> P) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ volatile int s_abort, s_sweep;
    __shared__ volatile int s_sets, s_ld, s_done[3];  // MULTI = false: this sweep's sets, loads of role 2, steps done
    const StepDims D(P.b, P.h);
    const int n = P.n, b = P.b, h = P.h, ldab = P.ldab, ldb = D.ldb, ldu = D.ldu;
    T *const AB = P.AB;
    using SM = StepSmem<T, RT, Q>;
    constexpr int TN = RT == 1 ? 1 : (RT == 2 ? 2 : 4);   // columns per tile of the thin products
    constexpr int DN = RT == 1 ? 1 : 2;
    // (FP64: an SM's second block in another role than its first: a chain beside a C2 half)
    const int turn = sizeof(T) == 8 ? 2 * (int)(blockIdx.x / P.sms) : 0;
    const int role = MULTI ? ((int)blockIdx.x + turn) & 3 : (int)(threadIdx.x >> 7);
    StepGroup g;
    g.nt = MULTI ? kStepThreadsMulti : kStepThreadsRole;
    g.tid = MULTI ? (int)threadIdx.x : (int)(threadIdx.x & 127);
    g.bar = MULTI ? 1 : 1 + role;
    g.cap = wait_cap(P.err);
    g.err = P.err;
    g.abort = &s_abort;
    const int warp = g.tid >> 5, lane = g.tid & 31, nw = g.nt >> 5;
    // this role's buffers
    T *base = (T *)smem;
    T *sets = base;  // MULTI: one set; else kStepSets of them, shared by the roles
    base += (MULTI ? 1 : kStepSets) * D.set_elems();
    if (!MULTI) base += role == 0 ? 0 : (role == 1 ? SM::role0(D) : SM::role0(D) + SM::role1(D));
    T *const Ms = base, *const Ws = Ms + ldb * D.b4, *const Xtra = Ws + ldb * D.h4;
    {
        // every pad that a tile may read is finite from here on
        const size_t e = SM::bytes(b, h, MULTI) / sizeof(T);
        for (size_t k = threadIdx.x; k < e; k += blockDim.x) ((T *)smem)[k] = T(0);
    }
    if (threadIdx.x == 0) s_abort = 0;
    auto set_of = [&](int j) { return sets + (MULTI ? 0 : (j % kStepSets) * D.set_elems()); };
    auto ring_of = [&](int s, int j) {
        return P.ring + ((size_t)(s % P.slots) * kStepSets + j % kStepSets) * (size_t)D.set_elems();
    };
    // rows [0, m) x all b columns of M of the step at r0 into Ms, rows up to b4 zeroed
    auto load_m = [&](int r0, int m) {
        constexpr int U = 8;
        for (int c0 = warp; c0 < b; c0 += nw * U) {
            T v[U][RT];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int t = 0; t < RT; ++t) {
                    const int c = c0 + nw * u, a = lane + 32 * t;
                    v[u][t] = c < b && a < m ? __ldcg(AB + (b + a - c) + (size_t)(r0 + c) * ldab) : T(0);
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int t = 0; t < RT; ++t) {
                    const int c = c0 + nw * u, a = lane + 32 * t;
                    if (c < b && a < D.b4) Ms[a + c * ldb] = v[u][t];
                }
        }
    };
    // W = M (U T) (m x h)
    auto make_w = [&](const T *set, int m, int kk) {
        grp_outer<T, 4, TN, false, false>(
            g.tid, g.nt, m, h, kk, Ms, ldb, set + 2 * ldb * D.h4, ldu, (const T *)nullptr, 0, (const T *)nullptr, 0,
            [&](int i, int c, T v) { Ws[i + c * ldb] = v; });
    };

    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            // (after a failed wait of any group: no further sweep)
            s_sweep = s_abort ? P.nsweeps : atomicAdd(P.ctr + (MULTI ? role : 0), 1);
            s_sets = s_ld = 0;
            s_done[0] = s_done[1] = s_done[2] = 0;
        }
        __syncthreads();
        const int s = s_sweep;
        if (s >= P.nsweeps) break;
        const int i = s + 1;
        const int J = step_num_steps(n, b, h, i), Jp = i > 1 ? step_num_steps(n, b, h, i - 1) : 0;
        int *const mine = P.flags + (size_t)s * kStepFlags;
        const int *const prev = mine - kStepFlags;
        bool ok = true;
        // progress of this role for the next sweep (after the group's barrier)
        auto publish = [&](int j) {
            g.sync();
            if (g.tid == 0) {
                if (!MULTI) {
                    __threadfence_block();
                    s_done[role] = j;
                }
                st_release(mine + role, j);
                if (!MULTI && role == 2) st_release(mine + 3, j);
            }
        };
        // set j produced by role 0 is in this role's shared memory; ld > 0: and the
        // role with the other half of C2 has read M of step ld
        auto need_set = [&](int j, int ld = 0) {
            if constexpr (MULTI) {
                const bool failed = (g.tid == 0 && g.flag_failed(mine + 6, j)) ||
                                    (g.tid == 32 && g.flag_failed(mine + 2 + (role ^ 1), ld));
                if (!g.sync_ok(failed)) return false;
                const float4 *src = (const float4 *)ring_of(s, j);
                float4 *dst = (float4 *)sets;
                batched_copy<float4, 4>(
                    D.set_elems() * (int)sizeof(T) / 16, g.tid, g.nt, [&](int k) { return __ldcg(src + k); },
                    [&](int k, float4 v) { dst[k] = v; });
                g.sync();
                return true;
            } else {
                return g.sync_ok(g.tid == 0 && g.local_failed(&s_sets, j));
            }
        };

        if (role == 0) {
            // ------------------------------------------------ role 0: the chain
            T *const G = Xtra, *const xs = G + 4 * Q * (4 * Q + 4), *const tau = xs + 2 * 32 * RT, *const red = tau + 4 * Q;
            const int qbar = MULTI ? 2 : g.bar;
            if constexpr (MULTI) {
                // the ring slot is free once the sweep that used it is complete
                if (s >= P.slots) {
                    const int *old = P.flags + (size_t)(s - P.slots) * kStepFlags;
                    const int Jo = step_num_steps(n, b, h, i - P.slots);
                    ok = g.wait4(old, 0, Jo, Jo, Jo);
                }
            }
            for (int j = 0; j <= J && ok; ++j) {
                const int r0 = i * h + (j - 1) * b;  // first row of H_j
                if (i > 1) ok = g.wait4(prev, min(j + 1, Jp), min(j + 1, Jp), min(j, Jp), min(j, Jp));
                if (!ok) break;
                const int m = min(n - (j == 0 ? i * h : r0 + b), b);  // rows of the block to factorise
                const bool next = j < J;                              // m >= 2
                if (j > 0 && m > 0) {
                    const T *set = set_of(j);
                    load_m(r0, m);
                    g.sync();
                    make_w(set, m, b);
                    g.sync();
                    grp_outer<T, 4, TN, false, false>(
                        g.tid, g.nt, m, h, h, Ws, ldb, set, ldb, (const T *)nullptr, 0, (const T *)nullptr, 0,
                        [&](int a, int c, T v) { Ms[a + c * ldb] -= v; });
                    g.sync();
                }
                T a[Q][RT];
                if (next && warp < 4) {
#pragma unroll
                    for (int q = 0; q < Q; ++q)
#pragma unroll
                        for (int t = 0; t < RT; ++t) {
                            const int c = warp + 4 * q, row = lane + 32 * t;
                            T v = T(0);
                            if (c < h && row < m)
                                v = j > 0 ? Ms[row + c * ldb]
                                          : __ldcg(AB + (h + row - c) + (size_t)(i * h - h + c) * ldab);
                            a[q][t] = v;
                        }
                    const int r = step_qr<T, RT, Q>(warp, a, m, h, xs, G, tau, red, qbar);
                    // the set's place is free once step j + 1 - kStepSets is complete everywhere
                    if (!MULTI)
                        ok = g.sync_ok(g.tid == 0 && (g.local_failed(&s_done[1], j + 1 - kStepSets) ||
                                                      g.local_failed(&s_done[2], j + 1 - kStepSets)));
                    step_make_set<T, RT, Q>(warp, a, m, r, D, set_of(j + 1), G, tau, qbar);
                }
                g.sync();
                if (next) {
                    if constexpr (MULTI) {
                        if (j + 1 > kStepSets)
                            ok = g.wait4(mine, 0, j + 1 - kStepSets, j + 1 - kStepSets, j + 1 - kStepSets);
                        float4 *dst = (float4 *)ring_of(s, j + 1);
                        const float4 *src = (const float4 *)sets;
                        for (int k = g.tid; k < D.set_elems() * (int)sizeof(T) / 16; k += g.nt) dst[k] = src[k];
                        g.sync();
                        if (g.tid == 0) st_release(mine + 6, j + 1);
                    } else if (g.tid == 0) {
                        __threadfence_block();
                        s_sets = j + 1;
                    }
                }
                // C1 back, once roles 2 (and 3) have read M
                if (j > 0 && m > 0) {
                    bool failed = false;
                    if constexpr (MULTI) {
                        if (g.tid < 2) failed = g.flag_failed(mine + 4 + g.tid, j);
                    } else if (g.tid == 0) {
                        failed = g.local_failed(&s_ld, j);
                    }
                    if (!g.sync_ok(failed)) break;
                }
                if (next) {
                    if (warp < 4) {
#pragma unroll
                        for (int q = 0; q < Q; ++q)
#pragma unroll
                            for (int t = 0; t < RT; ++t) {
                                const int c = warp + 4 * q, row = lane + 32 * t;
                                if (c < h && row < m) {
                                    const int d = (j > 0 ? b : h) + row - c, col = j > 0 ? r0 + c : i * h - h + c;
                                    AB[d + (size_t)col * ldab] = row <= c ? a[q][t] : T(0);
                                }
                            }
                    }
                } else if (m > 0) {
                    for (int k = g.tid; k < m * h; k += g.nt) {
                        const int row = k % m, c = k / m;
                        AB[(b + row - c) + (size_t)(r0 + c) * ldab] = Ms[row + c * ldb];
                    }
                }
                publish(j);
            }
        } else if (role == 1) {
            // --------------------------------------- role 1: the diagonal blocks
            T *const Zs = Xtra;
            for (int j = 1; j <= J; ++j) {
                const int r0 = i * h + (j - 1) * b, m = min(n - r0, b);
                // self-check: the step lies in the matrix, and there is a next one if and
                // only if two rows or more are left for it (every access of all roles is
                // bounded by the rows that n leaves, so a wrong count touches nothing else)
                if (g.tid == 0 && (r0 < h || m < 2 || (j < J) != (n - r0 - b >= 2))) latch_error(P.err, SEV_ERR_INTERNAL);
                if (i > 1 && !g.wait4(prev, 0, min(j + 1, Jp), min(j, Jp), min(j, Jp))) break;
                // lower triangle, mirrored (zeros past m)
                constexpr int U = RT == 4 ? 4 : 8;
                for (int c0 = warp; c0 < D.b4; c0 += nw * U) {
                    T v[U][RT];
#pragma unroll
                    for (int u = 0; u < U; ++u)
#pragma unroll
                        for (int t = 0; t < RT; ++t) {
                            const int c = c0 + nw * u, a = lane + 32 * t;
                            v[u][t] = c < m && a < m && a >= c ? __ldcg(AB + (a - c) + (size_t)(r0 + c) * ldab) : T(0);
                        }
#pragma unroll
                    for (int u = 0; u < U; ++u)
#pragma unroll
                        for (int t = 0; t < RT; ++t) {
                            const int c = c0 + nw * u, a = lane + 32 * t;
                            if (c < D.b4 && a < D.b4 && a >= c) {
                                Ms[a + c * ldb] = v[u][t];
                                Ms[c + a * ldb] = v[u][t];
                            }
                        }
                }
                if (!need_set(j)) break;
                const T *U0 = set_of(j), *UTc = U0 + ldb * D.h4;
                make_w(U0, m, m);
                g.sync();
                // Z = (U T)^T W, then V = U Z / 2 - W in place of W
                grp_dot<T, 2, DN>(g.tid, g.nt, D.h4, D.h4, D.b4, UTc, ldb, Ws, ldb,
                                  [&](int a, int c, T v) { Zs[c + a * ldu] = v; });
                g.sync();
                grp_outer<T, 4, TN, false, false>(
                    g.tid, g.nt, m, h, h, U0, ldb, Zs, ldu, (const T *)nullptr, 0, (const T *)nullptr, 0,
                    [&](int a, int c, T v) { Ws[a + c * ldb] = fmat(T(0.5), v, -Ws[a + c * ldb]); });
                g.sync();
                grp_outer<T, 4, RT == 1 ? 2 : 4, true, true>(g.tid, g.nt, m, m, h, U0, ldb, Ws, ldb, Ws, ldb, U0, ldb,
                                                             [&](int a, int c, T v) {
                                                                 if (a >= c)
                                                                     AB[(a - c) + (size_t)(r0 + c) * ldab] =
                                                                         Ms[a + c * ldb] + v;
                                                             });
                publish(j);
            }
        } else {
            // ------------------------- roles 2, 3: the other columns of M, half each
            T *const Zt = Ws;  // (Z is formed once W has been used)
            const int w2 = b - h;
            int c_lo = h, nc = w2;
            if constexpr (MULTI) {
                const int half = ((w2 + 1) / 2 + 3) & ~3;
                if (role == 2) {
                    nc = min(half, w2);
                } else {
                    c_lo = h + min(half, w2);
                    nc = w2 - min(half, w2);
                }
            }
            bool have = false;  // the set in shared memory is H_j's (MULTI)
            for (int j = 1; j <= J; ++j) {
                const int r0 = i * h + (j - 1) * b, m = min(n - (r0 + b), b);
                if (i > 1 && !g.wait4(prev, min(j + 1, Jp), min(j + 1, Jp), min(j, Jp), min(j, Jp))) break;
                if (m > 0) {
                    load_m(r0, m);
                    g.sync();
                    if (g.tid == 0) {
                        if (MULTI)
                            st_release(mine + 2 + role, j);  // flags 4, 5
                        else {
                            __threadfence_block();
                            s_ld = j;
                        }
                    }
                    if (!(MULTI && have) && !need_set(j)) break;
                    const T *U0 = set_of(j);
                    make_w(U0, m, b);
                    g.sync();
                    const bool next = j < J;
                    // M is written back once every role that needs all of it has read it:
                    // role 0 before it makes set j + 1, in the last step before it is
                    // complete; the other half's role as its flag says
                    if (!next) {
                        bool failed = false;
                        if constexpr (MULTI) {
                            if (g.tid == 0) failed = g.flag_failed(mine, j);
                            if (g.tid == 32) failed = g.flag_failed(mine + 2 + (role ^ 1), j);
                        } else if (g.tid == 0) {
                            failed = g.local_failed(&s_done[0], j);
                        }
                        if (!g.sync_ok(failed)) break;
                    }
                    auto c2 = [&](int a, int c, T v) {
                        T &x = Ms[a + c * ldb];
                        x -= v;
                        if (!next) AB[(b + a - c) + (size_t)(r0 + c) * ldab] = x;
                    };
                    // TN rows of U are read at once, from a multiple of TN on; other
                    // targets: FP64 starts before c_lo and drops what lies there, FP32 reads
                    // single rows (starting early costs FP32 128 -> 32 2%, the other branch
                    // FP64 64 -> 16 3%, both without need)
                    if constexpr (sizeof(T) == 8) {
                        const int off = c_lo & (TN - 1);
                        grp_outer<T, 4, TN, false, false>(g.tid, g.nt, m, nc + off, h, Ws, ldb, U0 + c_lo - off, ldb,
                                                          (const T *)nullptr, 0, (const T *)nullptr, 0,
                                                          [&](int a, int c, T v) {
                                                              if (c >= off) c2(a, c_lo - off + c, v);
                                                          });
                    } else if (c_lo % TN == 0) {
                        grp_outer<T, 4, TN, false, false>(g.tid, g.nt, m, nc, h, Ws, ldb, U0 + c_lo, ldb,
                                                          (const T *)nullptr, 0, (const T *)nullptr, 0,
                                                          [&](int a, int c, T v) { c2(a, c_lo + c, v); });
                    } else {
                        grp_outer<T, 4, 1, false, false>(g.tid, g.nt, m, nc, h, Ws, ldb, U0 + c_lo, ldb,
                                                         (const T *)nullptr, 0, (const T *)nullptr, 0,
                                                         [&](int a, int c, T v) { c2(a, c_lo + c, v); });
                    }
                    g.sync();
                    if (next) {
                        if (!need_set(j + 1, j)) break;
                        have = true;
                        const T *U1 = set_of(j + 1), *UTc = U1 + ldb * D.h4;
                        grp_dot<T, 2, DN>(g.tid, g.nt, D.h4, nc, D.b4, UTc, ldb, Ms + c_lo * ldb, ldb,
                                          [&](int a, int c, T v) { Zt[c + a * ldb] = v; });
                        g.sync();
                        grp_outer<T, 4, TN, false, false>(
                            g.tid, g.nt, m, nc, h, U1, ldb, Zt, ldb, (const T *)nullptr, 0, (const T *)nullptr, 0,
                            [&](int a, int c, T v) {
                                AB[(b + a - c_lo - c) + (size_t)(r0 + c_lo + c) * ldab] = Ms[a + (c_lo + c) * ldb] - v;
                            });
                    }
                }
                publish(j);
            }
        }
    }
}

// -------------------------------------------------------------------- host
inline bool step_shape_ok(int b, int h) { return b >= 2 && b <= 128 && h <= 64; }
inline int step_rt(int b) { return b <= 32 ? 1 : (b <= 64 ? 2 : 4); }
inline int step_q(int h) { return h <= 8 ? 2 : (h <= 16 ? 4 : (h <= 32 ? 8 : 16)); }

// Sweeps in flight at most: sweep i runs two steps behind sweep i - 1.
constexpr int kStepMaxSlots = 160;
inline int step_slots(int n, int b, int h) {
    const int busy = step_num_steps(n, b, h, 1) / 2 + 4, ns = step_num_sweeps(n, h);
    const int s = busy < kStepMaxSlots ? busy : kStepMaxSlots;
    return s < ns ? s : ns;
}
inline size_t step_workspace(int n, int b, int h) {
    if (!step_shape_ok(b, h)) return 0;
    const int ns = step_num_sweeps(n, h);
    Carver c(nullptr);
    c.take<int>((size_t)kStepFlags * (ns + 1) + 8);
    c.take<double>((size_t)step_slots(n, b, h) * kStepSets * StepDims(b, h).set_elems());
    return c.bytes();
}

template <typename T, int RT, int Q, bool MULTI>
int launch_step(sev_ctx *hd, int n, T *AB, int ldab, int b, int h, void *ws, size_t ws_bytes) {
    const size_t smem = StepSmem<T, RT, Q>::bytes(b, h, MULTI);
    if (smem + 1024 > hd->smem_optin) return SEV_ERR_UNSUPPORTED;
    if (ws_bytes < step_workspace(n, b, h)) return SEV_ERR_WORKSPACE;
    auto kern = band_step_kernel<T, RT, Q, MULTI>;
    SEV_CUDA(allow_smem(hd, (const void *)kern));
    const int threads = MULTI ? kStepThreadsMulti : 3 * kStepThreadsRole;
    int per_sm = 0;
    SEV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    if (per_sm < 1) return SEV_ERR_UNSUPPORTED;
    StepArgs<T> P;
    P.n = n;
    P.ldab = ldab;
    P.b = b;
    P.h = h;
    P.AB = AB;
    P.err = hd->d_err;
    P.nsweeps = step_num_sweeps(n, h);
    int groups = hd->sm_count * per_sm / (MULTI ? 4 : 1);
    const int most = MULTI ? step_slots(n, b, h) : step_num_steps(n, b, h, 1) / 2 + 4;
    if (groups > most) groups = most;
    // The steps of a wide FP64 band keep an SM's FP64 pipes busy, and a second CTA on
    // the SM stretches its step: one CTA per SM until more than twice as many sweeps
    // could run (32 -> 16 at n = 3001 23.5 -> 19.8 ms, 64 -> 16 at 8192 102 -> 90),
    // above that all of them, the second CTA of an SM in another role than the
    // first (32 -> 16 at n = 6000: 57.3 ms with one CTA per SM, 55.7 with two of the
    // same role, 49.7).  Narrow bands lose by it (4 -> 2 at n = 512).
    P.sms = hd->sm_count < 8 ? 4 : hd->sm_count & ~3;
    if (MULTI && sizeof(T) == 8 && b >= 32 && groups > P.sms / 4 && most <= P.sms / 2) groups = P.sms / 4;
    if (groups > P.nsweeps) groups = P.nsweeps;
    if (groups < 1) groups = 1;
    P.slots = groups;
    Carver c(ws);
    const size_t nflags = (size_t)kStepFlags * (P.nsweeps + 1) + 8;
    P.flags = c.take<int>(nflags);
    P.ctr = P.flags + nflags - 8;
    P.ring = (T *)c.take<double>((size_t)step_slots(n, b, h) * kStepSets * StepDims(b, h).set_elems());
    SEV_CUDA(cudaMemsetAsync(P.flags, 0, sizeof(int) * nflags, hd->stream));
    // The four CTAs of a sweep need one another, so they have to start together: a
    // cooperative launch.  (Launched freely, some roles of a sweep could hold SMs
    // while a cooperative grid on another stream -- a panel, a bisection -- held the
    // rest and waited for these: neither went on until a wait ran out.  Clusters of
    // four would do as well, but only 36 of them fit at once where 38 sweeps do:
    // 128 -> 32 at n = 16384 47.0 ms against 45.7, 32 -> 16 at n = 3001 in FP64 24.7
    // against 19.9, two CTAs of a cluster sharing an SM.)  One CTA per sweep goes on by
    // itself, whatever part of the grid runs.
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.gridDim = dim3((unsigned)(MULTI ? 4 * groups : groups));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = hd->stream;
    cfg.attrs = at;
    cfg.numAttrs = MULTI ? 1 : 0;
    timing_begin(hd, K_BAND_CHASE);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, P);
    timing_end(hd, K_BAND_CHASE);
    return e == cudaSuccess ? SEV_OK : SEV_ERR_CUDA;
}

}  // namespace sev
