// band.cu -- band-to-band reduction b -> h (Algorithm 4.2) on packed lower
// band storage, as one persistent kernel per stage.
//
// Chase (i, j) (1-based, as in the algorithm): with h the target width,
//   o_qr.r = (i-1)h + (j-1)b + h
//   j = 1: o_qr.c = o_qr.r - h, o_v = 0,     o_up.c = o_qr.r,      n_c = min(n - o_up.c, 2b)
//   j > 1: o_qr.c = o_qr.r - b, o_v = b - h, o_up.c = o_qr.c + h,  n_c = min(n - o_up.c, 3b - h)
//   n_r = min(n - o_qr.r, b); the chase exists while n - o_qr.r >= 2
// and performs: QR of B[qr rows, qr cols] (n_r x h); write [R; 0];
// W = B[up cols, qr rows] U T; V = -W; V[v rows] += 1/2 U (T^T (U^T W[v rows]));
// B[qr rows, up cols] += U V^T and the mirrored B[up cols, qr rows] += V U^T.
// With lower storage the mirrored pair is one entry: rows of W outside the
// qr rows get X <- X - (X U T) U^T (one-sided), the qr-row block gets the
// symmetric rank-2 update U V^T + V U^T.
//
// Schedule.  A CTA takes sweeps i in increasing order (global counter) and
// runs its chases j = 1, 2, ... (the grid is capped to the ~J/3 sweeps that
// can progress together); chase (i, j) waits until sweep i-1 has
// completed chase j+2 (or all of its chases).  Chase (i, j) overlaps chase
// (i-1, j+2) -- its bulge rows [o+2b-h, o+2b) are the rows that (i-1, j+2)
// factorises -- so the pipeline t = 2i + j that the Fig. 2 caption pictures
// is not legal; this rule gives t = 3i + j and reproduces the sequential
// order bit for bit.  Sweeps are handed out in order and each CTA finishes
// its sweep before taking another, so every awaited sweep is held by a
// running CTA: the waits cannot deadlock.  Every wait is capped; on expiry
// the kernel latches SEV_ERR_TIMEOUT and returns.
//
// This is the general form, for bands wider than 128 and shapes that the step
// kernel (band_step.cuh) does not take.
#include "common.cuh"

namespace sev {

__host__ __device__ __forceinline__ int band_num_chases(int n, int b, int h, int i) {
    const int r = n - i * h;
    return r < 2 ? 0 : (n - 2 - i * h) / b + 1;
}
__host__ __device__ __forceinline__ int band_num_sweeps(int n, int h) { return n >= 2 ? (n - 2) / h : 0; }

// Band element (r, c) with r >= c; out-of-range indices are a bug: they are
// not dereferenced, the thread's flag `bad` is set and 0 is returned.  The
// flag is a register (OR-ed over the CTA at the end of the kernel): a flag
// in memory would be a store between consecutive loads and keep them from
// being in flight together.
template <typename T>
__device__ __forceinline__ T bld(const T *AB, int ldab, int n, int r, int c, int &bad) {
    const int d = r - c;
    if (d < 0 || d >= ldab || r >= n || c < 0) {
        bad = 1;
        return T(0);
    }
    return __ldcg(AB + d + (size_t)c * ldab);
}
template <typename T>
__device__ __forceinline__ void bst(T *AB, int ldab, int n, int r, int c, T v, int &bad) {
    const int d = r - c;
    if (d < 0 || d >= ldab || r >= n || c < 0) {
        bad = 1;
        return;
    }
    AB[d + (size_t)c * ldab] = v;
}
// Shared memory of one chase: U, U T, the block X being updated, W, T, two
// small products, tau and a reduction scratch.
template <typename T>
struct ChaseSmem {
    T *Us, *UTs, *Xs, *Ws, *Ts, *Zs, *Z2s, *tau;
    double *red;
    int ldb1, ldh1;
    __device__ ChaseSmem(unsigned char *base, int b, int h) {
        ldb1 = b + 4;  // 16-byte aligned columns for vector loads where b is a multiple of 4
        ldh1 = h + 1;
        Us = (T *)base;
        UTs = Us + (size_t)ldb1 * h;
        Xs = UTs + (size_t)ldb1 * h;
        Ws = Xs + (size_t)ldb1 * b;
        Ts = Ws + (size_t)ldb1 * h;
        Zs = Ts + (size_t)ldh1 * h;
        Z2s = Zs + (size_t)ldh1 * h;
        tau = Z2s + (size_t)ldh1 * h;
        size_t off = (size_t)((unsigned char *)(tau + h + 3 * 128) - base);
        off = (off + 15) & ~(size_t)15;
        red = (double *)(base + off);
    }
};

// (3 x 128 entries are spare: the size also decides which shapes the library takes)
template <typename T>
size_t band_smem_bytes(int b, int h) {
    const size_t ldb1 = b + 4, ldh1 = h + 1;
    size_t e = 3 * ldb1 * h + ldb1 * b + 3 * ldh1 * h + h + 3 * 128;
    size_t bytes = e * sizeof(T);
    bytes = (bytes + 15) & ~(size_t)15;
    return bytes + 32 * sizeof(double);
}
// The qr-row diagonal block X_d (n_r x n_r, mirrored in S.Xs) after U, T
// and U T are formed: W_d = X_d (U T); S = U^T W_d; Z = T^T S; V_d = -W_d +
// U Z / 2; X_d += U V_d^T + V_d U^T; the lower triangle written back.
// VEC: 16-byte loads of FP32 operands (b a multiple of 4).
template <typename T, bool VEC>
__device__ void chase_diag_update(T *AB, int ldab, int n, int n_r, int nr, int o_qr_r, ChaseSmem<T> &S, int &bad) {
    const int ldb1 = S.ldb1, ldh1 = S.ldh1;
    const int tid = threadIdx.x, nt = blockDim.x;
    cta_mm<T, 4, 4, false, VEC>(n_r, nr, n_r, T(1), S.Xs, ldb1, S.UTs, ldb1, 0, nullptr, 0, nullptr, 0, T(0), S.Ws,
                                 ldb1);
    __syncthreads();
    cta_gemm<T, true, false>(nr, nr, n_r, T(1), S.Us, ldb1, S.Ws, ldb1, T(0), S.Zs, ldh1);
    __syncthreads();
    // Z = T^T S, every entry at once (T upper triangular): Z(a, c) = sum_{q <= a} T(q, a) S(q, c)
    for (int idx = tid; idx < nr * nr; idx += nt) {
        const int a = idx % nr, c = idx / nr;
        T z = 0;
        for (int q = 0; q <= a; ++q) z += S.Ts[q + (size_t)a * ldh1] * S.Zs[q + (size_t)c * ldh1];
        S.Z2s[a + (size_t)c * ldh1] = z;
    }
    __syncthreads();
    cta_mm<T, 4, 4, false, VEC>(n_r, nr, nr, T(0.5), S.Us, ldb1, S.Z2s, ldh1, 0, nullptr, 0, nullptr, 0, T(-1),
                                 S.Ws, ldb1);
    __syncthreads();
    const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    if (n_r >= 64) {
        // X_d += [U V_d] [V_d U]^T on the tiles on or below the diagonal
        cta_mm<T, 8, 8, true, VEC, true>(n_r, n_r, nr, T(1), S.Us, ldb1, S.Ws, ldb1, nr, S.Ws, ldb1, S.Us, ldb1, T(1),
                                          S.Xs, ldb1);
        __syncthreads();
        // lower triangle, down the columns (band storage: rows of a column contiguous)
        for (int c = warp; c < n_r; c += nw)
            for (int r = c + lane; r < n_r; r += 32)
                bst(AB, ldab, n, o_qr_r + r, o_qr_r + c, S.Xs[r + (size_t)c * ldb1], bad);
    } else {
        for (int c = warp; c < n_r; c += nw)
            for (int r = c + lane; r < n_r; r += 32) {
                T s = 0;
                for (int m = 0; m < nr; ++m)
                    s += S.Us[r + (size_t)m * ldb1] * S.Ws[c + (size_t)m * ldb1] +
                         S.Ws[r + (size_t)m * ldb1] * S.Us[c + (size_t)m * ldb1];
                bst(AB, ldab, n, o_qr_r + r, o_qr_r + c, S.Xs[r + (size_t)c * ldb1] + s, bad);
            }
    }
}

// One chase (i, j) performed by the whole CTA, its QR in shared memory.
template <typename T, bool VEC>
__device__ void band_chase(T *AB, int ldab, int n, int b, int h, int i, int j, ChaseSmem<T> &S, int &bad) {
    const int o_qr_r = (i - 1) * h + (j - 1) * b + h;
    int o_qr_c, o_v, o_up_c, lim;
    if (j == 1) {
        o_qr_c = o_qr_r - h;
        o_v = 0;
        o_up_c = o_qr_r;
        lim = 2 * b;
    } else {
        o_qr_c = o_qr_r - b;
        o_v = b - h;
        o_up_c = o_qr_c + h;
        lim = 3 * b - h;
    }
    const int n_r = min(n - o_qr_r, b);
    const int n_c = min(n - o_up_c, lim);
    const int ldb1 = S.ldb1, ldh1 = S.ldh1;
    const int tid = threadIdx.x, nt = blockDim.x;

    // 1. QR of the n_r x h block
    batched_copy<T>(
        n_r * h, tid, nt, [&](int k) { return bld(AB, ldab, n, o_qr_r + k % n_r, o_qr_c + k / n_r, bad); },
        [&](int k, T v) { S.Xs[k % n_r + (size_t)(k / n_r) * ldb1] = v; });
    __syncthreads();
    const int nr = cta_qr(n_r, h, S.Xs, ldb1, S.tau, S.red);
    // 2. B[qr rows, qr cols] = [R; 0]
    for (int idx = tid; idx < n_r * h; idx += nt) {
        const int r = idx % n_r, c = idx / n_r;
        const T v = (r <= c) ? S.Xs[r + (size_t)c * ldb1] : T(0);
        bst(AB, ldab, n, o_qr_r + r, o_qr_c + c, v, bad);
    }
    if (nr == 0) {
        __syncthreads();
        return;
    }
    cta_extract_u(n_r, nr, nr, S.Xs, ldb1, S.Us, ldb1);
    // 3. T (from G = U^T U by one warp's recurrence when h <= 32) and U T
    if (nr <= 32) {
        __syncthreads();
        cta_gemm<T, true, false>(nr, nr, n_r, T(1), S.Us, ldb1, S.Us, ldb1, T(0), S.Zs, ldh1);
        __syncthreads();
        form_t_from_g(nr, S.Zs, ldh1, S.tau, S.Ts, ldh1);
    } else {
        __syncthreads();
        cta_form_t(n_r, nr, S.Us, ldb1, S.tau, S.Ts, ldh1, S.Zs, ldh1);
    }
    cta_mm<T, 4, 4, false, VEC>(n_r, nr, nr, T(1), S.Us, ldb1, S.Ts, ldh1, 0, nullptr, 0, nullptr, 0, T(0), S.UTs,
                                 ldb1);
    __syncthreads();
    // 4. the qr-row diagonal block X_d (n_r x n_r): two-sided update (the
    //    stored lower triangle, read down its columns, then mirrored)
    batched_copy<T>(
        n_r * n_r, tid, nt,
        [&](int k) {
            const int r = k % n_r, c = k / n_r;
            return r >= c ? bld(AB, ldab, n, o_qr_r + r, o_qr_r + c, bad) : T(0);
        },
        [&](int k, T v) {
            const int r = k % n_r, c = k / n_r;
            if (r >= c) S.Xs[r + (size_t)c * ldb1] = v;
        });
    __syncthreads();
    for (int idx = tid; idx < n_r * n_r; idx += nt) {
        const int r = idx % n_r, c = idx / n_r;
        if (r < c) S.Xs[r + (size_t)c * ldb1] = S.Xs[c + (size_t)r * ldb1];
    }
    __syncthreads();
    chase_diag_update<T, VEC>(AB, ldab, n, n_r, nr, o_qr_r, S, bad);
    __syncthreads();
    // 5. the other rows of W (above: [0, o_v), below: [o_v + n_r, n_c)):
    //    X <- X - (X U T) U^T, in chunks of at most b rows
    for (int part = 0; part < 2; ++part) {
        const int a_begin = part == 0 ? 0 : o_v + n_r;
        const int a_end = part == 0 ? o_v : n_c;
        for (int a0 = a_begin; a0 < a_end; a0 += b) {
            const int rows = min(b, a_end - a0);
            if (part == 0) {
                // rows above the qr rows: element (row, col) is stored as (col, row), contiguous
                // along col -- consecutive threads take consecutive columns
                batched_copy<T>(
                    rows * n_r, tid, nt,
                    [&](int k) { return bld(AB, ldab, n, o_qr_r + k % n_r, o_up_c + a0 + k / n_r, bad); },
                    [&](int k, T v) { S.Xs[k / n_r + (size_t)(k % n_r) * ldb1] = v; });
            } else {
                batched_copy<T>(
                    rows * n_r, tid, nt,
                    [&](int k) { return bld(AB, ldab, n, o_up_c + a0 + k % rows, o_qr_r + k / rows, bad); },
                    [&](int k, T v) { S.Xs[k % rows + (size_t)(k / rows) * ldb1] = v; });
            }
            __syncthreads();
            cta_mm<T, 4, 4, false, VEC>(rows, nr, n_r, T(1), S.Xs, ldb1, S.UTs, ldb1, 0, nullptr, 0, nullptr, 0, T(0),
                                         S.Ws, ldb1);
            __syncthreads();
            // X <- X - W U^T: register-tiled for wide blocks, else folded into the stores
            const bool tiled = n_r >= 64;
            if (tiled) {
                cta_mm<T, 8, 8, true, VEC>(rows, n_r, nr, T(-1), S.Ws, ldb1, S.Us, ldb1, 0, nullptr, 0, nullptr, 0,
                                            T(1), S.Xs, ldb1);
                __syncthreads();
            }
            auto updated = [&](int r, int c) {
                T v = S.Xs[r + (size_t)c * ldb1];
                if (!tiled)
                    for (int m = 0; m < nr; ++m) v -= S.Ws[r + (size_t)m * ldb1] * S.Us[c + (size_t)m * ldb1];
                return v;
            };
            if (part == 0) {
                for (int idx = tid; idx < rows * n_r; idx += nt) {
                    const int c = idx % n_r, r = idx / n_r;
                    bst(AB, ldab, n, o_qr_r + c, o_up_c + a0 + r, updated(r, c), bad);
                }
            } else {
                for (int idx = tid; idx < rows * n_r; idx += nt) {
                    const int r = idx % rows, c = idx / rows;
                    bst(AB, ldab, n, o_up_c + a0 + r, o_qr_r + c, updated(r, c), bad);
                }
            }
            __syncthreads();
        }
    }
}

// Capped wait of one thread until sweep s - 1 has completed `need` chases;
// false on expiry, here or elsewhere (then the error word is set).
__device__ __forceinline__ bool wait_progress(const int *progress, int s, int need, long long cap, int *err) {
    return wait_flag(&progress[s - 1], need, cap, err, [&] { return any_gave_up(err); }) >= 0;
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(kThreads) band_chase_kernel(int n, T *AB, int ldab, int b, int h, int nsweeps,
                                                               int *progress, int *sweep_ctr, int *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    ChaseSmem<T> S(smem, b, h);
    __shared__ int s_sweep, s_abort;
    const long long cap = wait_cap(err);
    int bad = 0;  // this thread met an index outside the band
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            s_sweep = atomicAdd(sweep_ctr, 1);
            s_abort = 0;
        }
        __syncthreads();
        const int s = s_sweep;
        if (s >= nsweeps) break;
        const int i = s + 1;
        const int J = band_num_chases(n, b, h, i);
        const int Jprev = i > 1 ? band_num_chases(n, b, h, i - 1) : 0;
        for (int j = 1; j <= J; ++j) {
            if (i > 1) {
                if (threadIdx.x == 0 && !wait_progress(progress, s, min(j + 2, Jprev), cap, err)) s_abort = 1;
                __syncthreads();
                if (s_abort) return;
            }
            band_chase<T, VEC>(AB, ldab, n, b, h, i, j, S, bad);
            __syncthreads();
            // the release store orders the CTA's writes (made visible to
            // thread 0 by the barrier above) before the progress flag
            if (threadIdx.x == 0) st_release(&progress[s], j);
        }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) latch_error(err, SEV_ERR_INTERNAL);
}

size_t band_chase_workspace(int n, int h) {
    Carver c(nullptr);
    c.take<int>((size_t)band_num_sweeps(n, h) + 1);
    c.take<int>(1);
    return c.bytes();
}
size_t band_workspace(int n, int b, int h) {
    const size_t chase = band_chase_workspace(n, h), step = band_step_workspace(n, b, h);
    return chase > step ? chase : step;
}

template <typename T>
int launch_band_to_band(sev_ctx *hd, int n, T *AB, int ldab, int b, int h, void *ws, size_t ws_bytes) {
    const int nsweeps = band_num_sweeps(n, h);
    if (nsweeps <= 0) return SEV_OK;
    if (ws_bytes < band_chase_workspace(n, h)) return SEV_ERR_WORKSPACE;
    const size_t smem = band_smem_bytes<T>(b, h);
    if (smem > hd->smem_optin) return SEV_ERR_UNSUPPORTED;
    // bands up to 128: the step kernel; this file's chase serves wider bands, the
    // shapes the step kernel has no buffers for, and a workspace without room
    // for its exchange buffers
    if (ws_bytes >= band_workspace(n, b, h)) {
        const int rc = launch_band_step(hd, n, AB, ldab, b, h, ws, ws_bytes);
        if (rc != SEV_ERR_UNSUPPORTED) return rc;
    }
    Carver c(ws);
    int *progress = c.take<int>((size_t)nsweeps + 1);
    int *ctr = c.take<int>(1);
    SEV_CUDA(cudaMemsetAsync(progress, 0, sizeof(int) * ((size_t)nsweeps + 1), hd->stream));
    SEV_CUDA(cudaMemsetAsync(ctr, 0, sizeof(int), hd->stream));
    // a width that is no multiple of 4 has columns that 16-byte loads cannot serve
    auto kern = sizeof(T) == 4 && b % 4 == 0 ? band_chase_kernel<T, sizeof(T) == 4> : band_chase_kernel<T, false>;
    SEV_CUDA(allow_smem(hd, (const void *)kern));
    int per_sm = 0;
    SEV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem));
    if (per_sm < 1) return SEV_ERR_UNSUPPORTED;
    int grid = hd->sm_count * per_sm;
    // sweep i runs ~3 chases behind sweep i - 1, so about J/3 sweeps (J the
    // chases of the first) progress at once; CTAs beyond that would only poll
    // the progress flags of their predecessors and load the L2 with it
    const int busy = band_num_chases(n, b, h, 0) / 3 + 8;
    if (grid > busy) grid = busy;
    if (grid > nsweeps) grid = nsweeps;
    SEV_LAUNCH(hd, K_BAND_CHASE, kern, grid, kThreads, smem, n, AB, ldab, b, h, nsweeps, progress, ctr, hd->d_err);
    return SEV_OK;
}

template int launch_band_to_band<float>(sev_ctx *, int, float *, int, int, int, void *, size_t);
template int launch_band_to_band<double>(sev_ctx *, int, double *, int, int, int, void *, size_t);
template size_t band_smem_bytes<float>(int, int);
template size_t band_smem_bytes<double>(int, int);

}  // namespace sev
