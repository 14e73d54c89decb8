// band_tri.cu -- the last band reduction, b -> 1 (Algorithm 4.2 with k = b,
// h = 1), for b <= 32, as a sliding-window bulge chase.
//
// With h = 1 every chase (i, j) is ONE Householder reflector H_j on the qr
// rows [o, o + n_r), o = i + (j-1) b, n_r = min(n - o, b).  Step (i, j) here
// does everything that H_j is still owed, and what makes H_{j+1}:
//   D: the diagonal block [o, o + n_r)^2 gets H_j X H_j = X - v w^T - w v^T
//      with p = tau X v, w = p - (tau/2)(p^T v) v;
//   M: the block of rows [o + b, o + 2b) and columns [o, o + b) gets M H_j,
//      then its first column gives the reflector H_{j+1} (the column becomes
//      [beta; 0]) and the other columns get H_{j+1} M.
// Step (i, 0) forms H_1 from column i - 1.  (Algorithm 4.2 applies H_{j+1} to
// those columns in chase j + 1; nothing reads them in between, so doing it
// here gives the same matrix, and M is read and written once per sweep
// instead of twice.)
//
// Order of the steps.  Step (i, j) touches columns [o, o + b) only, and of
// those the last one (o + b - 1) together with row o + 2b - 1 are the only
// places where it meets step (i - 1, j + 1), whose rows and columns start at
// o + b - 1.  Step (i - 1, j + 2) starts at column o + 2b - 1.  So (i, j)
// needs (i - 1, j + 1) complete and runs beside (i - 1, j + 2): sweep i
// trails sweep i - 1 by TWO steps, 2 n steps for the whole stage.  (With the
// column of H_{j+1} annihilated in chase j + 1, as printed, chases (i, j) and
// (i - 1, j + 2) share the entry beta and the lag is three.)
//
// What bounds it: the chain of one step -- loads from shared memory, the
// M H_j product, the pair-float sum of squares, the reflector scalars, the
// H_{j+1} M product -- times 2 n; the band itself is read from L2 once per
// group of G sweeps.  So D and M are two warps, every lane of a warp holds
// B^2 / 32 entries (a row or column is spread over 32 / B lanes), the ring
// is a power of two (no divisions in the addresses) and there is one barrier
// per step.  Measured (GB300): 16 -> 1 at
// n = 16384 in FP32 162.5 -> 37.2 ms (lag three, one warp a sweep, two
// barriers a step: 6.8K cycles a step, now ~1.8K), n = 2048 20.2 -> 4.5 ms,
// n = 3001 in FP64 73.3 -> 25.6 ms.
//
// Schedule.  A CTA takes G consecutive sweeps (sweep i0 + g on warps 2g and
// 2g + 1) and steps them together: at step t sweep g performs step t - 2g.
// The band columns the group touches live in a shared-memory ring (2b
// diagonals each): a loader warp brings columns in (16-byte asynchronous
// copies that signal an mbarrier per step, so that polling the previous
// group and copying overlap), and a writer warp writes them back once the
// group's last sweep has passed them (after its step j, columns below
// o + b are final) and publishes j with a release store; the next group's
// loader waits (acquire, capped) for j >= ts + 1 before loading the columns of
// step ts -- the only global synchronisation.  Groups are handed out in order
// by a global counter and each CTA finishes its group before taking another,
// so every awaited group is held by a running CTA.
#include "tri_step.cuh"

namespace sev {

__device__ __forceinline__ void cp_async16(void *dst, const void *src, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ unsigned tri_smem(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void tri_mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tri_smem(bar)), "r"(count) : "memory");
}
// Arrives once all asynchronous copies this thread has issued have landed.
__device__ __forceinline__ void tri_mbar_arrive_copies(uint64_t *bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tri_smem(bar)) : "memory");
}
__device__ __forceinline__ void tri_mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tri_smem(bar)) : "memory");
}
__device__ __forceinline__ bool tri_mbar_test(uint64_t *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(tri_smem(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void named_bar(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Columns the ring holds: the steps in flight span (2G - 1) b columns, the
// loader runs ahead and the writer behind by a few steps more; a power of two.
template <int B, int G>
__host__ __device__ constexpr int tri_ring_cols() {
    int c = 1;
    while (c < (2 * G + 4) * B + 2) c *= 2;
    return c;
}
constexpr int kTriBars = 8;  // mbarriers of the loader's steps

template <typename T, int B, int G>
__global__ void __launch_bounds__((2 * G + 3) * 32, 1)
    band_tri_kernel(int n, T *AB, int ldab, int nsweeps, int ngroups, int *progress, int *group_ctr, int *err,
                    int async_ok) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int LDW = 2 * B, CAP = tri_ring_cols<B, G>(), S = CAP * LDW;
    T *const w = (T *)smem;
    T *const vbuf = w + S;                     // G x 2 x kTriVec
    T *const wbuf = vbuf + 2 * G * kTriVec;    // G x kTriVec
    __shared__ __align__(8) uint64_t avail[kTriBars];
    __shared__ int s_group;
    __shared__ volatile int s_abort, s_done, s_wblo;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0)
        for (int q = 0; q < kTriBars; ++q) tri_mbar_init(&avail[q], 32);
    const long long cap = wait_cap(err);
    int step0 = 0;  // loader steps of the groups this CTA has finished

    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const int g = atomicAdd(group_ctr, 1);
            s_group = g;
            s_abort = 0;
            s_done = 0;
            s_wblo = g * G;  // = i0 - 1
        }
        __syncthreads();
        const int gi = s_group;
        if (gi >= ngroups) break;
        const int i0 = 1 + gi * G;
        const int nact = min(G, nsweeps - i0 + 1);
        const int il = i0 + nact - 1;
        const int Jf = tri_chases(n, B, i0), Jl = tri_chases(n, B, il);
        const int Jprev = gi > 0 ? tri_chases(n, B, i0 - 1) : 0;
        const int tmax = Jl + 2 * (nact - 1);

        if (warp < 2 * G) {
            // ------------------------------------------------------ compute
            const int g = warp >> 1;
            const bool diag = warp & 1;
            const int i = i0 + g;
            const int Ji = g < nact ? tri_chases(n, B, i) : -1;
            T rv[TriLanes<B>::CPL], rtau = T(0);  // the bulge warp's pending reflector
#pragma unroll
            for (int q = 0; q < TriLanes<B>::CPL; ++q) rv[q] = T(0);
            named_bar(1, (2 * G + 1) * 32);
            for (int t = 0; t <= tmax; ++t) {
                const int j = t - 2 * g;
                if (j >= 0 && j <= Ji) {  // (after an abort the steps run on stale data: every access stays in the ring)
                    const int o = i + (j - 1) * B;
                    T *vb = vbuf + (2 * g + (j & 1)) * kTriVec, *vn = vbuf + (2 * g + ((j + 1) & 1)) * kTriVec;
                    T *wb = wbuf + g * kTriVec;
                    // an interior step whose block lies in one piece in the ring
                    const bool plain = o + 2 * B <= n && ((o * LDW) & (S - 1)) + B * LDW <= S;
                    if (diag) {
                        if (j > 0) {
                            if (plain)
                                tri_diag<T, B, S, true, false>(w, n, o, vb, wb);
                            else
                                tri_diag<T, B, S, false, true>(w, n, o, vb, wb);
                        }
                    } else if (j == 0) {
                        tri_first<T, B, S>(w, n, i, vn, rv, rtau);
                    } else if (plain) {
                        tri_bulge<T, B, S, true, false>(w, n, o, rv, rtau, vn);
                    } else {
                        tri_bulge<T, B, S, false, true>(w, n, o, rv, rtau, vn);
                    }
                }
                __syncwarp();
                named_bar(1, (2 * G + 1) * 32);
            }
        } else if (warp == 2 * G) {
            // -------------------------------------------------------- gate
            // takes part in every step barrier: it has waited for the columns
            // of the coming step before it arrives, and tells the writer and
            // the loader which steps are complete
            for (int t = -1; t <= tmax; ++t) {
                if (lane == 0 && t + 1 <= Jf) {
                    const int st = step0 + t + 1;
                    const long long t0 = clock64();
                    while (!tri_mbar_test(&avail[st % kTriBars], (st / kTriBars) & 1) && !s_abort) {
                        if (wait_expired(t0, cap)) {
                            latch_timeout(err);
                            s_abort = 1;
                        }
                    }
                }
                __syncwarp();
                named_bar(1, (2 * G + 1) * 32);
                if (lane == 0) {
                    __threadfence_block();
                    s_done = t + 1;
                }
            }
        } else if (warp == 2 * G + 1) {
            // ------------------------------------------------------- loader
            int c0 = i0 - 1, seen = 0;
            for (int ts = 0; ts <= Jf; ++ts) {
                const int hi = ts >= Jf ? n : min(n, i0 + ts * B);
                int ok = 1;
                if (lane == 0) {
                    // the previous group's last sweep has passed these columns
                    if (gi > 0 && ts + 1 > seen) {
                        seen = wait_flag(&progress[gi - 1], ts + 1 <= Jprev ? ts + 1 : kTriInf, cap, err,
                                         [&] { return any_gave_up(err) || s_abort; });
                        ok = seen >= 0;
                    }
                    const long long t0 = clock64();
                    // ring space, and the mbarrier's previous phase consumed
                    while (ok && (s_wblo < hi - CAP || s_done < ts - kTriBars + 1)) {
                        if (s_abort) ok = 0;
                        if (wait_expired(t0, cap)) {
                            latch_timeout(err);
                            ok = 0;
                        }
                    }
                    if (!ok) s_abort = 1;
                    __threadfence_block();
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                uint64_t *bar = &avail[(step0 + ts) % kTriBars];
                constexpr int EPC = 16 / (int)sizeof(T);               // elements per 16-byte chunk
                constexpr int CH = LDW / EPC > 0 ? LDW / EPC : 1;      // chunks per column
                if (async_ok && hi - c0 == B && hi + LDW <= n) {
                    // a full step away from the matrix end: no bounds, all copies at once
                    const T *src = AB + (size_t)c0 * ldab;
                    const int ring = c0 * LDW;
#pragma unroll
                    for (int k = 0; k < (B * CH + 31) / 32; ++k) {
                        const int q = lane + 32 * k;
                        if (B * CH % 32 == 0 || q < B * CH)
                            cp_async16(w + ((ring + q * EPC) & (S - 1)), src + (size_t)(q / CH) * ldab + (q % CH) * EPC, 16);
                    }
                    tri_mbar_arrive_copies(bar);
                } else if (async_ok) {
                    // 16-byte copies, zero-filled past the matrix end
                    for (int q = lane; q < (hi - c0) * CH; q += 32) {
                        const int c = c0 + q / CH, d0 = (q % CH) * EPC;
                        int valid = n - c - d0;
                        valid = valid < 0 ? 0 : (valid > EPC ? EPC : valid);
                        const T *src = valid > 0 ? AB + d0 + (size_t)c * ldab : AB;
                        cp_async16(w + ((c * LDW + d0) & (S - 1)), src, valid * (int)sizeof(T));
                    }
                    tri_mbar_arrive_copies(bar);
                } else {
                    batched_copy<T, 16>(
                        (hi - c0) * LDW, lane, 32,
                        [&](int k) {
                            const int c = c0 + k / LDW, d = k % LDW;
                            return (c + d < n) ? __ldcg(AB + d + (size_t)c * ldab) : T(0);
                        },
                        [&](int k, T v) { w[((c0 + k / LDW) * LDW + k % LDW) & (S - 1)] = v; });
                    tri_mbar_arrive(bar);
                }
                c0 = max(c0, hi);
            }
            if (async_ok) cp_async_wait_all();  // no copy in flight when the CTA moves on or leaves
        } else {
            // ------------------------------------------------------- writer
            int lo = i0 - 1, written = 0;
            while (written <= tmax) {
                int td = 0;
                if (lane == 0) {
                    const long long t0 = clock64();
                    while ((td = s_done) <= written && !s_abort) {
                        if (wait_expired(t0, cap)) {
                            latch_timeout(err);
                            s_abort = 1;
                        }
                    }
                    __threadfence_block();
                }
                td = __shfl_sync(0xffffffffu, td, 0);
                if (__shfl_sync(0xffffffffu, s_abort, 0)) break;
                written = td;  // steps 0 .. td - 1 are complete
                const int jl = td - 1 - 2 * (nact - 1);
                if (jl < 1) continue;
                const bool done = jl >= Jl;
                const int fin = done ? n : min(n, il + jl * B);
                constexpr int EPC = 16 / (int)sizeof(T), CH = LDW / EPC > 0 ? LDW / EPC : 1;
                // whole steps (several, if compute has run ahead) away from the matrix end
                for (; async_ok && lo + B <= fin && lo + B + LDW <= n; lo += B) {
                    T *dst = AB + (size_t)lo * ldab;
                    const int ring = lo * LDW;
                    constexpr int K = (B * CH + 31) / 32;
                    uint4 v[K];
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        v[k] = *reinterpret_cast<const uint4 *>(w + ((ring + (lane + 32 * k) * EPC) & (S - 1)));
#pragma unroll
                    for (int k = 0; k < K; ++k) {
                        const int q = lane + 32 * k;
                        if (B * CH % 32 == 0 || q < B * CH)
                            *reinterpret_cast<uint4 *>(dst + (size_t)(q / CH) * ldab + (q % CH) * EPC) = v[k];
                    }
                }
                for (int idx = lane; idx < (fin - lo) * LDW; idx += 32) {
                    const int c = lo + idx / LDW, d = idx % LDW;
                    if (c + d < n) AB[d + (size_t)c * ldab] = w[(c * LDW + d) & (S - 1)];
                }
                if (fin > lo) lo = fin;
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    s_wblo = lo;
                    // the release store orders the warp's write-back before the flag
                    st_release(&progress[gi], done ? kTriInf : jl);
                }
            }
        }
        __syncthreads();
        if (s_abort) return;
        step0 += Jf + 1;
    }
}

template <typename T, int B, int G>
static int launch_tri(sev_ctx *h, int n, T *AB, int ldab, int *progress, int *ctr, int nsweeps) {
    const int ngroups = (nsweeps + G - 1) / G;
    const size_t smem = sizeof(T) * ((size_t)tri_ring_cols<B, G>() * 2 * B + 3 * G * kTriVec);
    if (smem > h->smem_optin) return SEV_ERR_UNSUPPORTED;
    SEV_CUDA(cudaMemsetAsync(progress, 0, sizeof(int) * (size_t)ngroups, h->stream));
    SEV_CUDA(cudaMemsetAsync(ctr, 0, sizeof(int), h->stream));
    auto kern = band_tri_kernel<T, B, G>;
    SEV_CUDA(allow_smem(h, (const void *)kern));
    int per_sm = 0;
    SEV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, (2 * G + 3) * 32, smem));
    if (per_sm < 1) return SEV_ERR_UNSUPPORTED;
    // groups start ~2G steps apart and each runs ~J + 2G steps, so about
    // J / (2G) of them are busy at once; more CTAs would only poll
    const int J1 = tri_chases(n, B, 1);
    int grid = h->sm_count * per_sm;
    const int busy = J1 / (2 * G) + 16;
    if (grid > busy) grid = busy;
    if (grid > ngroups) grid = ngroups;
    // 16-byte asynchronous copies need a 16-byte-aligned band and column stride
    const int async_ok =
        ((uintptr_t)AB % 16 == 0) && ((size_t)ldab * sizeof(T)) % 16 == 0 && (2 * B * sizeof(T)) % 16 == 0;
    SEV_LAUNCH(h, K_BAND_TRI, kern, grid, (2 * G + 3) * 32, smem, n, AB, ldab, nsweeps, ngroups, progress, ctr,
               h->d_err, async_ok);
    return SEV_OK;
}

// Sweeps per CTA (two warps each): more of them spread the hand-over between
// groups (~5 us) over more sweeps, fewer leave each scheduler (and, in FP64,
// the one FP64 pipe of each scheduler) fewer warps to serve.  16 -> 1 at
// n = 16384, FP32: 4 sweeps 44.4 ms, 6 37.2, 8 38.5; n = 3001, FP64: 2 sweeps
// 26.4 ms, 3 25.6, 4 28.1.
#ifndef SEV_TRI_G_F32
#define SEV_TRI_G_F32 6
#endif
#ifndef SEV_TRI_G_F64
#define SEV_TRI_G_F64 3
#endif
#ifndef SEV_TRI_G32
#define SEV_TRI_G32 4
#endif

int band_tri_supported(int b, int elem) { return b == 2 || b == 4 || b == 8 || b == 16 || (b == 32 && elem == 4); }

size_t band_tri_workspace(int n) {
    Carver c(nullptr);
    c.take<int>((size_t)n + 1);
    c.take<int>(1);
    return c.bytes();
}

template <typename T>
int launch_band_tri(sev_ctx *h, int n, T *AB, int ldab, int b, void *ws, size_t ws_bytes) {
    const int nsweeps = n >= 3 ? n - 2 : 0;
    if (nsweeps <= 0) return SEV_OK;
    if (ws_bytes < band_tri_workspace(n)) return SEV_ERR_WORKSPACE;
    Carver c(ws);
    int *progress = c.take<int>((size_t)n + 1);
    int *ctr = c.take<int>(1);
    constexpr int G = sizeof(T) == 4 ? SEV_TRI_G_F32 : SEV_TRI_G_F64;
    switch (b) {
        case 2: return launch_tri<T, 2, G>(h, n, AB, ldab, progress, ctr, nsweeps);
        case 4: return launch_tri<T, 4, G>(h, n, AB, ldab, progress, ctr, nsweeps);
        case 8: return launch_tri<T, 8, G>(h, n, AB, ldab, progress, ctr, nsweeps);
        case 16: return launch_tri<T, 16, G>(h, n, AB, ldab, progress, ctr, nsweeps);
        case 32:
            if constexpr (sizeof(T) == 4) return launch_tri<T, 32, SEV_TRI_G32>(h, n, AB, ldab, progress, ctr, nsweeps);
            return SEV_ERR_UNSUPPORTED;
        default: return SEV_ERR_UNSUPPORTED;
    }
}

template int launch_band_tri<float>(sev_ctx *, int, float *, int, int, void *, size_t);
template int launch_band_tri<double>(sev_ctx *, int, double *, int, int, void *, size_t);

}  // namespace sev
