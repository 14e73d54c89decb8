// update.cu -- the two-sided trailing update of the full-to-band reduction
// (Eq. 4.1 as used in Algorithm 4.1) and the full-to-band driver.
//
// Per panel, with U (N x b) and T (b x b) from panel.cu and A22 the lower-
// stored trailing matrix:
//   Y  = A22 U                       (symm: reads A22 symmetrically)
//   M  = U^T Y,  Zh = T^T M T / 2    (X = Y T = W T in the algorithm's notation:
//   V  = U Zh - Y T                   Zh = T^T U^T X / 2, V = U Zh - X, the V_1
//                                     line of Algorithm 4.1)
//   A22 <- A22 + U V^T + V U^T       (syr2k, lower tiles only)
//
// The FP64 form runs all of it on SIMT tiles (64 x 64 outputs, 4 x 4 per
// thread, DFMA); the mixed form's symm runs on larger FP32 tiles
// (symm_f32_kernel) and its syr2k on the tensor cores (update_tc.cu).
#include <cuda_bf16.h>

#include "common.cuh"

namespace sev {

template <typename T>
int panel_factor(sev_ctx *h, int N, int b, T *P, int lda, T *U, T *Tm, void *ws);
template <typename T>
size_t panel_workspace(sev_ctx *h, int n, int b);
template <typename T>
int tc_update_supported(sev_ctx *h, int N, int b);
template <typename T>
void tc_panels(int N, int b, void *ws, __nv_bfloat16 **P, __nv_bfloat16 **Q, int *K6p);
template <typename T>
int tc_syr2k(sev_ctx *h, int N, int b, T *A22, int lda, void *ws);
template <typename T>
size_t tc_workspace(int n, int b);
template <typename T>
int tc_symm_supported(sev_ctx *h, int N, int b, const T *A22, int lda);
template <typename T>
int tc_symm(sev_ctx *h, int N, int b, const T *A22, int lda, const T *U, T *ypart, int max_splits, int *splits,
            void *ws);

constexpr int BM = 64, BK = 16, PADT = 4;

// A 64 x TN output tile of 256 threads, rows tx + 16 i, columns ty + 16 j
// (TN = 32 for bands up to 32: a 64-wide tile would do twice the work).
template <typename T, int TN>
struct Tile {
    T As[BK][BM + PADT];
    T Bs[BK][TN + PADT];
};

template <typename T, int TN>
__device__ __forceinline__ void tile_mma(const Tile<T, TN> &t, T (&acc)[4][TN / 16]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int k = 0; k < BK; ++k) {
        T a[4], bb[TN / 16];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = t.As[k][tx + 16 * i];
#pragma unroll
        for (int j = 0; j < TN / 16; ++j) bb[j] = t.Bs[k][ty + 16 * j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TN / 16; ++j) acc[i][j] += a[i] * bb[j];
    }
}

// One thread's share of a slab, loaded into registers: element (m, k) of the
// A slab and (k, n) of the B slab of the step at k0.
template <typename T>
__device__ __forceinline__ void symm_slab_a(T (&ra)[4], const T *A, int lda, int N, int m0, int k0, int kend) {
    const bool below = k0 + BK <= m0, above = k0 >= m0 + BM;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int idx = threadIdx.x + 256 * r;
        // below and on the diagonal block: down the columns; above it A(m, k) = A(k, m): along k
        const int m = above ? idx >> 4 : idx & 63, k = above ? idx & 15 : idx >> 6;
        const int gm = m0 + m, gk = k0 + k;
        T v = T(0);
        if (gm < N && gk < kend)
            v = (below || (!above && gm >= gk)) ? A[(size_t)gm + (size_t)gk * lda] : A[(size_t)gk + (size_t)gm * lda];
        ra[r] = v;
    }
}

// Partial products of Y = A22 U (A22 symmetric N x N, its lower triangle
// stored): CTA (x, y, z) sums rows [z kchunk, (z + 1) kchunk) of the K range for
// the 64 x TN tile (x, y); the splits are summed in order by uty_kernel.
// What bounds it: in FP64 the FP64 pipes (2 FMAs per cycle and SM), so the
// host picks the number of splits that fills whole waves of CTAs; the next
// slab's loads are in flight while this one is multiplied.  n = 3001, b = 32,
// FP64: 148.7 ms per reduction with 64-wide tiles on one wave of 47 CTAs,
// now 16.9 ms (floor 15.0 ms at
// 1.2 TFLOP/s).
template <typename T, int TN>
__global__ void __launch_bounds__(256) symm_kernel(int N, int b, const T *__restrict__ A, int lda,
                                                   const T *__restrict__ U, int ldu, int kchunk,
                                                   T *__restrict__ Yout, size_t split_stride) {
    __shared__ Tile<T, TN> t;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * TN;
    const int kbeg = blockIdx.z * kchunk, kend = min(N, kbeg + kchunk);
    T *Y = Yout + (size_t)blockIdx.z * split_stride;
    T acc[4][TN / 16] = {};
    T ra[4], rb[TN / 16];
    auto slab_b = [&](int k0) {
#pragma unroll
        for (int r = 0; r < TN / 16; ++r) {
            const int idx = threadIdx.x + 256 * r, k = idx & 15, n = idx >> 4;
            rb[r] = (k0 + k < kend && n0 + n < b) ? U[(size_t)(k0 + k) + (size_t)(n0 + n) * ldu] : T(0);
        }
    };
    if (kbeg < kend) {
        symm_slab_a<T>(ra, A, lda, N, m0, kbeg, kend);
        slab_b(kbeg);
    }
    for (int k0 = kbeg; k0 < kend; k0 += BK) {
        const bool above = k0 >= m0 + BM;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int idx = threadIdx.x + 256 * r;
            t.As[above ? idx & 15 : idx >> 6][above ? idx >> 4 : idx & 63] = ra[r];
        }
#pragma unroll
        for (int r = 0; r < TN / 16; ++r) {
            const int idx = threadIdx.x + 256 * r;
            t.Bs[idx & 15][idx >> 4] = rb[r];
        }
        __syncthreads();
        if (k0 + BK < kend) {
            symm_slab_a<T>(ra, A, lda, N, m0, k0 + BK, kend);
            slab_b(k0 + BK);
        }
        tile_mma(t, acc);
        __syncthreads();
    }
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < TN / 16; ++j) {
            const int m = m0 + tx + 16 * i, n = n0 + ty + 16 * j;
            if (m < N && n < b) Y[(size_t)m + (size_t)n * N] = acc[i][j];
        }
}

// Y = A22 U for FP32 data: 128 x 64 output tiles, 8 x 4 outputs per thread,
// K in steps of 16 through double-buffered shared memory (the next step's
// loads in registers while this one is multiplied), float4 loads of A22 in
// whichever orientation is contiguous (columns below the diagonal block,
// rows -- A(m, k) = A(k, m) -- above it, transposed into shared memory),
// and the K range split over blockIdx.z with per-split partial tiles
// (summed in a fixed order by uty_kernel) so that every SM has work.
// Needs lda % 4 == 0 and a 16-byte-aligned A22.
constexpr int SBM = 128, SBN = 64, SBK = 16;

struct SymmSmem {
    float As[2][SBK][SBM + 4];
    float Bs[2][SBK][SBN + 4];
};

__device__ __forceinline__ void symm_load_a(float4 (&ra)[2], float (&rs)[8], bool &vec, int &mode, const float *A,
                                            int lda, int N, int m0, int k0) {
    const int tid = threadIdx.x;
    const bool inside = m0 + SBM <= N && k0 + SBK <= N;
    if (inside && k0 + SBK <= m0) {  // strictly below: columns are contiguous
        mode = 0;
        vec = true;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int idx = tid + r * 256, k = idx >> 5, mq = idx & 31;
            ra[r] = *reinterpret_cast<const float4 *>(A + (size_t)(m0 + 4 * mq) + (size_t)(k0 + k) * lda);
        }
    } else if (inside && k0 >= m0 + SBM) {  // strictly above: A(m, k) = A(k, m), rows contiguous
        mode = 1;
        vec = true;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int idx = tid + r * 256, m = idx >> 2, kq = idx & 3;
            ra[r] = *reinterpret_cast<const float4 *>(A + (size_t)(k0 + 4 * kq) + (size_t)(m0 + m) * lda);
        }
    } else {  // crosses the diagonal block or the matrix edge: element by element
        mode = 2;
        vec = false;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int idx = tid + r * 256, m = idx & (SBM - 1), k = idx >> 7;
            const int gm = m0 + m, gk = k0 + k;
            float v = 0.f;
            if (gm < N && gk < N) v = gm >= gk ? A[(size_t)gm + (size_t)gk * lda] : A[(size_t)gk + (size_t)gm * lda];
            rs[r] = v;
        }
    }
}

__device__ __forceinline__ void symm_store_a(SymmSmem &S, int buf, const float4 (&ra)[2], const float (&rs)[8],
                                             int mode) {
    const int tid = threadIdx.x;
    if (mode == 0) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int idx = tid + r * 256, k = idx >> 5, mq = idx & 31;
            *reinterpret_cast<float4 *>(&S.As[buf][k][4 * mq]) = ra[r];
        }
    } else if (mode == 1) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int idx = tid + r * 256, m = idx >> 2, kq = idx & 3;
            S.As[buf][4 * kq + 0][m] = ra[r].x;
            S.As[buf][4 * kq + 1][m] = ra[r].y;
            S.As[buf][4 * kq + 2][m] = ra[r].z;
            S.As[buf][4 * kq + 3][m] = ra[r].w;
        }
    } else {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int idx = tid + r * 256, m = idx & (SBM - 1), k = idx >> 7;
            S.As[buf][k][m] = rs[r];
        }
    }
}

__device__ __forceinline__ void symm_load_b(float (&rb)[4], const float *U, int ldu, int N, int b, int k0, int n0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int idx = threadIdx.x + r * 256, k = idx & (SBK - 1), n = idx >> 4;
        const int gk = k0 + k, gn = n0 + n;
        rb[r] = (gk < N && gn < b) ? U[(size_t)gk + (size_t)gn * ldu] : 0.f;
    }
}

__device__ __forceinline__ void symm_store_b(SymmSmem &S, int buf, const float (&rb)[4]) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int idx = threadIdx.x + r * 256, k = idx & (SBK - 1), n = idx >> 4;
        S.Bs[buf][k][n] = rb[r];
    }
}

__global__ void __launch_bounds__(256) symm_f32_kernel(int N, int b, const float *__restrict__ A, int lda,
                                                       const float *__restrict__ U, int ldu, int kchunk,
                                                       float *__restrict__ Yout, int ldy, size_t split_stride) {
    __shared__ __align__(16) SymmSmem S;
    const int m0 = blockIdx.x * SBM, n0 = blockIdx.y * SBN;
    const int kbeg = blockIdx.z * kchunk, kend = min(N, kbeg + kchunk);
    float *Y = Yout + (size_t)blockIdx.z * split_stride;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    float4 ra[2];
    float rs[8], rb[4];
    bool vec;
    int mode;
    int buf = 0;
    if (kbeg < kend) {
        symm_load_a(ra, rs, vec, mode, A, lda, N, m0, kbeg);
        symm_load_b(rb, U, ldu, N, b, kbeg, n0);
        symm_store_a(S, 0, ra, rs, mode);
        symm_store_b(S, 0, rb);
    }
    __syncthreads();
    for (int k0 = kbeg; k0 < kend; k0 += SBK) {
        const bool more = k0 + SBK < kend;
        if (more) {
            symm_load_a(ra, rs, vec, mode, A, lda, N, m0, k0 + SBK);
            symm_load_b(rb, U, ldu, N, b, k0 + SBK, n0);
        }
        // rows beyond kend in this step are zero-padded only at the matrix
        // edge; split boundaries are multiples of SBK
#pragma unroll
        for (int k = 0; k < SBK; ++k) {
            const float4 a0 = *reinterpret_cast<const float4 *>(&S.As[buf][k][4 * tx]);
            const float4 a1 = *reinterpret_cast<const float4 *>(&S.As[buf][k][64 + 4 * tx]);
            const float4 bv = *reinterpret_cast<const float4 *>(&S.Bs[buf][k][4 * ty]);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float bw[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bw[j], acc[i][j]);
        }
        if (more) {
            symm_store_a(S, buf ^ 1, ra, rs, mode);
            symm_store_b(S, buf ^ 1, rb);
        }
        __syncthreads();
        buf ^= 1;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int m = m0 + (i < 4 ? 4 * tx + i : 64 + 4 * tx + i - 4);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + 4 * ty + j;
            if (m < N && n < b) Y[(size_t)m + (size_t)n * ldy] = acc[i][j];
        }
    }
}

// M_p = U_p^T Y_p (b x b) for row chunk p, with Y = the sum of the symmetric
// product's split partials in split order (written back when there is more
// than one; the tiles of a chunk that share Y columns write them once).
template <typename T, int TN>
__global__ void __launch_bounds__(256)
    uty_kernel(int N, int b, int chunk, const T *__restrict__ U, int splits, const T *__restrict__ ypart,
               size_t split_stride, T *__restrict__ Y, T *__restrict__ part) {
    constexpr int TM = TN, KB = 32;  // TM x TN outputs, KB rows at a time
    __shared__ T As[KB][TM + 1], Bs[KB][TN + 1];
    const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN, p = blockIdx.z;
    const int kbeg = p * chunk, kend = min(N, kbeg + chunk);
    constexpr int PER = TN / 16;
    T acc[PER][PER] = {};
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    constexpr int L = KB * TN / 256;  // elements per thread and operand
    for (int k0 = kbeg; k0 < kend; k0 += KB) {
        T ru[L], ry[L];
        const int k = threadIdx.x & 31, gk = k0 + k;
#pragma unroll
        for (int r = 0; r < L; ++r) {
            const int c = (threadIdx.x >> 5) + 8 * r;
            ru[r] = (gk < kend && m0 + c < b) ? U[(size_t)gk + (size_t)(m0 + c) * N] : T(0);
            ry[r] = (gk < kend && n0 + c < b) ? ypart[(size_t)gk + (size_t)(n0 + c) * N] : T(0);
        }
        for (int z = 1; z < splits; ++z)
#pragma unroll
            for (int r = 0; r < L; ++r) {
                const int c = (threadIdx.x >> 5) + 8 * r;
                if (gk < kend && n0 + c < b) ry[r] += ypart[(size_t)z * split_stride + gk + (size_t)(n0 + c) * N];
            }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < L; ++r) {
            const int c = (threadIdx.x >> 5) + 8 * r;
            As[k][c] = ru[r];
            Bs[k][c] = ry[r];
            if (splits > 1 && m0 == 0 && gk < kend && n0 + c < b) Y[(size_t)gk + (size_t)(n0 + c) * N] = ry[r];
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < KB; ++kk) {
            T a[PER], bb[PER];
#pragma unroll
            for (int i = 0; i < PER; ++i) a[i] = As[kk][tx + 16 * i];
#pragma unroll
            for (int j = 0; j < PER; ++j) bb[j] = Bs[kk][ty + 16 * j];
#pragma unroll
            for (int i = 0; i < PER; ++i)
#pragma unroll
                for (int j = 0; j < PER; ++j) acc[i][j] += a[i] * bb[j];
        }
    }
    T *P = part + (size_t)p * b * b;
#pragma unroll
    for (int i = 0; i < PER; ++i)
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int m = m0 + tx + 16 * i, n = n0 + ty + 16 * j;
            if (m < b && n < b) P[m + (size_t)n * b] = acc[i][j];
        }
}

// M = sum_p M_p, entry by entry, the partials in a fixed order (deterministic).
template <typename T>
__global__ void __launch_bounds__(256) uty_sum_kernel(int bb, int nparts, const T *__restrict__ part, T *__restrict__ M) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= bb) return;
    T s[4] = {};
    int p = 0;
    for (; p + 4 <= nparts; p += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) s[u] += part[(size_t)(p + u) * bb + idx];
    for (; p < nparts; ++p) s[0] += part[(size_t)p * bb + idx];
    M[idx] = (s[0] + s[1]) + (s[2] + s[3]);
}

// Zh = T^T M T / 2 (b x b, T upper triangular), NC columns per CTA: R = M T(:, c)
// in shared memory, then T^T R; a warp's lanes share a dot product.
template <typename T, int NC>
__global__ void __launch_bounds__(256) uty_zh_kernel(int b, const T *__restrict__ M, const T *__restrict__ Tm,
                                                     T *__restrict__ Zh) {
    extern __shared__ __align__(16) unsigned char smem[];
    T *Ts = (T *)smem, *Rs = Ts + (size_t)b * NC;  // T's columns of this CTA; R (b x NC)
    const int c0 = blockIdx.x * NC, nc = min(NC, b - c0);
    for (int idx = threadIdx.x; idx < b * nc; idx += 256) Ts[idx] = Tm[(size_t)c0 * b + idx];
    __syncthreads();
    // R(a, c) = sum_{q <= c} M(a, q) T(q, c): thread per entry, M read along a
    for (int idx = threadIdx.x; idx < b * nc; idx += 256) {
        const int a = idx % b, c = idx / b;
        T s0 = 0, s1 = 0;
        int q = 0;
        for (; q + 1 <= c0 + c; q += 2) {
            s0 += M[a + (size_t)q * b] * Ts[q + (size_t)c * b];
            s1 += M[a + (size_t)(q + 1) * b] * Ts[q + 1 + (size_t)c * b];
        }
        if (q <= c0 + c) s0 += M[a + (size_t)q * b] * Ts[q + (size_t)c * b];
        Rs[idx] = s0 + s1;
    }
    __syncthreads();
    // Zh(a, c) = sum_{q <= a} T(q, a) R(q, c) / 2: a warp per entry row a, lanes over q
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int a = warp; a < b; a += 8) {
        T s[NC] = {};
        for (int q = lane; q <= a; q += 32) {
            const T tq = Tm[q + (size_t)a * b];
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (c < nc) s[c] += tq * Rs[q + (size_t)c * b];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < NC; ++c) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (lane == c && c < nc) Zh[a + (size_t)(c0 + c) * b] = T(0.5) * s[c];
    }
}

// V = U Zh - Y T for the 64 x TN tile (x, y).  With P and Q (mixed form) V
// itself is not stored: the tile's U and V go straight into the BF16 operand
// panels of the tensor-core update (see tc_syr2k), rows of 64 at a time.
template <typename T, int TN>
__global__ void __launch_bounds__(256)
    vform_kernel(int N, int b, const T *__restrict__ U, const T *__restrict__ Y, const T *__restrict__ Zh,
                 const T *__restrict__ Tm, T *__restrict__ V, int K6p, __nv_bfloat16 *__restrict__ P,
                 __nv_bfloat16 *__restrict__ Q) {
    __shared__ Tile<T, TN> t;
    __shared__ T Vs[BM][TN + 1];
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * TN;
    T acc[4][TN / 16] = {};
    // K = 2b: U against Zh, then Y against -T
    for (int h = 0; h < 2; ++h) {
        const T *A = h ? Y : U, *B = h ? Tm : Zh;
        const int klen = h ? min(b, n0 + TN) : b;  // T is upper triangular
        for (int k0 = 0; k0 < klen; k0 += BK) {
            T ra[4], rb[TN / 16];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int idx = threadIdx.x + 256 * r, m = idx & 63, k = idx >> 6;
                ra[r] = (m0 + m < N && k0 + k < b) ? A[(size_t)(m0 + m) + (size_t)(k0 + k) * N] : T(0);
            }
#pragma unroll
            for (int r = 0; r < TN / 16; ++r) {
                const int idx = threadIdx.x + 256 * r, k = idx & 15, n = idx >> 4;
                const T v = (k0 + k < b && n0 + n < b) ? B[(k0 + k) + (size_t)(n0 + n) * b] : T(0);
                rb[r] = h ? -v : v;
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int idx = threadIdx.x + 256 * r;
                t.As[idx >> 6][idx & 63] = ra[r];
            }
#pragma unroll
            for (int r = 0; r < TN / 16; ++r) {
                const int idx = threadIdx.x + 256 * r;
                t.Bs[idx & 15][idx >> 4] = rb[r];
            }
            __syncthreads();
            tile_mma(t, acc);
        }
    }
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    if (P == nullptr) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TN / 16; ++j) {
                const int m = m0 + tx + 16 * i, n = n0 + ty + 16 * j;
                if (m < N && n < b) V[(size_t)m + (size_t)n * N] = acc[i][j];
            }
        return;
    }
    if constexpr (sizeof(T) == 4) {
        // V's tile to rows, then U's: a row's columns are contiguous in P and Q
        float vv[BM * TN / 256];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TN / 16; ++j) Vs[tx + 16 * i][ty + 16 * j] = acc[i][j];
        __syncthreads();
        const int c = threadIdx.x % TN, r0 = threadIdx.x / TN;
        constexpr int RS = 256 / TN;
#pragma unroll
        for (int q = 0; q < BM / RS; ++q) vv[q] = Vs[r0 + RS * q][c];
        __syncthreads();
        for (int idx = threadIdx.x; idx < BM * TN; idx += 256) {
            const int m = idx & 63, n = idx >> 6;
            Vs[m][n] = (m0 + m < N && n0 + n < b) ? U[(size_t)(m0 + m) + (size_t)(n0 + n) * N] : T(0);
        }
        __syncthreads();
        const int gc = n0 + c;
#pragma unroll
        for (int q = 0; q < BM / RS; ++q) {
            const int r = r0 + RS * q, gr = m0 + r;
            if (gr >= N) continue;
            if (gc < b) {
                const float u = Vs[r][c], v = vv[q];
                const __nv_bfloat16 uh = __float2bfloat16_rn(u), vh = __float2bfloat16_rn(v);
                const __nv_bfloat16 ul = __float2bfloat16_rn(u - __bfloat162float(uh));
                const __nv_bfloat16 vl = __float2bfloat16_rn(v - __bfloat162float(vh));
                __nv_bfloat16 *p = P + (size_t)gr * K6p + gc, *w = Q + (size_t)gr * K6p + gc;
                p[0] = uh, w[0] = vh;
                p[b] = vh, w[b] = uh;
                p[2 * b] = uh, w[2 * b] = vl;
                p[3 * b] = vh, w[3 * b] = ul;
                p[4 * b] = ul, w[4 * b] = vh;
                p[5 * b] = vl, w[5 * b] = uh;
            }
            // the padding of K to whole 64-wide boxes
            if (blockIdx.y == 0)
                for (int k = 6 * b + c; k < K6p; k += TN) {
                    P[(size_t)gr * K6p + k] = __float2bfloat16_rn(0.f);
                    Q[(size_t)gr * K6p + k] = __float2bfloat16_rn(0.f);
                }
        }
    }
}

// A22 += U V^T + V U^T on the lower tiles (tile (I, J), I >= J).
template <typename T>
__global__ void __launch_bounds__(256) syr2k_kernel(int N, int b, T *__restrict__ A, int lda, const T *__restrict__ U,
                                                    int ldu, const T *__restrict__ V, int ldv) {
    constexpr int BN = 64;
    __shared__ Tile<T, BN> t;
    const long x = blockIdx.x;
    int I = (int)((sqrt(8.0 * (double)x + 1.0) - 1.0) * 0.5);
    while ((long)(I + 1) * (I + 2) / 2 <= x) ++I;
    while ((long)I * (I + 1) / 2 > x) --I;
    const int J = (int)(x - (long)I * (I + 1) / 2);
    const int m0 = I * BM, n0 = J * BN;
    T acc[4][4] = {};
    const int K2 = 2 * b;
    for (int k0 = 0; k0 < K2; k0 += BK) {
        for (int idx = threadIdx.x; idx < BM * BK; idx += blockDim.x) {
            const int m = idx % BM, k = idx / BM;
            const int gm = m0 + m, gk = k0 + k;
            T v = 0;
            if (gm < N && gk < K2) v = gk < b ? U[(size_t)gm + (size_t)gk * ldu] : V[(size_t)gm + (size_t)(gk - b) * ldv];
            t.As[k][m] = v;
        }
        for (int idx = threadIdx.x; idx < BK * BN; idx += blockDim.x) {
            const int n = idx % BN, k = idx / BN;
            const int gk = k0 + k, gn = n0 + n;
            T v = 0;
            if (gn < N && gk < K2) v = gk < b ? V[(size_t)gn + (size_t)gk * ldv] : U[(size_t)gn + (size_t)(gk - b) * ldu];
            t.Bs[k][n] = v;
        }
        __syncthreads();
        tile_mma(t, acc);
        __syncthreads();
    }
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int m = m0 + tx + 16 * i, n = n0 + ty + 16 * j;
            if (m < N && n < N && m >= n) A[(size_t)m + (size_t)n * lda] += acc[i][j];
        }
}

// --------------------------------------------------------------- driver
template <typename T>
struct F2BBuffers {
    T *U, *Y, *V, *Tm, *Zm, *part, *ypart;
    unsigned long long *comm;
    size_t comm_words;
    void *panel_ws, *tc_ws;
};

// Partial products of Y kept at most: FP64 at moderate orders takes up to 16
// splits (whole waves of CTAs), else 8.
template <typename T>
static int symm_max_splits(int n) {
    return sizeof(T) == 8 && n <= 8192 ? 16 : 8;
}

// Row chunks of U^T Y: 64 rows or more each, at most 128.
static int uty_chunk(int N) {
    const int c = ((N + 127) / 128 + 31) / 32 * 32;
    return c < 64 ? 64 : c;
}
static int uty_parts(int N) { return (N + uty_chunk(N) - 1) / uty_chunk(N); }

template <typename T>
static void carve_f2b(Carver &c, F2BBuffers<T> &B, sev_ctx *h, int n, int b, bool tc) {
    B.U = c.take<T>((size_t)n * b);
    B.Y = c.take<T>((size_t)n * b);
    B.V = c.take<T>((size_t)n * b);
    B.Tm = c.take<T>((size_t)b * b);
    B.Zm = c.take<T>((size_t)b * b);
    B.part = c.take<T>((size_t)129 * b * b);  // the chunks' partial products, then their sum
    B.ypart = c.take<T>((size_t)symm_max_splits<T>(n) * n * b);
    B.tc_ws = tc ? (void *)c.take<char>(tc_workspace<T>(n, b)) : nullptr;
    B.comm_words = panel_coop_words<T>(h, b);
    B.comm = c.take<unsigned long long>(B.comm_words);
    B.panel_ws = c.take<char>(panel_workspace<T>(h, n, b));
}

template <typename T>
size_t full_to_band_workspace(sev_ctx *h, int n, int b) {
    Carver c(nullptr);
    F2BBuffers<T> B;
    carve_f2b<T>(c, B, h, n, b, true);
    return c.bytes();
}

// An FP32 matrix without 16-byte aligned columns (an odd order in contiguous
// storage: three orders of four) is multiplied in FP32 by SIMT tiles -- the
// tensor-core product needs TMA, and its BF16x3 splits are less exact, so such
// matrices do not change over to it.  The SIMT kernel with 16-byte loads and a
// split K range wants aligned columns too, so the reduction runs on an aligned
// copy of the lower triangle, made by the pass that looks for NaN and Inf:
// n = 2731, b = 64 7.1 -> 1.6 ms of products per reduction for ~10 us of
// copying.  Below ~512 rows it makes no difference.
template <typename T>
size_t full_to_band_copy_bytes(sev_ctx *h, int n, int b, const T *A, int lda) {
    if (sizeof(T) != 4 || n - b < 512 || b >= n - 1) return 0;
    if (lda % 4 == 0 && ((uintptr_t)A & 15) == 0) return 0;
    return (sizeof(T) * (size_t)copy_ld(n) * n + 255) & ~(size_t)255;
}

template <typename T>
int launch_full_to_band(sev_ctx *h, int n, T *A, int lda, int b, T *AB, int ldab, void *ws, size_t ws_bytes,
                        bool fp32_product) {
    if (n <= 0) return SEV_OK;
    if (ws_bytes < full_to_band_workspace<T>(h, n, b)) return SEV_ERR_WORKSPACE;
    Carver c(ws);
    F2BBuffers<T> B;
    carve_f2b<T>(c, B, h, n, b, true);
    bool comm_clear = false;
    for (int k = 0;; ++k) {
        const int c0 = k * b, r0 = c0 + b;
        if (r0 >= n) break;
        const int N = n - r0;
        if (N < 2) break;
        T *P = A + (size_t)r0 + (size_t)c0 * lda;
        T *A22 = A + (size_t)r0 + (size_t)r0 * lda;
        int rc;
        if (panel_coop_supported<T>(h, N, b)) {
            // the panel on all SMs at once; the tree serves panels too tall for
            // the GPU's registers, wider bands and a prescribed leaf size
            if (!comm_clear) {
                SEV_CUDA(cudaMemsetAsync(B.comm, 0, sizeof(unsigned long long) * B.comm_words, h->stream));
                comm_clear = true;
            }
            rc = panel_coop_factor<T>(h, N, b, P, lda, B.U, B.Tm, B.comm, (unsigned)k * (unsigned)(b + 2));
        } else {
            rc = panel_factor<T>(h, N, b, P, lda, B.U, B.Tm, B.panel_ws);
        }
        if (rc) return rc;
        const bool tc = tc_update_supported<T>(h, N, b);
        // partial products of Y = A22 U
        int splits = 1;
        if (!fp32_product && tc_symm_supported<T>(h, N, b, A22, lda)) {
            rc = tc_symm<T>(h, N, b, A22, lda, B.U, B.ypart, symm_max_splits<T>(n), &splits, B.tc_ws);
            if (rc) return rc;
        } else if (sizeof(T) == 4 && lda % 4 == 0 && ((uintptr_t)A22 & 15) == 0) {
            // split K until the grid covers ~2 CTAs per SM
            const int mt = (N + SBM - 1) / SBM, nt = (b + SBN - 1) / SBN;
            while (splits < 8 && mt * nt * splits < 2 * h->sm_count && N / (splits * 2) >= 256) splits *= 2;
            const int kchunk = ((N + splits - 1) / splits + SBK - 1) / SBK * SBK;
            SEV_LAUNCH(h, K_SYMM, symm_f32_kernel, dim3(mt, nt, splits), 256, 0, N, b, (const float *)A22, lda,
                       (const float *)B.U, N, kchunk, (float *)B.ypart, N, (size_t)N * b);
        } else {
            const int tn = b <= 32 ? 32 : 64, mt = (N + BM - 1) / BM, nt = (b + tn - 1) / tn;
            // the number of splits that leaves the last wave of CTAs fullest
            // (one CTA keeps an SM's FP64 pipes busy), each of 64 rows or more
            float best = 0.f;
            for (int z = 1; z <= symm_max_splits<T>(n) && (z == 1 || N / z >= 64); ++z) {
                const float waves = (float)(mt * nt * z) / (float)h->sm_count;
                const float eff = waves / ceilf(waves) * (waves < 2.f ? 0.9f : 1.f);
                if (eff > best + 0.01f) {
                    best = eff;
                    splits = z;
                }
            }
            const int kchunk = ((N + splits - 1) / splits + BK - 1) / BK * BK;
            splits = (N + kchunk - 1) / kchunk;
            if (tn == 32)
                SEV_LAUNCH(h, K_SYMM, (symm_kernel<T, 32>), dim3(mt, nt, splits), 256, 0, N, b, A22, lda, B.U, N, kchunk,
                           B.ypart, (size_t)N * b);
            else
                SEV_LAUNCH(h, K_SYMM, (symm_kernel<T, 64>), dim3(mt, nt, splits), 256, 0, N, b, A22, lda, B.U, N, kchunk,
                           B.ypart, (size_t)N * b);
        }
        // M = U^T Y; Zh = T^T M T / 2; V = U Zh - Y T (= U (T^T U^T X) / 2 - X with X = Y T)
        const T *Y = splits > 1 ? B.Y : B.ypart;
        const int chunk = uty_chunk(N), parts = uty_parts(N);
        T *Msum = B.part + (size_t)parts * b * b;
        __nv_bfloat16 *bp = nullptr, *bq = nullptr;
        int K6p = 0;
        if (tc) tc_panels<T>(N, b, B.tc_ws, &bp, &bq, &K6p);
        const size_t s_zh = sizeof(T) * (size_t)b * 8;
        auto vform = [&](auto tnc) -> int {
            constexpr int TN = decltype(tnc)::value;
            const int nt = (b + TN - 1) / TN;
            SEV_LAUNCH(h, K_VFORM_UTX, (uty_kernel<T, TN>), dim3(nt, nt, parts), 256, 0, N, b, chunk, B.U, splits,
                       B.ypart, (size_t)N * b, B.Y, B.part);
            SEV_LAUNCH(h, K_VFORM_REDUCE, uty_sum_kernel<T>, (b * b + 255) / 256, 256, 0, b * b, parts, B.part, Msum);
            SEV_LAUNCH(h, K_VFORM_REDUCE, (uty_zh_kernel<T, 4>), (b + 3) / 4, 256, s_zh, b, Msum, B.Tm, B.Zm);
            SEV_LAUNCH(h, K_VFORM_V, (vform_kernel<T, TN>), dim3((N + BM - 1) / BM, nt), 256, 0, N, b, B.U, Y, B.Zm,
                       B.Tm, B.V, K6p, bp, bq);
            return SEV_OK;
        };
        rc = b <= 32 ? vform(std::integral_constant<int, 32>{}) : vform(std::integral_constant<int, 64>{});
        if (rc) return rc;
        // A22 += U V^T + V U^T
        if (tc) {
            rc = tc_syr2k<T>(h, N, b, A22, lda, B.tc_ws);
            if (rc) return rc;
        } else {
            const long nt = (N + BM - 1) / BM;
            SEV_LAUNCH(h, K_SYR2K, syr2k_kernel<T>, (unsigned)(nt * (nt + 1) / 2), 256, 0, N, b, A22, lda, B.U, N, B.V,
                       N);
        }
    }
    return launch_band_from_dense<T>(h, n, A, lda, b, AB, ldab);
}

template int launch_full_to_band<float>(sev_ctx *, int, float *, int, int, float *, int, void *, size_t, bool);
template int launch_full_to_band<double>(sev_ctx *, int, double *, int, int, double *, int, void *, size_t, bool);
template size_t full_to_band_copy_bytes<float>(sev_ctx *, int, int, const float *, int);
template size_t full_to_band_copy_bytes<double>(sev_ctx *, int, int, const double *, int);
template size_t full_to_band_workspace<float>(sev_ctx *, int, int);
template size_t full_to_band_workspace<double>(sev_ctx *, int, int);

}  // namespace sev
