// tri_step.cuh -- the steps of the b -> 1 reduction (Algorithm 4.2 with h = 1) on
// a column window of the packed band in shared memory: D (diagonal block) and
// M (block below, next reflector) of step (i, j) as band_tri.cu describes them,
// each by one warp.  Shared by the sliding-window kernel (band_tri.cu: D and M
// on two warps, the window a ring) and the batched kernel (batched.cu: both on
// one warp, the window the whole band).
#pragma once
#include "common.cuh"

namespace sev {

constexpr int kTriInf = 1 << 30;

__host__ __device__ __forceinline__ int tri_chases(int n, int b, int i) {
    const int r = n - i;
    return r < 2 ? 0 : (n - 2 - i) / b + 1;
}

// Lane layout of a B x B block: lane = r + B g holds row (or column) r,
// entries g, g + LPR, g + 2 LPR, ... of it; lanes past B LPR hold nothing.
template <int B>
struct TriLanes {
    static constexpr int LPR = 32 / B < B ? 32 / B : B;  // lanes per row
    static constexpr int CPL = B / LPR;                  // entries per lane
    static constexpr int ON = B * LPR;                   // lanes in use
};

// Element k of the ring counted from element `base` (base < S).  WRAP = false:
// the caller knows that the block it works on does not cross the ring's end,
// so the offsets are immediates of the loads and stores.
template <typename T, int S, bool WRAP>
__device__ __forceinline__ T &tri_at(T *w, int base, int k) {
    return WRAP ? w[(base + k) & (S - 1)] : w[base + k];
}
constexpr int kTriVec = 40;  // spacing of the per-sweep vector buffers (v: B entries, tau at B)

// Sum over the LPR lanes that share a row / over the B rows of a lane group.
template <int B, typename T>
__device__ __forceinline__ T tri_sum_row(T s) {
#pragma unroll
    for (int off = B; off < TriLanes<B>::ON; off <<= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
}

// tri_house for a column whose squares leave the range of its type, or a zero
// one: the column is held times a power of two.  Beside larger entries an
// inexact tau would spoil these, and in a matrix of that scale the column is not
// negligible.  A function of its own: rare, and its registers stay out of the
// steps.  (The test for it costs FP64 1-2% of the stage -- 16 -> 1 at n = 3001
// 23.0 -> 23.2 ms -- and FP32 nothing.)
template <typename T>
struct TriHouse {
    T v, tau, beta;
};
template <int B>
__device__ __noinline__ TriHouse<float> tri_house_scaled(float x, int r, int nr, float sc) {
    const float y = x * sc;
    const F2 acc = warp_sum_f2<B>(two_prod(y, y));
    TriHouse<float> h;
    float inv;
    house_scalars_f2s(__shfl_sync(0xffffffffu, y, 0), acc, &h.tau, &h.beta, &inv);
    h.beta /= sc;
    h.v = r == 0 ? 1.f : (r < nr ? y * inv : 0.f);
    return h;
}
template <int B>
__device__ __noinline__ TriHouse<double> tri_house_scaled(double x, int r, int nr) {
    const unsigned hi = r < nr ? (unsigned)__double2hiint(x) & 0x7fffffffu : 0u;
    const int e = house_scale_exp(__reduce_max_sync(0xffffffffu, hi));
    const double y = x * pow2i(-e);
    const bool rest = r >= 1 && r < nr;
    double a = rest ? y * y : 0.0;
#pragma unroll
    for (int off = B / 2; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    TriHouse<double> h;
    double inv;
    house_scalars(__shfl_sync(0xffffffffu, y, 0), a, &h.tau, &h.beta, &inv);
    h.beta *= pow2i(e);
    h.v = r == 0 ? 1.0 : (rest ? y * inv : 0.0);
    return h;
}

// Reflector of x (row r of the column in every lane with that r; rows >= nr
// zero): v, tau and beta in every lane; squares and scalars FP64-accurate
// (pair-float for FP32 data).
template <typename T, int B>
__device__ __forceinline__ void tri_house(T x, int r, int nr, T &v, T &tau, T &beta) {
    const bool rest = r >= 1 && r < nr;
    if constexpr (sizeof(T) == 4) {
        const F2 acc = warp_sum_f2<B>(two_prod((float)x, (float)x));  // alpha^2 included
        float tf, bf, inf;
        house_scalars_f2s_core(__shfl_sync(0xffffffffu, (float)x, 0), acc, &tf, &bf, &inf);
        tau = (T)tf;
        beta = (T)bf;
        v = r == 0 ? T(1) : (rest ? x * (T)inf : T(0));
        if (house_f2_needs_scale(acc.hi)) {  // (the same in every lane; asked here the test is off the chain)
            const TriHouse<float> h = tri_house_scaled<B>((float)x, r, nr, house_f2_scale(acc.hi));
            tau = (T)h.tau, beta = (T)h.beta, v = (T)h.v;
        }
    } else {
        double a = rest ? (double)x * (double)x : 0.0;
#pragma unroll
        for (int off = B / 2; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        const double alpha = (double)__shfl_sync(0xffffffffu, x, 0), s = fma(alpha, alpha, a);
        if (house_needs_scale(s)) {  // (the same in every lane)
            const TriHouse<double> h = tri_house_scaled<B>((double)x, r, nr);
            tau = (T)h.tau, beta = (T)h.beta, v = (T)h.v;
            return;
        }
        double td, bd, id;
        house_scalars_core(alpha, s, &td, &bd, &id);
        tau = (T)td;
        beta = (T)bd;
        v = r == 0 ? T(1) : (rest ? x * (T)id : T(0));
    }
}

// This lane's entries of a vector whose entry r is held by the lanes of row r.
template <typename T, int B>
__device__ __forceinline__ void tri_spread(T x, T (&v)[TriLanes<B>::CPL]) {
    const int g = (threadIdx.x & 31) / B;
#pragma unroll
    for (int q = 0; q < TriLanes<B>::CPL; ++q) {
        const T e = __shfl_sync(0xffffffffu, x, g + TriLanes<B>::LPR * q);
        v[q] = TriLanes<B>::ON == 32 || g < TriLanes<B>::LPR ? e : T(0);
    }
}

// Step (i, 0): H_1 from column i - 1, rows [i, i + nr).
template <typename T, int B, int S>
__device__ __forceinline__ void tri_first(T *w, int n, int i, T *vn, T (&v)[TriLanes<B>::CPL], T &tau) {
    constexpr int LDW = 2 * B;
    const int lane = threadIdx.x & 31, r = lane % B;
    const int nr = min(n - i, B);
    T *px = w + (((i - 1) * LDW + 1 + r) & (S - 1));
    const T x = r < nr ? *px : T(0);
    T nv, beta;
    tri_house<T, B>(x, r, nr, nv, tau, beta);
    tri_spread<T, B>(nv, v);
    __syncwarp();
    if (lane < B) {
        if (r < nr) *px = r == 0 ? beta : T(0);
        vn[r] = nv;
        if (r == 0) vn[B] = tau;
    }
}

// M of step (i, j) by one warp: M H_j, then H_{j+1} from the first column and
// H_{j+1} M on the others.  v, tau: this lane's entries of v_j and tau_j on
// entry, of v_{j+1} and tau_{j+1} on return (also stored to vn for the warp
// of D).  FULL: M has b rows (sizes known at compile time).
template <typename T, int B, int S, bool FULL, bool WRAP>
__device__ __forceinline__ void tri_bulge(T *w, int n, int o, T (&v)[TriLanes<B>::CPL], T &tau, T *vn) {
    constexpr int LDW = 2 * B, LPR = TriLanes<B>::LPR, CPL = TriLanes<B>::CPL;
    const int lane = threadIdx.x & 31, r = lane % B, g = lane / B;
    const bool on = TriLanes<B>::ON == 32 || g < LPR;
    const int mb = FULL ? B : min(n - (o + B), B);
    if (!FULL && mb < 1) return;
    T x[CPL];
    const int base = (o * LDW) & (S - 1);
    const int xo = B + r;  // entry (row r, column 0); column c lies LDW - 1 further
#pragma unroll
    for (int q = 0; q < CPL; ++q)
        x[q] = (on && (FULL || r < mb)) ? tri_at<T, S, WRAP>(w, base + xo + g * (LDW - 1), LPR * q * (LDW - 1)) : T(0);
    T s = T(0), s1 = T(0);
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
        if (q & 1)
            s1 = fma(x[q], v[q], s1);
        else
            s = fma(x[q], v[q], s);
    }
    s = tau * tri_sum_row<B>(s + s1);
#pragma unroll
    for (int q = 0; q < CPL; ++q) x[q] = fma(-s, v[q], x[q]);
    const T x0 = __shfl_sync(0xffffffffu, x[0], r);
#pragma unroll
    for (int q = 0; q < CPL; ++q)
        if (on && (FULL || r < mb)) tri_at<T, S, WRAP>(w, base + xo + g * (LDW - 1), LPR * q * (LDW - 1)) = x[q];
    if (!FULL && mb < 2) return;
    __syncwarp();
    // the same block by columns: lane column r, rows g + LPR q
    T y[CPL];
    const int yo = base + B + r * (LDW - 1) + g;
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
        const int rr = g + LPR * q;
        y[q] = (on && (FULL || rr < mb)) ? tri_at<T, S, WRAP>(w, yo, LPR * q) : T(0);
    }
    T nv, nbeta;
    tri_house<T, B>(x0, r, mb, nv, tau, nbeta);
    tri_spread<T, B>(nv, v);
    if (lane < B) vn[r] = nv;
    if (lane == 0) vn[B] = tau;
    T z = T(0), z1 = T(0);
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
        if (q & 1)
            z1 = fma(v[q], y[q], z1);
        else
            z = fma(v[q], y[q], z);
    }
    z = tau * tri_sum_row<B>(z + z1);
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
        const int rr = g + LPR * q;
        T val = fma(-z, v[q], y[q]);
        if (r == 0) val = rr == 0 ? nbeta : T(0);
        if (on && (FULL || rr < mb)) tri_at<T, S, WRAP>(w, yo, LPR * q) = val;
    }
}

// D of step (i, j) by one warp.  vb: v_j, tau_j at vb[B]; wb: B entries of
// scratch.
template <typename T, int B, int S, bool FULL, bool WRAP>
__device__ __forceinline__ void tri_diag(T *w, int n, int o, const T *vb, T *wb) {
    constexpr int LDW = 2 * B, LPR = TriLanes<B>::LPR, CPL = TriLanes<B>::CPL;
    const int lane = threadIdx.x & 31, r = lane % B, g = lane / B;
    const bool on = TriLanes<B>::ON == 32 || g < LPR;
    const int nr = FULL ? B : min(n - o, B);
    T x[CPL], vc[CPL];
    const T tau = vb[B], vr = vb[r];
    const int base = (o * LDW) & (S - 1);
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
        const int c = g + LPR * q;
        const int off = c <= r ? c * (LDW - 1) + r : r * (LDW - 1) + c;
        vc[q] = on ? vb[c] : T(0);
        x[q] = (on && (FULL || (r < nr && c < nr))) ? tri_at<T, S, WRAP>(w, base, off) : T(0);
    }
    T p = T(0), p1 = T(0);
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
        if (q & 1)
            p1 = fma(x[q], vc[q], p1);
        else
            p = fma(x[q], vc[q], p);
    }
    p = tau * tri_sum_row<B>(p + p1);
    T ptv = p * vr;
#pragma unroll
    for (int off = B / 2; off > 0; off >>= 1) ptv += __shfl_xor_sync(0xffffffffu, ptv, off);
    const T wr = fma(T(-0.5) * tau * ptv, vr, p);
    if (lane < B) wb[r] = wr;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
        const int c = g + LPR * q;
        if (on && c <= r && (FULL || r < nr))
            tri_at<T, S, WRAP>(w, base + g * (LDW - 1) + r, LPR * q * (LDW - 1)) = fma(-vr, wb[c], fma(-wr, vc[q], x[q]));
    }
}

}  // namespace sev
