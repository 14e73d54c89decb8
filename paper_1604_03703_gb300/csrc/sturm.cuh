// sturm.cuh -- the Sturm count of the bisection (the number of sign changes of
// the leading principal minors of T - xI), shared by the single-matrix
// (bisect.cu) and the batched (batched.cu) bisection.  T is scaled so that its
// Gershgorin bound lies in [0.5, 1): every |d_i - x| <= 2 and e_i^2 <= 1.
#pragma once
#include "common.cuh"

namespace sev {

__device__ __forceinline__ double pow2_exact(int k) {  // 2^k, -1022 <= k <= 1023
    return __longlong_as_double((long long)(1023 + k) << 52);
}

// One step of the minors recurrence with t = d_i sc - x: u = e_{i-1}^2 a,
// p = t b - u; sign, zero test and exponent from the bits (integer work, so
// the FP64 pipe sees only the three operations), rescaling by a power of two
// when |p| leaves [2^-256, 2^256].  Two zero minors in a row: T splits here (e is
// zero, or negligible) behind a block that is singular at x, all further
// minors of the whole would vanish, and the count goes on with those of the
// rest by itself (1, t, ...).
__device__ __forceinline__ void sturm_step(double di, double e2i, double x, double sc, double &a, double &b,
                                           bool &neg, int &c) {
    const double t = __fma_rn(di, sc, -x);
    const double u = __dmul_rn(e2i, a);
    double p = __fma_rn(t, b, -u);
    long long pb = __double_as_longlong(p);
    if (((pb | __double_as_longlong(b)) << 1) == 0) {
        p = t;
        pb = __double_as_longlong(p);
        b = 1.0;
        neg = false;
    }
    const bool zero = (pb << 1) == 0;
    const bool pn = zero ? !neg : pb < 0;
    c += pn != neg;
    neg = pn;
    a = b;
    b = p;
    const int ex = (int)((pb >> 52) & 0x7FF);
    if (__builtin_expect(ex > 1023 + 256 || (ex < 1023 - 256 && !zero), 0)) {
        int k = 1023 - ex;
        k = k > 512 ? 512 : (k < -512 ? -512 : k);
        const double f = pow2_exact(k);
        a = __dmul_rn(a, f);
        b = __dmul_rn(b, f);
    }
}

// The count at x for d_i = ld_d(i), e_i^2 = ld_e(i) (loads of the next block
// issue ahead of this block's arithmetic).
//
// What bounds it: the FP64 pipe, 3 instructions of ~64 cycles per step and
// warp.  A branch on every p (sturm_step) kept the next step's t and u from
// being issued while p was in the pipe: 440 cycles a step with one warp per
// scheduler.  So blocks of U steps run without it: signs are shifted
// into a mask and counted at the end, and the pair is rescaled once a block by
// adding to the exponent fields.
// Same count: scaling (p_{i-1}, p_i) by a power of two changes no sign, and
// changes no rounding while nothing under- or overflows.  |p| grows by less
// than 2^2 a step, so nothing overflows.  `plain` says that no nonzero e_i^2
// is below 2^-322; then u does not underflow while every |p| of the block and
// before it is >= 2^-700.  A block with a smaller |p| (or p = 0, whose sign is
// defined by its predecessor, and behind which T may split) is run again step by
// step from where it began.
// Blocks of 8 in the single-matrix kernels (16384 eigenvalues at 1e-14: U = 4
// 79.2 ms, 8 76.5, 16 spills; 118.3 with the branch in every step), of 4 in the
// batched kernel, whose other phases need the registers.
constexpr int kSturmMinHi = (1023 - 700) << 20;
template <int kSturmU, typename LD, typename LE>
__device__ __forceinline__ int sturm_count_blocks(int n, LD ld_d, LE ld_e, double x, double sc, bool plain) {
    double a = 1.0, b = __fma_rn(ld_d(0), sc, -x);
    bool neg = b <= 0.0;  // p_0 = 1 > 0: a zero p_1 counts as negative
    int c = neg;
    double dn[kSturmU], en[kSturmU];
#pragma unroll
    for (int u = 0; u < kSturmU; ++u) {
        const int i = 1 + u;
        dn[u] = i < n ? ld_d(i) : 0.0;
        en[u] = i < n ? ld_e(i - 1) : 0.0;
    }
    for (int i0 = 1; i0 < n; i0 += kSturmU) {
        double dc[kSturmU], ec[kSturmU];
        const bool whole = i0 + 2 * kSturmU <= n;
#pragma unroll
        for (int u = 0; u < kSturmU; ++u) {
            dc[u] = dn[u];
            ec[u] = en[u];
            const int i = i0 + kSturmU + u;
            dn[u] = whole || i < n ? ld_d(i) : 0.0;
            en[u] = whole || i < n ? ld_e(i - 1) : 0.0;
        }
        bool redo = true;
        if (plain && i0 + kSturmU <= n) {
            double pa = a, pb = b, w = __dmul_rn(ec[0], a);
            unsigned signs = neg;
            int mn = 0x7fffffff;
#pragma unroll
            for (int u = 0; u < kSturmU; ++u) {
                const double t = __fma_rn(dc[u], sc, -x);
                const double wn = u + 1 < kSturmU ? __dmul_rn(ec[u + 1], pb) : 0.0;
                const double p = __fma_rn(t, pb, -w);
                const int hi = __double2hiint(p);
                signs = __funnelshift_l((unsigned)hi, signs, 1);
                mn = min(mn, hi & 0x7fffffff);
                pa = pb;
                pb = p;
                w = wn;
            }
            redo = mn < kSturmMinHi;
            if (!redo) {
                c += __popc((signs ^ (signs >> 1)) & ((1u << kSturmU) - 1));
                neg = signs & 1;
                const int hi = __double2hiint(pb), ex = (hi >> 20) & 0x7FF;
                int k = 1023 - ex;
                k = k > 512 ? 512 : (k < -512 ? -512 : k);
                k = (ex > 1023 + 256 || ex < 1023 - 256) ? k << 20 : 0;
                // (pa and pb are both of this block, so mn covers their exponents)
                a = __hiloint2double(__double2hiint(pa) + k, __double2loint(pa));
                b = __hiloint2double(hi + k, __double2loint(pb));
            }
        }
        if (redo) {
#pragma unroll
            for (int u = 0; u < kSturmU; ++u)
                if (i0 + u < n) sturm_step(dc[u], ec[u], x, sc, a, b, neg, c);
        }
    }
    return c;
}

}  // namespace sev
