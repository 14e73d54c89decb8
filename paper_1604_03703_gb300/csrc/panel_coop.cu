// panel_coop.cu -- the panel factorisation of the full-to-band reduction (the
// QR step of Algorithm 4.1) by the whole GPU at once: one cooperative kernel
// holds the N x b panel in registers, 32 RT rows per CTA, and runs the
// Householder QR column by column with ONE exchange between the CTAs per
// column.
//
// Why not the tree (Algorithm 3.2).  A tree of leaf and node QRs pays a chain
// of b columns at every one of its ~log2(N / 256) + 1 levels, then the way
// down, then the reconstruction of (U, T) from the explicit Q.  Its point is to
// exchange data once per level instead of once per column, which pays when an
// exchange costs much more than a column; between the SMs of one GPU an
// exchange through L2 takes ~0.7 us and a column of a leaf or node QR
// ~1.5-2 us.  Direct columns need neither the way down nor the reconstruction:
// U, tau and R are the result (the same reflectors: beta = -sgn(alpha) ||x||,
// tau in [1, 2]).  Measured (GB300): the whole panel step at n = 16384, b = 128
// (FP32) 276 -> 66 ms per reduction, n = 8192, b = 64 101 -> 19 ms, n = 2048, b =
// 64 16.1 -> 4.0 ms; n = 3001, b = 32 in FP64 200 -> 16 ms.
//
// One exchange per column.  With x = column k below row k (zero above) and
// v = e_k + x / (alpha - beta), the products v^T a_j that the reflector needs
// are a_kj + (x^T a_j) / (alpha - beta), so every CTA can send its share of
// x^T x and of x^T a_j for ALL columns j before tau and beta are known; for
// finished columns j < k the same expression is G(j, k) = v_j^T v_k, from
// which the last CTA forms the compact-WY factor T while it waits for the
// next exchange.  The panel is held times the power of two of its largest entry
// (exact; not x alone: x may be 1e-140 of it, and x^T a_j must not underflow before
// it is divided by alpha - beta); x^T x of FP32 data is summed error-free in pairs
// of floats.
//
// Exchange.  Every value travels as one 8-byte word (FP64: two) holding the
// 32 bits and a tag (panel and column), stored and polled with single 8-byte
// accesses: a word whose tag is right is complete, so no fence, flag or
// barrier is needed.  Two sets of words alternate: a CTA sends column k + 1
// only after it has read all of column k, so whoever has read column k + 1
// knows that column k's words may be overwritten.  Panels of up to 4096 rows
// (2048 over 64 columns, FP64 1024) run on one cluster of at most 16 CTAs, the words going from
// shared memory to shared memory; taller ones on the whole GPU (cooperative
// launch, at most one CTA per SM) through L2.  Every wait is capped and latches
// SEV_ERR_TIMEOUT on expiry.
//
// What bounds it: the chain of one column -- dot products and their warp sums,
// L2 store to load (~1.4K cycles), the sum over the CTAs, the reflector
// scalars, the update of column k + 1.  Every CTA reads every CTA's shares:
// C^2 b words per column, which is why the rows per CTA grow with N.
#include "regtile.cuh"

namespace sev {

// NW column warps and one more for the scalars.  8 column warps hold up to 64
// columns (fewer warps: fewer sums, barriers and copies of x per column); 16
// hold 128.
constexpr int kCoopMaxB = 128;

// ------------------------------------------------------- tagged words
// CL = false: words in global memory.  CL = true: every CTA of the cluster has
// the whole exchange buffer in its shared memory; a value is stored into each
// peer's copy (at the peer's address of the buffer) and polled in the own one.
__device__ __forceinline__ unsigned ll_peer(const void *own, int peer) {
    unsigned at;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(at)
                 : "r"((unsigned)__cvta_generic_to_shared(own)), "r"(peer));
    return at;
}
template <bool CL>
__device__ __forceinline__ void ll_put(unsigned long long *buf, unsigned peer, size_t word, unsigned v, unsigned tag) {
    const unsigned long long w = ((unsigned long long)tag << 32) | v;
    if constexpr (CL)
        asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(peer + 8 * (unsigned)word), "l"(w) : "memory");
    else
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(buf + word), "l"(w) : "memory");
}
template <bool CL>
__device__ __forceinline__ void ll_get2(const unsigned long long *p, unsigned long long &a, unsigned long long &b) {
    if constexpr (CL)
        asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];"
                     : "=l"(a), "=l"(b)
                     : "r"((unsigned)__cvta_generic_to_shared(p))
                     : "memory");
    else
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ bool ll_is(unsigned long long w, unsigned tag) { return (unsigned)(w >> 32) == tag; }

// A value of type T as tagged words: 1 for float, 2 for double.
template <typename T>
struct LLType;
template <>
struct LLType<float> {
    static constexpr int W = 1;
};
template <>
struct LLType<double> {
    static constexpr int W = 2;
};
template <bool CL>
__device__ __forceinline__ void ll_put_val(unsigned long long *buf, unsigned peer, size_t word, float v, unsigned tag) {
    ll_put<CL>(buf, peer, word, __float_as_uint(v), tag);
}
template <bool CL>
__device__ __forceinline__ void ll_put_val(unsigned long long *buf, unsigned peer, size_t word, double v, unsigned tag) {
    ll_put<CL>(buf, peer, word, (unsigned)__double2loint(v), tag);
    ll_put<CL>(buf, peer, word + 1, (unsigned)__double2hiint(v), tag);
}
__device__ __forceinline__ void coop_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Layout of the exchange buffer (in words) for at most cmax - 1 CTAs (cmax
// even): per column one entry per CTA, its share of x^T a_j, and behind them
// the entry of row k; then two words per CTA for its share of x^T x.
template <typename T>
struct CoopComm {
    static __host__ __device__ size_t col_words(int b, int cmax) { return (size_t)b * cmax * LLType<T>::W; }
    static __host__ __device__ size_t ssq_words(int cmax) { return (size_t)cmax * 2; }
    // two alternating sets of (columns, squares), then the largest entries
    static __host__ __device__ size_t set_words(int b, int cmax) { return col_words(b, cmax) + ssq_words(cmax); }
    static __host__ __device__ size_t words(int b, int cmax) { return 2 * set_words(b, cmax) + ssq_words(cmax); }
};

// A failed try of a polling loop: true when the wait has to be given up.
__device__ __forceinline__ bool coop_give_up(int tries, long long &t0, long long cap, int *err) {
    if (tries == 0) t0 = clock64();
    int stop = 0;
    if ((threadIdx.x & 31) == 0) {
        if ((tries & 31) == 31 && any_gave_up(err)) stop = 1;
        if (wait_expired(t0, cap)) {
            latch_timeout(err);
            stop = 1;
        }
    }
    return __shfl_sync(0xffffffffu, stop, 0) != 0;
}

// Totals over the C CTAs of QH of this warp's columns (warp + NW (q0 + q)) into
// sd, their entries of row k into sr (shared memory, by column).  Every lane
// polls its entries until all carry `tag` (the tags of a try are compared with
// one OR per word, nothing else is done before they fit) and sums them in
// order; false when the wait ran out.
template <typename T, int QH, int NW, bool CL>
__device__ __forceinline__ bool coop_collect(const unsigned long long *cols, int cmax, int C, int warp, int q0, int b,
                                             unsigned tag, long long cap, int *err, T *sd, T *sr) {
    const int lane = threadIdx.x & 31;
    constexpr int W = LLType<T>::W, PER = W == 1 ? 2 : 1;  // entries per 16-byte load
    const unsigned long long *base = cols + (size_t)(warp + NW * q0) * cmax * W + PER * W * lane;
    const size_t step = (size_t)NW * cmax * W;
    T sum[QH], row[QH];
#pragma unroll
    for (int q = 0; q < QH; ++q) sum[q] = row[q] = T(0);
    for (int c0 = 0; c0 <= C; c0 += 32 * PER) {
        const int c = c0 + PER * lane;
        const unsigned my = c <= C ? 0xffffffffu : 0u, my1 = W == 2 || c + 1 <= C ? my : 0u;
        unsigned long long x[QH], y[QH];
        long long t0 = 0;
        for (int tries = 0;; ++tries) {
#pragma unroll
            for (int q = 0; q < QH; ++q) {
                x[q] = y[q] = (unsigned long long)tag << 32;
                if (warp + NW * (q0 + q) < b && c <= C) ll_get2<CL>(base + q * step + (size_t)c0 * W, x[q], y[q]);
            }
            unsigned bad = 0;
#pragma unroll
            for (int q = 0; q < QH; ++q) bad |= (((unsigned)(x[q] >> 32) ^ tag) & my) | (((unsigned)(y[q] >> 32) ^ tag) & my1);
            if (__all_sync(0xffffffffu, bad == 0)) break;
            if (coop_give_up(tries, t0, cap, err)) return false;
        }
#pragma unroll
        for (int q = 0; q < QH; ++q) {
            if constexpr (W == 1) {
                const float v0 = __uint_as_float((unsigned)x[q]), v1 = __uint_as_float((unsigned)y[q]);
                sum[q] += c < C ? v0 : 0.f;
                sum[q] += c + 1 < C ? v1 : 0.f;
                row[q] = c == C ? v0 : (c + 1 == C ? v1 : row[q]);
            } else {
                const double v = __hiloint2double((int)(unsigned)y[q], (int)(unsigned)x[q]);
                sum[q] += c < C ? v : 0.0;
                row[q] = c == C ? v : row[q];
            }
        }
    }
    const T s = warp_sums_t<T, QH>(sum);
    const int j = warp + NW * (q0 + lane / (32 / QH));
    if ((lane & (32 / QH - 1)) == 0 && j < b) sd[j] = s;
    if (lane == (C / PER) % 32) {
#pragma unroll
        for (int q = 0; q < QH; ++q)
            if (warp + NW * (q0 + q) < b) sr[warp + NW * (q0 + q)] = row[q];
    }
    return true;
}

// A pair of words per entry i < cnt (lane takes i = lane, lane + 32, ...) and
// (ENTRY) one entry of the columns for lane 0, polled until tagged.  f(i ==
// lane, word0, word1) is called for every entry, in order, of the last try.
template <typename T, bool CL, bool ENTRY, typename F>
__device__ __forceinline__ bool coop_poll_pairs(const unsigned long long *p, int cnt, const unsigned long long *entry,
                                                T &val, unsigned tag, long long cap, int *err, F f) {
    const int lane = threadIdx.x & 31;
    long long t0 = 0;
    for (int tries = 0;; ++tries) {
        bool ok = true;
        if (ENTRY && lane == 0) {
            // (the 16-byte aligned pair that holds the entry)
            const bool odd = ((uintptr_t)entry & 8) != 0;
            unsigned long long a, b;
            ll_get2<CL>(entry - (odd ? 1 : 0), a, b);
            if constexpr (sizeof(T) == 4) {
                ok = ll_is(odd ? b : a, tag);
                val = __uint_as_float((unsigned)(odd ? b : a));
            } else {
                ok = ll_is(a, tag) && ll_is(b, tag);
                val = __hiloint2double((int)(unsigned)b, (int)(unsigned)a);
            }
        }
        for (int i = lane; i < cnt; i += 32) {
            unsigned long long a, b;
            ll_get2<CL>(p + 2 * (size_t)i, a, b);
            ok = ok && ll_is(a, tag) && ll_is(b, tag);
            f(i == lane, (unsigned)a, (unsigned)b);
        }
        if (__all_sync(0xffffffffu, ok)) return true;
        if (coop_give_up(tries, t0, cap, err)) return false;
    }
}

template <typename T, int RT>
struct CoopSmem {
    T xs[2][32 * RT];          // column k below row k
    T sd[kCoopMaxB], sr[kCoopMaxB];  // x^T a_j and row k of the column being formed
    T gs[kCoopMaxB];           // G(j, k), j < k (last CTA)
    T part[16 * 32];           // partial sums of a column of T (last CTA)
    T tau[kCoopMaxB];
    T sc[4];                   // tau, beta, 1 / (alpha - beta) of the column; the panel's scale
    int abort;
};

// Column kc of T by the last CTA, in two halves with a barrier between them:
// T(a, kc) = -tau sum_{q = a}^{kc - 1} T(a, q) G(q, kc) (forward, column-wise:
// Q = I - U T U^T).  Ts: column-major, ld b, zero below the diagonal.
template <typename T, int NW>
__device__ __forceinline__ void coop_t_partial(int b, int kc, const T *Ts, const T *gs, T *part) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nrg = (b + 31) / 32, nsl = NW / nrg;
    const int a = 32 * (warp % nrg) + lane, sl = warp / nrg;
    if (sl >= nsl) return;
    T s0 = T(0);
    if (a < b)
        for (int q = sl; q < kc; q += nsl) s0 = fmat(Ts[(size_t)q * b + a], gs[q], s0);
    if (a < b) part[sl * b + a] = s0;
}
template <typename T, int NW>
__device__ __forceinline__ void coop_t_column(int b, int kc, T *Ts, const T *tau, const T *part) {
    const int lane = threadIdx.x & 31;
    const int nsl = NW / ((b + 31) / 32);
    const T tk = tau[kc];
    for (int a = lane; a <= kc; a += 32) {
        T s = T(0);
        if (a < kc)
            for (int l = 0; l < nsl; ++l) s += part[l * b + a];
        Ts[(size_t)kc * b + a] = a == kc ? tk : -tk * s;
    }
}

// P: N x b panel (ldp).  On return U (N x b, ld N) holds the reflectors (unit
// lower trapezoidal), Tm (b x b) the compact-WY factor, and P the band block
// (R over zeros).  comm: exchange words; tags tag0 + 1 .. tag0 + b + 1 are
// unused so far in it.
template <typename T, int RT, int Q, int NW, bool CL>
__global__ void __launch_bounds__((NW + 1) * 32, 1)
    panel_coop_kernel(T *__restrict__ P, int ldp, int N, int b, T *__restrict__ U, T *__restrict__ Tm,
                      unsigned long long *comm, int cmax, unsigned tag0, int *err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CoopSmem<T, RT> &S = *reinterpret_cast<CoopSmem<T, RT> *>(smem_raw);
    T *Ts = reinterpret_cast<T *>(smem_raw + ((sizeof(CoopSmem<T, RT>) + 15) & ~(size_t)15));  // last CTA
    constexpr int R = 32 * RT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x, C = gridDim.x;
    const bool lastc = c == C - 1;
    const int row0 = c * R, rows = min(R, N - row0);
    const int nref = min(b, N - 1);
    const long long cap = wait_cap(err);
    using Comm = CoopComm<T>;
    if constexpr (CL) {
        // the exchange buffer of this CTA behind T; no tag may be found in what
        // the memory held before, nor a word arrive before that is so
        comm = reinterpret_cast<unsigned long long *>(Ts + (size_t)((b * b + 3) & ~3));
        const int nw = (int)Comm::words(b, cmax);
        for (int i = threadIdx.x; i < nw; i += blockDim.x) comm[i] = 0;
        coop_cluster_sync();
    }
    unsigned long long *const amx = comm + 2 * Comm::set_words(b, cmax);
    // A column warp's lanes lane / (32 / Q) = q serve column q, the peers dealt to
    // them; the scalar warp's lanes one peer each.  (Global memory: one place.)
    constexpr int LPQ = 32 / Q, NP = CL ? (16 + LPQ - 1) / LPQ : 1;
    unsigned peer[NP];
    int npeer = 0;
    if constexpr (CL) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int to = warp < NW ? (lane & (LPQ - 1)) + LPQ * i : lane;
            peer[i] = to < C ? ll_peer(comm, to) : 0;
            npeer += to < C && (warp < NW || i == 0);
        }
    } else {
        peer[0] = 0;
        npeer = (warp < NW ? (lane & (LPQ - 1)) : lane) == 0;
    }

    T a[Q][RT];
    if (warp < NW) {
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int t = 0; t < RT; ++t) {
                const int j = warp + NW * q, r = lane + 32 * t;
                a[q][t] = (j < b && r < rows) ? P[(size_t)(row0 + r) + (size_t)j * ldp] : T(0);
            }
    }
    if (threadIdx.x == 0) S.abort = 0;
    if (lastc)
        for (int i = threadIdx.x; i < b * b; i += blockDim.x) Ts[i] = T(0);
    // The panel's largest entry: the panel is held times its power of two, so that
    // no square or product that matters over- or underflows.
    {
        double m = 0.0;
        if (warp < NW) {
            T mt = T(0);
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int t = 0; t < RT; ++t) mt = max(mt, (T)fabs(a[q][t]));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mt = max(mt, __shfl_xor_sync(0xffffffffu, mt, o));
            if (lane == 0) S.part[warp] = mt;
        }
        __syncthreads();
        if (warp == NW) {
            m = lane < NW ? (double)S.part[lane] : 0.0;
            m = warp_max(m);
            if (npeer) ll_put_val<CL>(comm, peer[0], (amx - comm) + 2 * c, m, tag0 + 1);
            double g = 0.0;
            T none = T(0);
            const bool got = coop_poll_pairs<T, CL, false>(amx, C, nullptr, none, tag0 + 1, cap, err,
                                                                [&](bool first, unsigned lo, unsigned hi) {
                const double v = __hiloint2double((int)hi, (int)lo);
                g = first ? v : fmax(g, v);
            });
            g = warp_max(g);
            constexpr int EM = sizeof(T) == 8 ? 1000 : 126;
            int e2 = 0;
            if (g > 0.0 && isfinite(g)) (void)frexp(g, &e2);
            e2 = e2 > EM ? EM : (e2 < -EM ? -EM : e2);
            if (lane == 0) {
                S.sc[3] = (T)pow2i(-e2);
                if (!got) S.abort = 1;
            }
        }
    }
    __syncthreads();
    const T scale = S.sc[3], unscale = T(1) / scale;
    bool alive = !S.abort;
    if (warp < NW) {
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int t = 0; t < RT; ++t) a[q][t] *= scale;
    }
    if (warp == 0) {
#pragma unroll
        for (int t = 0; t < RT; ++t) S.xs[0][lane + 32 * t] = row0 + lane + 32 * t > 0 ? a[0][t] : T(0);
    }
    __syncthreads();

    for (int k = 0; k < nref && alive; ++k) {
        const unsigned tag = tag0 + 2 + k;
        const size_t set = (k & 1) * Comm::set_words(b, cmax), ssqw = set + Comm::col_words(b, cmax);
        const T *xk = S.xs[k & 1];
        if (warp < NW) {
            // ---- row k from the CTA that holds it, this CTA's shares of x^T a_j
            const int jq = warp + NW * (lane / LPQ);  // this lane's column to send
            if (c == 0) {
                T v = T(0);
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const T rv = __shfl_sync(0xffffffffu, rsel<RT>(a[q], k >> 5), k & 31);
                    v = lane / LPQ == q ? rv : v;
                }
                if (jq < b)
#pragma unroll
                    for (int i = 0; i < NP; ++i)
                        if (i < npeer)
                            ll_put_val<CL>(comm, peer[i], set + ((size_t)jq * cmax + C) * LLType<T>::W, v, tag);
            }
            T xr[RT];
#pragma unroll
            for (int t = 0; t < RT; ++t) xr[t] = xk[lane + 32 * t];
            T d[Q];
            if constexpr (sizeof(T) == 4) {
                float2 dd[Q / 2];
#pragma unroll
                for (int p = 0; p < Q / 2; ++p) dd[p] = make_float2(0.f, 0.f);
#pragma unroll
                for (int t = 0; t < RT; ++t) {
                    const float2 vv = make_float2(xr[t], xr[t]);
#pragma unroll
                    for (int p = 0; p < Q / 2; ++p) dd[p] = ffma2(vv, make_float2(a[2 * p][t], a[2 * p + 1][t]), dd[p]);
                }
#pragma unroll
                for (int p = 0; p < Q / 2; ++p) {
                    d[2 * p] = dd[p].x;
                    d[2 * p + 1] = dd[p].y;
                }
            } else {
#pragma unroll
                for (int q = 0; q < Q; ++q) d[q] = T(0);
#pragma unroll
                for (int t = 0; t < RT; ++t)
#pragma unroll
                    for (int q = 0; q < Q; ++q) d[q] = fmat(xr[t], a[q][t], d[q]);
            }
            const T mine = warp_sums_t<T, Q>(d);
            if (jq < b)
#pragma unroll
                for (int i = 0; i < NP; ++i)
                    if (i < npeer) ll_put_val<CL>(comm, peer[i], set + ((size_t)jq * cmax + c) * LLType<T>::W, mine, tag);
            if (lastc && k >= 1) coop_t_partial<T, NW>(b, k - 1, Ts, S.gs, S.part);
            constexpr int QH = Q > 4 && NW == 16 ? 4 : Q;  // (16 warps: 96 registers a thread)
            if (!CL) {
                // the slowest share is ~1.5K cycles away: a first look that fails only
                // loads the L2 (n = 8192 20.5 -> 19.3 ms of panels per reduction)
                const long long ts = clock64();
                while (clock64() - ts < 400) {
                }
            }
            bool ok = true;
#pragma unroll
            for (int q0 = 0; q0 < Q; q0 += QH)
                ok = ok && coop_collect<T, QH, NW, CL>(comm + set, cmax, C, warp, q0, b, tag, cap, err, S.sd, S.sr);
            if (!ok && lane == 0) S.abort = 1;
        } else {
            // ---- the scalar warp: x^T x over all CTAs, then tau, beta, 1 / (alpha - beta)
            bool ok = true;
            if constexpr (sizeof(T) == 4) {
                F2 p0{0.f, 0.f}, p1{0.f, 0.f};
#pragma unroll
                for (int t = 0; t < RT; t += 2) {
                    f2_add_sq(p0, (float)xk[lane + 32 * t]);
                    f2_add_sq(p1, (float)xk[lane + 32 * t + 32]);
                }
                const F2 mine = warp_sum_f2(f2_add(p0, p1));
                if (npeer) {
                    ll_put<CL>(comm, peer[0], ssqw + 2 * c, __float_as_uint(mine.hi), tag);
                    ll_put<CL>(comm, peer[0], ssqw + 2 * c + 1, __float_as_uint(mine.lo), tag);
                }
                F2 acc{0.f, 0.f};
                float alpha = 0.f;
                ok = coop_poll_pairs<float, CL, true>(comm + ssqw, C, comm + set + (size_t)k * cmax + C, alpha, tag, cap,
                                                      err, [&](bool first, unsigned hi, unsigned lo) {
                                                          const F2 v{__uint_as_float(hi), __uint_as_float(lo)};
                                                          acc = first ? v : f2_add(acc, v);
                                                      });
                alpha = __shfl_sync(0xffffffffu, alpha, 0);
                acc = warp_sum_f2(acc);
                float tau = 0.f, beta = 0.f, inv = 0.f;
                // a column 1e-16 times smaller than the panel's largest entry is a
                // zero column (its pair-float square would lose digits to underflow)
                if (fmaf(alpha, alpha, acc.hi) >= 1e-32f) house_scalars_f2(alpha, acc, &tau, &beta, &inv);
                if (lane == 0) {
                    S.sc[0] = (T)tau;
                    S.sc[1] = (T)beta;
                    S.sc[2] = (T)inv;
                    S.tau[k] = (T)tau;
                }
            } else {
                double s = 0.0;
#pragma unroll
                for (int t = 0; t < RT; ++t) {
                    const double x = (double)xk[lane + 32 * t];
                    s = fma(x, x, s);
                }
                s = warp_sum(s);
                if (npeer) ll_put_val<CL>(comm, peer[0], ssqw + 2 * c, s, tag);
                double acc = 0.0, alpha = 0.0;
                ok = coop_poll_pairs<double, CL, true>(comm + ssqw, C, comm + set + ((size_t)k * cmax + C) * 2, alpha, tag,
                                                       cap, err, [&](bool first, unsigned lo, unsigned hi) {
                                                           const double v = __hiloint2double((int)hi, (int)lo);
                                                           acc = first ? v : acc + v;
                                                       });
                acc = warp_sum(acc);
                alpha = __shfl_sync(0xffffffffu, alpha, 0);
                double tau = 0.0, beta = 0.0, inv = 0.0;
                // a column 1e-140 times smaller than the panel's largest entry is a
                // zero column (its square could not be told from underflow)
                if (fma(alpha, alpha, acc) >= 1e-280) house_scalars(alpha, acc, &tau, &beta, &inv);
                if (lane == 0) {
                    S.sc[0] = (T)tau;
                    S.sc[1] = (T)beta;
                    S.sc[2] = (T)inv;
                    S.tau[k] = (T)tau;
                }
            }
            if (!ok && lane == 0) S.abort = 1;
        }
        __syncthreads();
        alive = !S.abort;
        if (warp < NW) {
            // ---- a_j -= tau (v^T a_j) v for j > k; column k becomes (beta, v); G(j, k) for j < k
            const T tau = S.sc[0], beta = S.sc[1], inv = S.sc[2];
            T v[RT];
#pragma unroll
            for (int t = 0; t < RT; ++t) v[t] = row0 + lane + 32 * t == k ? T(1) : xk[lane + 32 * t] * inv;
            T ms[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int j = warp + NW * q;
                const T s = fmat(inv, S.sd[j], S.sr[j]);
                ms[q] = (j > k && j < b) ? -tau * s : T(0);
                if (lastc && lane == 0 && j < k) S.gs[j] = s;
            }
            if (warp == k % NW) {
                // column k itself.  (tau = 0: it is zero below row k, or far below the
                // rounding errors of the panel's other entries and dropped here)
                const unsigned pick = 1u << (k / NW);
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if ((pick >> q) & 1) {
#pragma unroll
                        for (int t = 0; t < RT; ++t) {
                            const int g = row0 + lane + 32 * t;
                            a[q][t] = g > k ? v[t] : (g == k && tau != T(0) ? beta : a[q][t]);
                        }
                    }
            }
            if (tau != T(0)) {
                if constexpr (sizeof(T) == 4) {
#pragma unroll
                    for (int t = 0; t < RT; ++t) {
                        const float2 vv = make_float2(v[t], v[t]);
#pragma unroll
                        for (int p = 0; p < Q / 2; ++p) {
                            const float2 r = ffma2(make_float2(ms[2 * p], ms[2 * p + 1]), vv,
                                                   make_float2(a[2 * p][t], a[2 * p + 1][t]));
                            a[2 * p][t] = r.x;
                            a[2 * p + 1][t] = r.y;
                        }
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < Q; ++q)
#pragma unroll
                        for (int t = 0; t < RT; ++t) a[q][t] = fmat(ms[q], v[t], a[q][t]);
                }
            }
            const int k1 = k + 1;
            if (k1 < nref && k1 % NW == warp) {
                T *xn = S.xs[k1 & 1];
                const unsigned pick = 1u << (k1 / NW);
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if ((pick >> q) & 1) {
#pragma unroll
                        for (int t = 0; t < RT; ++t)
                            xn[lane + 32 * t] = row0 + lane + 32 * t > k1 ? a[q][t] : T(0);
                    }
            }
        } else if (lastc && k >= 1) {
            coop_t_column<T, NW>(b, k - 1, Ts, S.tau, S.part);
        }
        __syncthreads();
    }
    // no CTA leaves while a peer may still store into its shared memory
    if constexpr (CL) {
        __syncwarp();
        coop_cluster_sync();
    }
    if (!alive) return;  // the error is latched; nothing was written
    // ---- the last column of T, then the results
    if (lastc) {
        if (nref > 0) {
            if (warp < NW) coop_t_partial<T, NW>(b, nref - 1, Ts, S.gs, S.part);
            __syncthreads();
            if (warp == NW) coop_t_column<T, NW>(b, nref - 1, Ts, S.tau, S.part);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < b * b; i += blockDim.x) Tm[i] = Ts[i];
    }
    if (warp < NW) {
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int t = 0; t < RT; ++t) {
                const int j = warp + NW * q, r = lane + 32 * t, g = row0 + r;
                if (j >= b || r >= rows) continue;
                T v = T(0);
                if (j < nref) v = g < j ? T(0) : (g == j ? T(1) : a[q][t]);
                U[(size_t)g + (size_t)j * N] = v;
                P[(size_t)g + (size_t)j * ldp] = g <= j ? a[q][t] * unscale : T(0);
            }
    }
}

// -------------------------------------------------------------------- host
// CTAs the exchange buffer in global memory has room for (one per SM, even).
static int coop_cmax(const sev_ctx *h) { return (h->sm_count + 2) / 2 * 2; }
constexpr int kCoopClMax = 16;  // CTAs of the largest cluster

template <typename T>
size_t panel_coop_words(const sev_ctx *h, int b) {
    return CoopComm<T>::words(b, coop_cmax(h));
}

// Rows per CTA (in units of 32) on the whole GPU: the fewest for which the CTAs
// stay a moderate number -- more rows mean more arithmetic per CTA and column,
// more CTAs mean more shares to read.  Over 64 columns (16 column warps, 96
// registers a thread) 256 rows do not fit the registers: 128 rows as long as the
// GPU has the CTAs (n = 16384, b = 128: 70.9 ms of panels per reduction against
// 82.4).  0: the panel does not fit the GPU.
template <typename T>
static int coop_rt(const sev_ctx *h, int N, bool wide) {
    if (wide && N <= 128 * h->sm_count) return 4;
    const int sizes[3] = {2, 4, 8}, room[3] = {sizeof(T) == 4 ? 0 : 96, sizeof(T) == 4 ? 32 : 128, h->sm_count};
    for (int i = 0; i < 3; ++i) {
        const int C = (N + 32 * sizes[i] - 1) / (32 * sizes[i]);
        if (C <= room[i] && C <= h->sm_count) return sizes[i];
    }
    return 0;
}

// The same on one cluster, whose CTAs exchange through shared memory (N = 2048,
// b = 64: 129 us a panel against 165 through L2); 0: not there.  FP64 keeps few rows per
// CTA (its FP64 pipes bound the column, not the exchange).  Over 64 columns 128
// rows per CTA here too, and taller panels on the whole GPU (70.9 -> 65.9 ms).
template <typename T>
static int coop_cl_rt(int N, bool wide) {
    if (wide) return N <= 128 * kCoopClMax ? 4 : 0;
    if (sizeof(T) == 8) return N <= 64 * kCoopClMax ? 2 : 0;
    return N <= 128 * 8 ? 4 : (N <= 256 * kCoopClMax ? 8 : 0);
}

template <typename T>
int panel_coop_supported(const sev_ctx *h, int N, int b) {
    if (h->leaf_rows_override > 0) return 0;  // the caller asked for a tree of that leaf size
    return b >= 1 && b <= (sizeof(T) == 4 ? 128 : 64) && coop_rt<T>(h, N, b > 64) > 0;
}

template <typename T, int RT>
static size_t coop_smem(int b) {
    return ((sizeof(CoopSmem<T, RT>) + 15) & ~(size_t)15) + sizeof(T) * (size_t)((b * b + 3) & ~3);
}

template <typename T, int RT, int Q, int NW>
static int panel_coop_run(sev_ctx *h, int N, int b, T *P, int lda, T *U, T *Tm, unsigned long long *comm, unsigned tag0) {
    const size_t smem = coop_smem<T, RT>(b);
    auto kern = panel_coop_kernel<T, RT, Q, NW, false>;
    SEV_CUDA(allow_smem(h, (const void *)kern));
    const int C = (N + 32 * RT - 1) / (32 * RT);
    int cmax = coop_cmax(h);
    void *args[] = {(void *)&P,    (void *)&lda,  (void *)&N,    (void *)&b,   (void *)&U,
                    (void *)&Tm,   (void *)&comm, (void *)&cmax, (void *)&tag0, (void *)&h->d_err};
    timing_begin(h, K_PANEL_COOP);
    SEV_CUDA(cudaLaunchCooperativeKernel((const void *)kern, C, (NW + 1) * 32, args, smem, h->stream));
    timing_end(h, K_PANEL_COOP);
    return SEV_OK;
}

// Index of a cluster instance (what the kernel needs of an SM differs among them).
template <typename T, int RT, int Q, int NW>
constexpr int coop_cl_index() {
    constexpr int i = sizeof(T) == 8 ? (Q == 8 ? 1 : 0) : (NW == 16 ? 6 : 2 + (RT == 8 ? 2 : 0) + (Q == 8 ? 1 : 0));
    static_assert(i < kPanelClKernels && (sizeof(T) == 8 ? RT == 2 && NW == 8 : RT == 4 || (RT == 8 && NW == 8)) &&
                      (Q == 4 || Q == 8) && (NW == 8 || Q == 8),
                  "one index per instance");
    return i;
}

// One cluster of C CTAs; SEV_ERR_UNSUPPORTED where the GPU cannot hold it.
template <typename T, int RT, int Q, int NW>
static int panel_coop_run_cl(sev_ctx *h, int N, int b, T *P, int lda, T *U, T *Tm) {
    const int C = (N + 32 * RT - 1) / (32 * RT), cmax = (C + 2) / 2 * 2;
    const size_t smem = coop_smem<T, RT>(b) + 8 * CoopComm<T>::words(b, cmax);
    if (smem > h->smem_optin) return SEV_ERR_UNSUPPORTED;
    auto kern = panel_coop_kernel<T, RT, Q, NW, true>;
    SEV_CUDA(allow_smem(h, (const void *)kern));
    SEV_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3((NW + 1) * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = h->stream;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (C > 8) {
        // clusters of more than 8 CTAs depend on the GPU's layout: asked once per
        // handle, kernel and size, for the kernel's widest panel
        signed char &ok = h->cluster_ok[coop_cl_index<T, RT, Q, NW>()][C];
        if (ok == 0) {
            int fit = 0;
            cfg.dynamicSmemBytes = coop_smem<T, RT>(Q * NW) + 8 * CoopComm<T>::words(Q * NW, cmax);
            ok = cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) == cudaSuccess && fit > 0 ? 1 : -1;
            cudaGetLastError();
            cfg.dynamicSmemBytes = smem;
        }
        if (ok < 0) return SEV_ERR_UNSUPPORTED;
    }
    timing_begin(h, K_PANEL_COOP);
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, kern, P, lda, N, b, U, Tm, (unsigned long long *)nullptr, cmax, 0u, h->d_err);
    timing_end(h, K_PANEL_COOP);
    if (e != cudaSuccess) {  // the whole-GPU kernel serves the panel (or meets the same error)
        cudaGetLastError();
        return SEV_ERR_UNSUPPORTED;
    }
    return SEV_OK;
}

template <typename T, int Q, int NW>
static int panel_coop_rt(sev_ctx *h, int N, int b, T *P, int lda, T *U, T *Tm, unsigned long long *comm, unsigned tag0) {
    constexpr bool wide = NW == 16;
    int rc = SEV_ERR_UNSUPPORTED;
    if constexpr (sizeof(T) == 8) {
        if (coop_cl_rt<T>(N, wide) == 2) rc = panel_coop_run_cl<T, 2, Q, NW>(h, N, b, P, lda, U, Tm);
    } else {
        if (coop_cl_rt<T>(N, wide) == 4) rc = panel_coop_run_cl<T, 4, Q, NW>(h, N, b, P, lda, U, Tm);
        if constexpr (!wide) {
            if (coop_cl_rt<T>(N, wide) == 8) rc = panel_coop_run_cl<T, 8, Q, NW>(h, N, b, P, lda, U, Tm);
        }
    }
    if (rc != SEV_ERR_UNSUPPORTED) return rc;
    switch (coop_rt<T>(h, N, wide)) {
        case 2:
            if constexpr (sizeof(T) == 8) return panel_coop_run<T, 2, Q, NW>(h, N, b, P, lda, U, Tm, comm, tag0);
            return SEV_ERR_UNSUPPORTED;
        case 4: return panel_coop_run<T, 4, Q, NW>(h, N, b, P, lda, U, Tm, comm, tag0);
        case 8: return panel_coop_run<T, 8, Q, NW>(h, N, b, P, lda, U, Tm, comm, tag0);
        default: return SEV_ERR_UNSUPPORTED;
    }
}

template <typename T>
int panel_coop_factor(sev_ctx *h, int N, int b, T *P, int lda, T *U, T *Tm, unsigned long long *comm, unsigned tag0) {
    if (b <= 32) return panel_coop_rt<T, 4, 8>(h, N, b, P, lda, U, Tm, comm, tag0);
    if (b <= 64) return panel_coop_rt<T, 8, 8>(h, N, b, P, lda, U, Tm, comm, tag0);
    if constexpr (sizeof(T) == 4) return panel_coop_rt<T, 8, 16>(h, N, b, P, lda, U, Tm, comm, tag0);
    return SEV_ERR_UNSUPPORTED;
}

template size_t panel_coop_words<float>(const sev_ctx *, int);
template size_t panel_coop_words<double>(const sev_ctx *, int);
template int panel_coop_supported<float>(const sev_ctx *, int, int);
template int panel_coop_supported<double>(const sev_ctx *, int, int);
template int panel_coop_factor<float>(sev_ctx *, int, int, float *, int, float *, float *, unsigned long long *, unsigned);
template int panel_coop_factor<double>(sev_ctx *, int, int, double *, int, double *, double *, unsigned long long *,
                                       unsigned);

}  // namespace sev
