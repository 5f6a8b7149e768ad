// ols_post.cu -- the fused OLS kernel with post-processing of the convolved
// output inside the kernel, before anything is written (Sec. 3.2: OLS's
// "optional post-processing" step; Sec. 4.3: per-element and non-local
// post-processing; Sec. 4.4: reducing the output before it leaves the GPU).
//
// Four epilogues of the bank kernel (ols_bank.cuh: the segment's spectrum kept in
// tensor memory for all filters; per filter the point-wise product, the inverse
// FFT and the discard of aliased samples):
// * POWER   (per element)   p_f[j] = |y_f[j]|^2, written as FP32 (half the
//   output bytes of y);
// * DETECT  (per element + selection) the candidates (f, j) whose power
//   reaches a threshold, appended to a caller list through one atomic per
//   warp and store step (warp-aggregated), nothing else written;
// * DERIV   (non-local)     the numerical derivative of y along j: central
//   differences (y[j+1] - y[j-1]) / 2 inside, one-sided differences at j = 0
//   and j = Nout-1.  Each segment advances by L-2 instead of L and starts one
//   output early, so every derivative it writes has both neighbours among
//   its own unaliased samples (the "immediate neighbourhood" of Sec. 4.3).
//   Inside the stream the difference is taken on the segment's spectrum; the
//   segments at its two ends exchange neighbours through shared memory.
// * PEAK    (non-local + selection) the peaks of the power (Sec. 4.4's peak
//   finding): (f, j) whose power reaches the threshold, is above the power of
//   j - 1 and at least that of j + 1 (no neighbour at the two ends of the
//   stream), appended like DETECT; segments laid out like DERIV.  Candidates
//   are rare, so a warp fetches neighbour powers (warp shuffles) only when
//   one of its lanes reaches the threshold; in segments of several warps each
//   warp's first and last thread also publish their 16 powers in a small
//   shared buffer for the neighbouring warps.
#include <cuda_runtime.h>
#include <cstdint>

#include "ols_bank.cuh"
#include "ols_internal.h"

namespace ols {

// Thread and register that hold sample n of a segment in the time domain (the inverse of
// Geo<>::base and off).
template <class G>
__device__ __forceinline__ int thread_of(int n) {
    return G::N == 8192 ? ((n >> 11) & 1) * 256 + (n & 255) : n % G::T;
}
template <class G>
__device__ __forceinline__ int reg_of(int n) {
    return G::N == 8192 ? ((n >> 8) & 7) + 8 * (n >> 12) : n / G::T;
}

// The peak test of one output with a candidate power pk (called by whole warps,
// only when some lane has a candidate: it stays out of the common path's
// register allocation).  Neighbours n - 1 and n + 1 of output n = k T + t are
// register k of threads t - 1 and t + 1: rotating shuffles within the W
// threads of the segment in a warp, whose wrap-around carries `up` (register
// k - 1 of thread T - 1, for thread 0) and `dn` (register k + 1 of thread 0,
// for thread T - 1); in segments of several warps, the threads at a warp's
// edge read the neighbouring warp's powers from `edge` instead.
template <int T>
__device__ __noinline__ bool peak_test(bool hit, float pk, float up, float dn, int t, int k, bool first, bool last,
                                       const float *edge) {
    constexpr int W = T < 32 ? T : 32;
    const int gl = t % W;
    float prv = __shfl_sync(0xffffffffu, up, gl == 0 ? W - 1 : gl - 1, W);
    float nxt = __shfl_sync(0xffffffffu, dn, gl == W - 1 ? 0 : gl + 1, W);
    if constexpr (T > 32) {
        constexpr int nw = T / 32;
        using G = Geo<(T == 512 ? 13 : T == 256 ? 12 : T == 128 ? 11 : 10)>;
        const int n = G::base(t) + G::off(k);
        if (gl == 0) {
            const int m = n > 0 ? n - 1 : 0;
            prv = edge[(nw + thread_of<G>(m) / 32) * 16 + reg_of<G>(m)];
        }
        if (gl == W - 1) {
            const int m = n < G::N - 1 ? n + 1 : n;
            nxt = edge[thread_of<G>(m) / 32 * 16 + reg_of<G>(m)];
        }
    }
    if (hit && !first) hit = pk > prv;
    if (hit && !last) hit = pk >= nxt;
    return hit;
}

// Append candidate (j, f, power) for every lane with `hit`: one atomic per
// warp (warp-aggregated); records past `cap` are dropped, the count is kept.
__device__ __forceinline__ void append_candidates(bool hit, long long j, int f, float pw, ols_candidate *cand,
                                                  unsigned long long *count, long long cap, long long Nout,
                                                  int *status) {
    const unsigned lane = threadIdx.x & 31u;
    const unsigned mask = __ballot_sync(0xffffffffu, hit);
    if (mask) {
        unsigned long long base = 0;
        const unsigned leader = __ffs(mask) - 1;
        if (lane == leader) base = atomicAdd(count, (unsigned long long)__popc(mask));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (hit) {
            const unsigned long long i = base + __popc(mask & ((1u << lane) - 1u));
            if (i < (unsigned long long)cap && in_bounds(j < Nout, status)) {
                ols_candidate c;
                c.j = j;
                c.f = f;
                c.power = pw;
                cand[i] = c;
            }
        }
        __syncwarp();       // the next filter's tensor-memory load is warp-wide
    }
}

// DERIV, a segment at an end of the stream (called by its own threads): y in
// circular order to the exchange buffer `buf`, padded q -> q + q/16; then each
// output reads its two neighbours, the one-sided ends at j = 0 and j = Nout - 1.
// drow: the filter's row of d.
template <int LOG2N, class BAR>
__device__ __forceinline__ void derivative_exchange(const float2 *x, float2 *drow, float2 *buf, int t,
                                                    const BankSegment &sg, const BAR &bar) {
    using G = Geo<LOG2N>;
    if constexpr (LOG2N == 13) bar();             // the buffers of both halves, free between two barriers
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int n = G::base(t) + G::off(k);
        buf[n + (n >> 4)] = x[k];
    }
    bar();
    float2 *dst = drow + (sg.j0 - sg.n0);
    // circular positions of outputs j = 0 and j = Nout-1, if in this segment
    const int n_first = sg.j0 == 0 ? sg.n0 : -2;
    const int n_last = (sg.Nout - sg.j0 == (long long)sg.span) ? sg.span - 1 + sg.n0 : -2;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int n = G::base(t) + G::off(k);
        if ((unsigned)(n - sg.n0) < (unsigned)sg.span &&
            in_bounds(sg.j0 - sg.n0 + n < sg.Nout && n >= 1 && n + 1 < G::N, sg.status)) {
            const int lo = (n == n_first) ? n : n - 1;
            const int hi = (n == n_last) ? n : n + 1;
            const float sc = (lo == n || hi == n) ? 1.f : 0.5f;
            const float2 a = buf[lo + (lo >> 4)], b = buf[hi + (hi >> 4)];
            __stcs(dst + n, make_float2((b.x - a.x) * sc, (b.y - a.y) * sc));
        }
    }
    if constexpr (LOG2N == 13) bar();
}
// The same as a call, which takes the two end segments' code and registers out of
// the loop that all others run: at N = 512 .. 2048 the loop spills 90 to 110 bytes with
// the code inline and nothing with the call (16 filters, 2^22 samples, N = 1024: 141
// -> 132 us; 3 filters, 300,000 samples, N = 512 / 1024 / 2048: 9.4 / 9.9 / 9.8 -> 8.4 / 8.7 / 9.6).
// At N = 256, 4096 and 8192 the call was slower (8 filters, 2e6 samples: 35.5 -> 36.1, 51.9 ->
// 55.2, 75.2 -> 81.7).
template <int LOG2N, class BAR>
__device__ __noinline__ void derivative_exchange_call(const float2 *x, float2 *drow, float2 *buf, int t, BankSegment sg,
                                                      BAR bar) {
    derivative_exchange<LOG2N>(x, drow, buf, t, sg, bar);
}

template <int MODE>
struct EpiPost {
    static constexpr bool WIDE = MODE == POST_POWER || MODE == POST_DETECT;
    // two loads of twiddles where one spills
    template <int LOG2N>
    static constexpr bool narrow() {
        return (MODE == POST_DERIV && LOG2N >= 10) || (MODE == POST_PEAK && LOG2N == 12);
    }
    // one of the exchange's three bits by shuffles (as the real form)
    static constexpr int XCH = WIDE ? XCHG_SHFL : XCHG_TMEM;
    // PEAK: warp-edge powers [2][T/32][16] floats per segment of several warps
    template <int LOG2N>
    static constexpr int edge() {
        return (MODE == POST_PEAK && Geo<LOG2N>::T > 32) ? (Geo<LOG2N>::T / 32) * 16 : 0;
    }
    const float2 *sig;
    void *out;                      // POWER: float [F][Nout]; DERIV: float2 [F][Nout]
    float thr;
    ols_candidate *cand;
    unsigned long long *count;
    long long cap;
    const float *dsin;              // DERIV: sin(2 pi nu / N) at each storage position, then its rounding errors
    __device__ __forceinline__ float2 sample(long long i) const { return __ldg(sig + i); }
    // DERIV: central differences of a circular sequence are the product of its
    // spectrum with i sin(2 pi nu / N).  The segment's spectrum is scaled once
    // for all its filters, so the inverse FFT yields the derivative itself and
    // no output needs its neighbours.  A segment holding the first or the last
    // output of the stream, whose differences are one-sided, keeps its plain
// spectrum and goes through the neighbour exchange below.  Device time of the
    // exchange for every segment (one CTA of 128 threads per segment group, one fewer per SM
    // for its registers) and of this, 16 filters: N = 1024, 2^22 samples 210 -> 125 us; N = 2048,
    // 2^23 samples 402 -> 286.
    __device__ __forceinline__ static bool at_end(const BankSegment &sg) {
        return sg.j0 == 0 || sg.Nout - sg.j0 == (long long)sg.span;
    }
    template <int LOG2N>
    __device__ __forceinline__ void spectrum(float2 *X, int t, const BankSegment &sg) const {
        if constexpr (MODE == POST_DERIV) {
            if (!at_end(sg)) {
                const float4 *p = reinterpret_cast<const float4 *>(dsin) + 4 * t;
                auto scale = [](float2 &x, float s, float r) {
                    x = make_float2(fmaf(-s, x.y, -r * x.y), fmaf(s, x.x, r * x.x));
                };
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 s = __ldg(p + q), r = __ldg(p + q + Geo<LOG2N>::N / 4);
                    scale(X[4 * q], s.x, r.x);
                    scale(X[4 * q + 1], s.y, r.y);
                    scale(X[4 * q + 2], s.z, r.z);
                    scale(X[4 * q + 3], s.w, r.w);
                }
            }
        }
    }
    template <int LOG2N, class BAR>
    __device__ __forceinline__ void store(const float2 *x, int f, int t, const BankSegment &sg, float2 *bufs, int &xc,
                                          const BAR &bar) const {
        using G = Geo<LOG2N>;
        const int v = G::base(t) - sg.n0;             // output v + off(k) of the segment in register k
        if constexpr (MODE == POST_POWER) {
            float *dst = static_cast<float *>(out) + (size_t)f * (size_t)sg.Nout + (sg.j0 + v);
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if ((unsigned)(v + G::off(k)) < (unsigned)sg.span && in_bounds(sg.j0 + v + G::off(k) < sg.Nout, sg.status))
                    __stcs(dst + G::off(k), fmaf(x[k].x, x[k].x, x[k].y * x[k].y));
        } else if constexpr (MODE == POST_DETECT) {
            // candidates are rare: one vote decides whether the warp has any at all
            float pw[16];
            bool any = false;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                pw[k] = fmaf(x[k].x, x[k].x, x[k].y * x[k].y);
                any |= (unsigned)(v + G::off(k)) < (unsigned)sg.span && pw[k] >= thr;
            }
            if (__any_sync(0xffffffffu, any)) {
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const bool hit = (unsigned)(v + G::off(k)) < (unsigned)sg.span && pw[k] >= thr;
                    append_candidates(hit, sg.j0 + (v + G::off(k)), f, pw[k], cand, count, cap, sg.Nout, sg.status);
                }
            }
        } else if constexpr (MODE == POST_PEAK) {
            constexpr int W = G::T < 32 ? G::T : 32;          // threads of the segment in one warp
            const int gl = t % W;
            float pw[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) pw[k] = fmaf(x[k].x, x[k].x, x[k].y * x[k].y);
            // segments of several warps: first[w][k] at edge[w * 16 + k], last[w][k] after them
            float *ed = reinterpret_cast<float *>(bufs + G::XBUFS * G::PADN);
            if constexpr (edge<LOG2N>() > 0) {
                if (gl == 0 || gl == W - 1) {
                    float4 *e = reinterpret_cast<float4 *>(ed + ((gl == 0 ? 0 : G::T / 32) + t / 32) * 16);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        e[q] = make_float4(pw[4 * q], pw[4 * q + 1], pw[4 * q + 2], pw[4 * q + 3]);
                }
                bar();
            }
            // first and last output of the stream (one neighbour only), if in this segment
            const long long rem = sg.Nout - sg.j0;
            const int k_first = sg.j0 == 0 ? 0 : -2;
            const int k_last = (sg.span > 0 && rem == (long long)sg.span) ? sg.span - 1 : -2;
            bool any = false;
#pragma unroll
            for (int k = 0; k < 16; ++k) any |= (unsigned)(v + G::off(k)) < (unsigned)sg.span && pw[k] >= thr;
            if (!__any_sync(0xffffffffu, any)) return;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int o = v + G::off(k);
                bool hit = (unsigned)o < (unsigned)sg.span && pw[k] >= thr &&
                           in_bounds(o + sg.n0 >= 1 && o + sg.n0 + 1 < G::N, sg.status);
                if (__any_sync(0xffffffffu, hit))
                    hit = peak_test<G::T>(hit, pw[k], (gl == W - 1) ? pw[k > 0 ? k - 1 : 0] : pw[k],
                                          (gl == 0) ? pw[k < 15 ? k + 1 : 15] : pw[k], t, k, o == k_first,
                                          o == k_last, ed);
                append_candidates(hit, sg.j0 + o, f, pw[k], cand, count, cap, sg.Nout, sg.status);
            }
        } else if (!at_end(sg)) {
            float2 *dst = static_cast<float2 *>(out) + (size_t)f * (size_t)sg.Nout + (sg.j0 + v);
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if ((unsigned)(v + G::off(k)) < (unsigned)sg.span && in_bounds(sg.j0 + v + G::off(k) < sg.Nout, sg.status))
                    __stcs(dst + G::off(k), x[k]);
        } else {
            float2 *drow = static_cast<float2 *>(out) + (size_t)f * (size_t)sg.Nout;
            float2 *buf = LOG2N == 13 ? bufs : bufs + (xc & 1) * G::PADN;      // not in use
            if constexpr (LOG2N != 13) ++xc;
            if constexpr (LOG2N >= 9 && LOG2N <= 11) {
                float2 y[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) y[k] = x[k];
                derivative_exchange_call<LOG2N>(y, drow, buf, t, sg, bar);
            } else {
                derivative_exchange<LOG2N>(x, drow, buf, t, sg, bar);
            }
        }
    }
};

cudaError_t post_prepare(ols_plan_s &p) {
    cudaError_t e = bank_prepare_any<EpiPost<POST_POWER>>(p.log2N);
    if (e == cudaSuccess) e = bank_prepare_any<EpiPost<POST_DETECT>>(p.log2N);
    if (e == cudaSuccess) e = bank_prepare_any<EpiPost<POST_DERIV>>(p.log2N);
    if (e == cudaSuccess) e = bank_prepare_any<EpiPost<POST_PEAK>>(p.log2N);
    return e;
}

template <int MODE>
static cudaError_t post_launch_mode(const ols_plan_s &p, const PostArgs &a, cudaStream_t st) {
    // derivative and peaks read the neighbours j - 1 and j + 1 of an output:
    // their segments start one sample early
    constexpr bool NEIGH = MODE == POST_DERIV || MODE == POST_PEAK;
    BankArgs b{};
    b.Hk = reinterpret_cast<const float4 *>(p.Hk);
    b.tw = p.twb;
    b.F = p.F;
    b.n0 = NEIGH ? p.M : p.M - 1;
    b.step = a.step;
    b.off = NEIGH ? -1 : 0;
    b.Ns = a.Ns;
    b.Nout = a.Nout;
    b.nseg = a.nseg;
    b.status = p.d_status;
    return bank_launch_any(p.log2N, b, EpiPost<MODE>{a.s, a.out, a.thr, a.cand, a.count, (long long)a.cap, p.dsin}, p.sm_count,
                           st);
}

cudaError_t post_launch(const ols_plan_s &p, const PostArgs &a, cudaStream_t st) {
    switch (a.mode) {
        case POST_POWER: return post_launch_mode<POST_POWER>(p, a, st);
        case POST_DETECT: return post_launch_mode<POST_DETECT>(p, a, st);
        case POST_DERIV: return post_launch_mode<POST_DERIV>(p, a, st);
        case POST_PEAK: return post_launch_mode<POST_PEAK>(p, a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ols
