// ols_bank.cuh -- the fused overlap-and-save kernel of a filter bank
// (Algorithm 2 / Sec. 3.4), shared by the plain, real-to-real and
// post-processing forms: one kernel; a segment's forward FFT is done on chip
// and its spectrum kept there, then for every filter: point-wise product with
// the filter's precomputed spectrum, inverse FFT, removal of the aliased
// samples and the form's epilogue (Sec. 3.2).
//
// * Each thread holds 16 points of a segment; a CTA of BLOCK threads holds
//   BLOCK / (N/16) segments in slots that exchange under barriers of their
//   own.  What bounds it: FP32 issue and the latency of the exchanges
//   between the passes, with the 16 resident warps that 128 registers allow;
//   no unit is saturated (filter bank, N = 2048: issue 64% and FMA pipe 57% of cycles, L1
//   data path 48%; 521 us against an HBM floor of 326).
// * Spectra of filter f + 1 are loaded into registers while filter f is
//   transformed.  The slots of a CTA run through the filters side by side, so
//   those loads hit L1 for most of them: one CTA of 512 threads per SM instead
//   of four of 128 took L1 hits from 11% to 35% of sectors and L2 reads down
//   by 31%.  (Spectra copied to shared memory by bulk copies and read from
//   there at the head of each filter, without registers held, were 17% slower;
//   the load latency is then exposed 32 times per segment.)
// * Work is shared out in steps (block of segments, filter): the grid is at
//   most the resident CTAs, each takes the same number of consecutive steps
//   (give or take one) and transforms a segment again where its share begins
//   inside one.  A long signal has no partly filled last wave; a short one
//   (37 segments of 32 filters: 37 busy CTAs of 608 with a segment each)
//   fills the chip.
// * Output stores carry the streaming hint, so that they do not push the
//   spectra out of L1 (2% on the filter bank).
// Device time (us) before (a CTA of 128 threads per segment group, all filters of it)
// and after, plain form, 32 filters of 2^22 samples: N = 256 (3e6 samples) 166 -> 142, 512
// 253 -> 208, 1024 257 -> 212, 2048 279 -> 262, 4096 333 -> 285, 8192 (24 filters) 340 -> 312;
// 65521 samples of 32 filters at N = 2048: 33 -> 10.
#pragma once

#include <cstdint>

#include "ols_fft_passes.cuh"
#include "ols_internal.h"
#include "tmem.cuh"

namespace ols {

template <int LOG2N, int BLOCK, class EPI>
struct BankGeo {
    using G = Geo<LOG2N>;
    static constexpr int SL = BLOCK / G::T;                 // segments in flight per CTA
    static_assert(SL >= 1 && (SL <= 15 || G::T <= 32), "one named barrier per slot");
    static constexpr int MINB = 512 / BLOCK;                // resident CTAs per SM: 16 warps, all tensor memory
    static constexpr uint32_t TMEM_COLS = (uint32_t)(BLOCK / 128) * 128u;
    static constexpr int SLOT = G::XBUFS * G::PADN + EPI::template edge<LOG2N>();   // float2 per slot
    static constexpr size_t USED = sizeof(float2) * (size_t)(SL * SLOT);
    // requested: enough that no more CTAs fit on an SM (228 KB) than tensor
    // memory can serve, so a CTA's tcgen05.alloc never waits
    static constexpr size_t CLAIM = (228u * 1024u) / (MINB + 1) + 1024u;
    static constexpr size_t SMEM = USED > CLAIM ? USED : CLAIM;
};

struct BankArgs {
    const float4 *Hk;       // [F][N] spectra in kernel layout
    const float2 *tw;       // twiddles (N = 8192: of N = 4096)
    int F;                  // spectra per segment
    int n0;                 // circular position of a segment's first output
    long long step;         // outputs per segment
    long long off;          // first input sample of segment 0
    long long Ns, Nout, nseg;
    long long total;        // steps: blocks of SL segments x F
    int *status;
};

// What an epilogue sees of its segment.
struct BankSegment {
    long long j0;           // first output
    int span;               // outputs of this segment (0: idle slot)
    int n0;
    long long Nout;
    int *status;
};

// y[f][j] written once, the aliased samples dropped.
struct EpiPlain {
    static constexpr bool WIDE = true;      // 512-thread CTAs at N = 4096 (see bank_launch)
    template <int LOG2N>
    static constexpr bool narrow() { return false; }
    static constexpr int XCH = XCHG_TMEM;
    template <int LOG2N>
    static constexpr int edge() { return 0; }
    const float2 *sig;
    float2 *y;
    __device__ __forceinline__ float2 sample(long long i) const { return __ldg(sig + i); }
    template <int LOG2N>
    __device__ __forceinline__ void spectrum(float2 *, int, const BankSegment &) const {}
    template <int LOG2N, class BAR>
    __device__ __forceinline__ void store(const float2 *x, int f, int t, const BankSegment &sg, float2 *, int &,
                                          const BAR &) const {
        using G = Geo<LOG2N>;
        const int v = G::base(t) - sg.n0;                 // output v + off(k) of the segment in register k
        float2 *dst = y + (size_t)f * (size_t)sg.Nout + (sg.j0 + v);
        if (sg.span == G::N - sg.n0) {           // a full segment: only the aliased samples are dropped
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if (v >= -G::off(k) && in_bounds(sg.j0 + v + G::off(k) < sg.Nout, sg.status)) __stcs(dst + G::off(k), x[k]);
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if ((unsigned)(v + G::off(k)) < (unsigned)sg.span && in_bounds(sg.j0 + v + G::off(k) < sg.Nout, sg.status))
                    __stcs(dst + G::off(k), x[k]);
        }
    }
};

// A segment's filters f .. fend - 1 of F, its spectrum in the thread's tensor-memory
// lane and filter f's in h: product, inverse FFT, epilogue (the loop of the bank
// and of the batch kernels).  At N = 256 a warp holds two segments, whose epilogues
// may take different branches (a full segment beside a ragged or idle one), while
// the tensor-memory accesses of the next filter, or of the next segment, are
// warp-wide: the warp meets again after each epilogue.
template <int LOG2N, class EPI, class TW, class LOADH, class BAR>
__device__ __forceinline__ void segment_filters(const EPI &epi, const TW &tw, float4 *h, const LOADH &load_h, int f,
                                                int fend, int F, const BankSegment &sg, float2 *bufs, int t, int &xc,
                                                const BAR &bar) {
    using G = Geo<LOG2N>;
    for (; f < fend; ++f) {
        float2 x[16];
        tmem::ld32(tw.base + 96, reinterpret_cast<float *>(x));
        tmem::wait_ld();
#pragma unroll
        for (int j2 = 0; j2 < 8; ++j2) {
            x[2 * j2] = cmul(x[2 * j2], make_float2(h[j2].x, h[j2].y));
            x[2 * j2 + 1] = cmul(x[2 * j2 + 1], make_float2(h[j2].z, h[j2].w));
        }
        load_h(f + 1 == F ? 0 : f + 1);          // of this segment, or the first of the next
        inverse_passes<LOG2N, G::NP - 1>(x, bufs, tw, t, xc, bar);
        epi.template store<LOG2N>(x, f, t, sg, bufs, xc, bar);
        if constexpr (G::T < 32) __syncwarp();
    }
}

template <int LOG2N, int BLOCK, class EPI>
__global__ void __launch_bounds__(BLOCK, (BankGeo<LOG2N, BLOCK, EPI>::MINB))
ols_bank_kernel(const BankArgs a, const EPI epi) {
    using G = Geo<LOG2N>;
    using BG = BankGeo<LOG2N, BLOCK, EPI>;
    extern __shared__ float4 smem_raw[];
    __shared__ uint32_t tbase;
    const int slot = threadIdx.x / G::T;
    const int t = threadIdx.x % G::T;
    float2 *bufs = reinterpret_cast<float2 *>(smem_raw) + slot * BG::SLOT;
    const SegmentBarrier<G::T> bar{1 + slot};
    // tensor memory: per thread its twiddles (columns 0..95) and, from column
    // 96 on, its 16 points of the segment's spectrum
    if (threadIdx.x < 32) tmem::alloc(&tbase, BG::TMEM_COLS);
    tmem::fence_before_sync();
    __syncthreads();
    tmem::fence_after_sync();
    const TwTmem<LOG2N, EPI::XCH, EPI::template narrow<LOG2N>()> tw{tbase + tmem::lane_bits() + (uint32_t)(threadIdx.x / 128) * 128u, tw_odd<LOG2N>(a.tw, t)};
    tw_tmem_fill<LOG2N, EPI::XCH>(a.tw, tw.base, t);
    const uint32_t xcol = tw.base + 96;

    // this CTA's share of the steps
    const long long each = a.total / gridDim.x, more = a.total % gridDim.x, b = blockIdx.x;
    const long long s0 = each * b + (b < more ? b : more);
    long long todo = each + (b < more ? 1 : 0);
    long long blk = s0 / a.F;
    int f = (int)(s0 - blk * a.F);
    float4 h[8];
    auto load_h = [&](int ff) {
        const float4 *hp = a.Hk + (size_t)ff * (G::N / 2) + t;
#pragma unroll
        for (int j2 = 0; j2 < 8; ++j2)
            if (in_bounds(ff < a.F, a.status)) h[j2] = load_spectrum(hp + j2 * G::T);
    };
    load_h(f);
    int xc = 0;
    for (; todo > 0; ++blk, f = 0) {
        const long long seg = blk * BG::SL + slot;
        const bool active = seg < a.nseg;
        BankSegment sg;
        sg.j0 = active ? seg * a.step : 0;
        const long long rem = active ? a.Nout - sg.j0 : 0;
        sg.span = (int)(rem < a.step ? rem : a.step);
        sg.n0 = a.n0;
        sg.Nout = a.Nout;
        sg.status = a.status;
        {
            // samples start + base(t) + off(k) inside [0, Ns), zero elsewhere
            float2 X[16];
            const long long start = sg.j0 + a.off;
            const long long avail = active ? a.Ns - start : 0;
            const int lim = (int)(avail < G::N ? avail : G::N);
            const int first = start < 0 ? (int)-start : 0;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int n = G::base(t) + G::off(k);
                X[k] = (n >= first && n < lim && in_bounds(start + n >= 0 && start + n < a.Ns, a.status))
                           ? epi.sample(start + n)
                           : make_float2(0.f, 0.f);
            }
            forward_passes<LOG2N, 0>(X, bufs, tw, t, xc, bar);
            epi.template spectrum<LOG2N>(X, t, sg);
            if constexpr (G::T < 32) __syncwarp();   // the warp's two segments may have branched apart
            tmem::st32(xcol, reinterpret_cast<const float *>(X));
            tmem::wait_st();
        }
        const int fend = a.F - f < todo ? a.F : f + (int)todo;
        todo -= fend - f;
        segment_filters<LOG2N>(epi, tw, h, load_h, f, fend, a.F, sg, bufs, t, xc, bar);
    }
    tmem::fence_before_sync();
    __syncthreads();
    tmem::fence_after_sync();
    if (threadIdx.x < 32) tmem::dealloc(tbase, BG::TMEM_COLS);
}

template <int LOG2N, int BLOCK, class EPI>
cudaError_t bank_prepare_block() {
    return cudaFuncSetAttribute(ols_bank_kernel<LOG2N, BLOCK, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)BankGeo<LOG2N, BLOCK, EPI>::SMEM);
}

template <int LOG2N, int BLOCK, class EPI>
cudaError_t bank_launch_block(BankArgs a, const EPI &epi, int sm_count, cudaStream_t st) {
    using BG = BankGeo<LOG2N, BLOCK, EPI>;
    a.total = (a.nseg + BG::SL - 1) / BG::SL * a.F;
    const long long cap = (long long)BG::MINB * sm_count;
    const int grid = (int)(a.total < cap ? a.total : cap);
    ols_bank_kernel<LOG2N, BLOCK, EPI><<<grid, BLOCK, BG::SMEM, st>>>(a, epi);
    return cudaGetLastError();
}

// Block size of a call.  One CTA of 512 threads per SM shares the spectra's L1
// lines among the most segments (32 filters, 2^21 samples, blocks of 512 / 256 / 128: N = 512
// 107 / 112 / 110 us, 1024 109 / 117 / 115, 2048 135 / 145 / 137; N = 256 93 / 92 / 93).  With fewer
// than four steps per SM two CTAs of 256 start and end sooner (32 filters, 2^15 samples: N = 256
// 7.0 / 6.4 us, 1024 8.9 / 7.7, 2048 10.1 / 8.7; from 2^17 samples on the two are within 2%).  While CTAs of
// 128 threads, four per SM, leave at most one step each, they set up sooner and reach
// more SMs (one filter, 2^16 samples, 256 / 128: N = 256 4.3 / 3.5 us, 512 5.0 / 3.9, 2048 5.4 / 4.3; 32 filters,
// 2^15 samples, N = 512 7.4 / 7.2, 2048 8.7 / 7.9).  At N = 4096 a 512-thread CTA holds only two
// segments: it pays from four spectra per segment on, and not for the derivative and
// the peaks, whose epilogues spill or stay longer at its barriers (2^22 samples, 512 / 256: 32 filters plain 284 /
// 310 us, power 282 / 301, derivative 357 / 335, peaks 320 / 315; 8 filters plain 84 / 89; 2 filters 32.5 / 31.6; one
// filter 23.6 / 21.8).  N = 8192 needs 512 threads for its one segment.
template <int LOG2N, class EPI>
cudaError_t bank_prepare() {
    cudaError_t e = bank_prepare_block<LOG2N, 512, EPI>();
    if constexpr (LOG2N != 13) {
        if (e == cudaSuccess) e = bank_prepare_block<LOG2N, 256, EPI>();
    }
    if constexpr (LOG2N < 12) {
        if (e == cudaSuccess) e = bank_prepare_block<LOG2N, 128, EPI>();
    }
    return e;
}
template <int LOG2N, class EPI>
cudaError_t bank_launch(const BankArgs &a, const EPI &epi, int sm_count, cudaStream_t st) {
    if constexpr (LOG2N == 13) {
        return bank_launch_block<LOG2N, 512>(a, epi, sm_count, st);
    } else {
        constexpr int SL = 512 / Geo<LOG2N>::T;
        const long long steps = (a.nseg + SL - 1) / SL * a.F;
        if constexpr (LOG2N == 12) {
            if (!EPI::WIDE || a.F < 4) return bank_launch_block<LOG2N, 256>(a, epi, sm_count, st);
        } else {
            constexpr int SL1 = 128 / Geo<LOG2N>::T;
            if ((a.nseg + SL1 - 1) / SL1 * a.F <= 4ll * sm_count)
                return bank_launch_block<LOG2N, 128>(a, epi, sm_count, st);
        }
        if (steps < 4ll * sm_count) return bank_launch_block<LOG2N, 256>(a, epi, sm_count, st);
        return bank_launch_block<LOG2N, 512>(a, epi, sm_count, st);
    }
}

// One form's kernels for every segment length.
template <class EPI>
cudaError_t bank_prepare_any(int log2N) {
    switch (log2N) {
        case 8: return bank_prepare<8, EPI>();
        case 9: return bank_prepare<9, EPI>();
        case 10: return bank_prepare<10, EPI>();
        case 11: return bank_prepare<11, EPI>();
        case 12: return bank_prepare<12, EPI>();
        case 13: return bank_prepare<13, EPI>();
        default: return cudaErrorInvalidValue;
    }
}
template <class EPI>
cudaError_t bank_launch_any(int log2N, const BankArgs &a, const EPI &epi, int sm_count, cudaStream_t st) {
    switch (log2N) {
        case 8: return bank_launch<8>(a, epi, sm_count, st);
        case 9: return bank_launch<9>(a, epi, sm_count, st);
        case 10: return bank_launch<10>(a, epi, sm_count, st);
        case 11: return bank_launch<11>(a, epi, sm_count, st);
        case 12: return bank_launch<12>(a, epi, sm_count, st);
        case 13: return bank_launch<13>(a, epi, sm_count, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ols
