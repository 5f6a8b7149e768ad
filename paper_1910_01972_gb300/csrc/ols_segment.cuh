// ols_segment.cuh -- one segment of Algorithm 2 for all filters of its problem,
// the batched kernels' body (the loop of ols_bank_kernel with the plain
// epilogue, so results are bitwise those of per-problem calls): load the
// segment (zero past Ns), forward FFT, spectrum into the thread's TMEM lane
// (columns 96..127), then for every filter the point-wise product with its
// spectrum (the next filter's in flight), inverse FFT, and store of the samples
// not aliased that fall inside the output.
#pragma once

#include "ols_bank.cuh"

namespace ols {

// BAR: the barrier of the segment's exchanges (the whole CTA, or only the
// segment's own threads).
template <int LOG2N, class TW, class BAR>
__device__ __forceinline__ void ols_segment(const BatchProblemDev &P, const float2 *__restrict__ sig,
                                            float2 *__restrict__ y, const TW &tw, long long seg, float2 *bufs, int t,
                                            int &xc, const BAR &bar) {
    using G = Geo<LOG2N>;
    const EpiPlain epi{sig, y};
    const bool active = seg < P.nseg;
    const int F = P.F;
    const float4 *Hk = P.Hk;
    BankSegment sg;
    sg.j0 = active ? seg * P.L : 0;
    const long long rem = active ? P.Nout - sg.j0 : 0;
    sg.span = (int)(rem < P.L ? rem : P.L);
    sg.n0 = P.M - 1;
    sg.Nout = P.Nout;
    sg.status = P.status;
    const uint32_t xcol = tw.base + 96;
    {
        float2 X[16];
        const long long avail = active ? P.Ns - sg.j0 : 0;
        const int lim = (int)(avail < G::N ? avail : G::N);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int n = G::base(t) + G::off(k);
            X[k] = (n < lim && in_bounds(sg.j0 + n < P.Ns, sg.status)) ? epi.sample(sg.j0 + n) : make_float2(0.f, 0.f);
        }
        forward_passes<LOG2N, 0>(X, bufs, tw, t, xc, bar);
        tmem::st32(xcol, reinterpret_cast<const float *>(X));
        tmem::wait_st();
    }
    float4 h[8];
    auto load_h = [&](int ff) {
        const float4 *hp = Hk + (size_t)ff * (G::N / 2) + t;
#pragma unroll
        for (int j2 = 0; j2 < 8; ++j2)
            if (in_bounds(ff < F, sg.status)) h[j2] = load_spectrum(hp + j2 * G::T);
    };
    load_h(0);
    segment_filters<LOG2N>(epi, tw, h, load_h, 0, F, F, sg, bufs, t, xc, bar);
}

}  // namespace ols
