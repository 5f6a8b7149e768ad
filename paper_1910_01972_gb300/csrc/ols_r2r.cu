// ols_r2r.cu -- the fused overlap-and-save convolution of a REAL signal with
// a bank of REAL filters (the paper's R2R variant, Sec. 3.4 and Algorithm 2).
//
// The paper runs its R2R kernel on half-length complex FFTs (Stockham
// autosort, with real-to-complex and complex-to-real post-processing).  Here
// the saving of the real data is taken along the filter axis instead, which
// keeps the reorder-free complex kernel of the C2C path:
// * filters are paired, g_p = h_{2p} + i h_{2p+1} (p < ceil(F/2); the last
//   pair of an odd bank has a zero imaginary part), and the plan holds the
//   spectra of the complex sequences g_p;
// * a segment a of the real signal is transformed as a complex sequence with
//   zero imaginary part (its spectrum A is Hermitian);
// * for each pair, one inverse FFT of A G_p gives a * g_p = a * h_{2p} +
//   i (a * h_{2p+1}); both convolutions are real, so the real part is the
//   output of filter 2p and the imaginary part that of filter 2p+1
//   (linearity of Eq. 1).
// Per two output streams: one N-point complex inverse FFT, the same work as
// two N/2-point transforms plus the post-processing of the paper's form, and
// the stores and the signal read move 4-byte real samples.  The forward FFT
// of the segment is done once per segment and amortised over the pairs.
#include <cuda_runtime.h>
#include <cstdint>

#include "ols_bank.cuh"
#include "ols_internal.h"

namespace ols {

// g[p][k] = (h[2p][k], h[2p+1][k]) with h[F][M] real; the missing partner of
// an odd F is zero.
__global__ void pack_real_pairs_kernel(const float *__restrict__ h, int M, int F, float2 *__restrict__ g) {
    const int Fc = (F + 1) / 2;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)Fc * M) return;
    const int p = (int)(i / M), k = (int)(i % M);
    const float re = h[(size_t)(2 * p) * M + k];
    const float im = (2 * p + 1 < F) ? h[(size_t)(2 * p + 1) * M + k] : 0.f;
    g[i] = make_float2(re, im);
}

cudaError_t launch_pack_real_pairs(const float *h, int M, int F, float2 *g, cudaStream_t st) {
    const long long total = (long long)((F + 1) / 2) * M;
    const int blocks = (int)((total + 255) / 256);
    pack_real_pairs_kernel<<<blocks, 256, 0, st>>>(h, M, F, g);
    return cudaGetLastError();
}

// Real samples in, one inverse FFT per filter pair, its real and imaginary
// parts stored as the pair's two output rows.
struct EpiReal {
    static constexpr bool WIDE = true;
    template <int LOG2N>
    static constexpr bool narrow() { return false; }
    static constexpr int XCH = XCHG_SHFL;
    template <int LOG2N>
    static constexpr int edge() { return 0; }
    const float *sig;
    float *y;
    int F;                  // real filters (F spectra of the bank kernel: pairs)
    __device__ __forceinline__ float2 sample(long long i) const { return make_float2(__ldg(sig + i), 0.f); }
    template <int LOG2N>
    __device__ __forceinline__ void spectrum(float2 *, int, const BankSegment &) const {}
    template <int LOG2N, class BAR>
    __device__ __forceinline__ void store(const float2 *x, int p, int t, const BankSegment &sg, float2 *, int &,
                                          const BAR &) const {
        using G = Geo<LOG2N>;
        const int v = G::base(t) - sg.n0;
        float *dre = y + (size_t)(2 * p) * (size_t)sg.Nout + (sg.j0 + v);
        // the pair test is uniform: taken once per filter pair, so each store
        // below is a plain predicated store
        if (2 * p + 1 < F) {
            float *dim = dre + sg.Nout;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const bool ok = (unsigned)(v + G::off(k)) < (unsigned)sg.span &&
                                in_bounds(sg.j0 + v + G::off(k) < sg.Nout, sg.status);
                if (ok) __stcs(dre + G::off(k), x[k].x);
                if (ok) __stcs(dim + G::off(k), x[k].y);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if ((unsigned)(v + G::off(k)) < (unsigned)sg.span && in_bounds(sg.j0 + v + G::off(k) < sg.Nout, sg.status))
                    __stcs(dre + G::off(k), x[k].x);
        }
    }
};

cudaError_t r2r_prepare(ols_plan_s &p) { return bank_prepare_any<EpiReal>(p.log2N); }

cudaError_t r2r_launch(const ols_plan_s &p, const float *s, int64_t Ns, float *y, int64_t L, int64_t nseg,
                       int64_t Nout, cudaStream_t st) {
    BankArgs a{};
    a.Hk = reinterpret_cast<const float4 *>(p.Hk);
    a.tw = p.twb;
    a.F = (p.F + 1) / 2;
    a.n0 = p.M - 1;
    a.step = L;
    a.off = 0;
    a.Ns = Ns;
    a.Nout = Nout;
    a.nseg = nseg;
    a.status = p.d_status;
    return bank_launch_any(p.log2N, a, EpiReal{s, y, p.F}, p.sm_count, st);
}

}  // namespace ols
