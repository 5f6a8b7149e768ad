// ols_forward.cu -- the fused overlap-and-save convolution (FP32): the bank
// kernel with a plain store (Algorithm 2, Sec. 3.2 and 3.4).
#include <cuda_runtime.h>
#include <cstdint>

#include "ols_internal.h"
#include "ols_bank.cuh"

namespace ols {

cudaError_t prepare_forward(ols_plan_s &p) { return bank_prepare_any<EpiPlain>(p.log2N); }

cudaError_t launch_forward(const ols_plan_s &p, const float2 *s, int64_t Ns, float2 *y, int64_t L,
                           int64_t nseg, int64_t Nout, cudaStream_t st, int *launches) {
    BankArgs a{};
    a.Hk = reinterpret_cast<const float4 *>(p.Hk);
    a.tw = p.twb;
    a.F = p.F;
    a.n0 = p.M - 1;
    a.step = L;
    a.off = 0;
    a.Ns = Ns;
    a.Nout = Nout;
    a.nseg = nseg;
    a.status = p.d_status;
    *launches = 1;
    return bank_launch_any(p.log2N, a, EpiPlain{s, y}, p.sm_count, st);
}

// Host mirror of Geo<>: the twiddle tables and spectral order are built from it.
PassPlan make_pass_plan(int log2N) {
    PassPlan pp{};
    pp.log2N = log2N;
    pp.N = 1 << log2N;
    pp.T = pp.N / 16;
    pp.np = (log2N + 3) / 4;
    const int rl = (log2N % 4) ? (1 << (log2N % 4)) : 16;
    int off = 0;
    for (int p = 0; p < pp.np; ++p) {
        pp.radix[p] = (p == pp.np - 1) ? rl : 16;
        pp.stride[p] = (p == pp.np - 1) ? 1 : (pp.N >> (4 * (p + 1)));
        pp.tw_off[p] = off;
        if (p < pp.np - 1) off += 15 * pp.stride[p];
    }
    pp.twn = off;
    return pp;
}

}  // namespace ols
