// ols_tc64.cu -- the tensor-core split-precision form at N = 4096: two
// radix-64 stages as matrix products of K = 128.
//
// A 4096-point inverse transform with n = 64 n1 + n2 and nu = nu1 + 64 nu2 is
//   Z[nu1, n2]   = sum_nu2 Y[nu1 + 64 nu2] e(n2 nu2 / 64)         (stage 1)
//   x[64 n1 + n2] = sum_nu1 (Z[nu1, n2] e(n2 nu1 / 4096)) e(n1 nu1 / 64)   (stage 2)
// with e(a) = exp(2 pi i a): two products with the same 64-point DFT, as a real
// 128 x 128 matrix B = [[C, S], [-S, C]].  A CTA of 512 threads holds two
// segments as the 128 rows of an MMA tile; 16-bit split operands and the three
// products hi B_hi + hi B_lo + lo B_hi as in ols_tc.cu, FP32 accumulation.
// * Stage 1: row (segment, nu1); the thread (row, quarter c of nu2) multiplies
//   its 16 points by the filter's spectrum, splits them and stores them to its
//   TMEM lane as the A operand.
// * Stage 2: the contraction runs over stage 1's rows, so its A operand goes
//   through shared memory, where a thread writes its 16 n2 as contiguous
//   columns (M-major operand, 16-byte stores without bank conflicts); this
//   store is the transform's only exchange.  Row (segment, n2), so a warp
//   stores 32 consecutive outputs.
// * The forward transform of a segment is the same two stages on the conjugate
//   of the signal (its result conjugated), so one matrix serves both.
// * Software pipeline over the filters: while the tensor cores run stage 1 of
//   filter i - 1 and stage 2 of filter i - 2, the threads prepare stage 1 of
//   filter i; then they read both results, which frees the tensor cores for
//   stage 1 of filter i, store filter i - 2 and twiddle filter i - 1.  The warps
//   meet only on mbarriers with the warp that issues the MMAs.  The segments'
//   spectra wait in shared memory (in registers they made the kernel spill,
//   and beside 224 KB of shared memory there is hardly an L1 to spill to).
// What bounds it: the tensor cores (53% of cycles active, ncu) and, where they
// idle, the threads' latencies.  A filter and segment pair takes 48 MMAs of
// 128 x 128 x 16 (65 cycles each in a loop of nothing else, 3100 in all), the
// threads about 2900 issue cycles beside them, of 5700 that a step takes.
// Three radix-16 stages (ols_tc.cu) need a third of the multiply-adds but split,
// store, wait and exchange three times, and their threads' work bounds them:
// 64 filters, 2^22 samples 1146 us there, 734 here (FP16; the FP32 kernel 569).
// Small calls too (device time, radix-16 form / here, though a CTA copies 96 KB of tables first): one
// filter of 613 samples 13.4 / 13.1 us, of 300,000 13.7 / 13.9; 8 filters of 40,000 32 / 14.
// Spectra prefetched a filter ahead were 4% slower: their registers spill.
// Scale (an exact power of two): the segment's spectrum x 16, undone in the output.
// Both inverse operands, Y and Z, are averages of phase-rotated outputs of the
// segment's circular convolution, so |Y|, |Z| <= |s| sqrt(M) for a unit-L2 filter (a
// tone in its matched filter reaches it): at most 16 x 1.42 x 64 = 1454 for |s| <= 1.42, and FP16's
// 65504 from |s| sqrt(M) = 4094 on (x 512: from 128 on).  The forward transform's
// second operand is at most 64 |s|.  At the other end FP16 runs out of bits below
// 2^-14.  Errors (1e-6) of uniform signals of amplitude 2^-10, 2^-6, 2^-3 and 1 through random
// filters: 130, 8, 1.2, 0.68 (stage 2's operands at an eighth of this: 180, 11, 1.5, 0.69; the
// radix-16 form 210, 13, 2.1, 1.2); of a tone of 2^-10 in its matched filter (M = 512), against
// the samples as split: 1.3 (2.2; 2.6).  The split itself costs that tone 2.5.
// Waits are bounded as in ols_tc.cu.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "ols_fft_passes.cuh"
#include "ols_internal.h"
#include "ols_tc_split.cuh"

namespace ols {

namespace tc64 {

constexpr int kMat = 128 * 128 * 2;                 // one 16-bit operand matrix, bytes
constexpr int kSmemA = 2 * kMat;                    // after B hi, B lo: stage 2's A (hi, lo)
constexpr int kSmemX = kSmemA + 2 * kMat;           // the two segments' spectra: 8192 complex
constexpr int kSmemTw = kSmemX + 8192 * 8;          // twiddles: 4096 complex
constexpr int kSmem = kSmemTw + 4096 * 8;
constexpr uint32_t kD1 = 256, kD2 = 384;            // TMEM columns: stage 1's A (two of 128), D1, D2

__device__ __forceinline__ uint64_t desc(uint32_t addr) {
    // no swizzle; 2048 bytes between groups of 8 along K, 128 along M or N; descriptor version 1
    uint64_t d = (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)(2048 >> 4) << 16;
    d |= (uint64_t)(128 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}
// kind::f16: D FP32, A and B FP16 or BF16, M = N = 128; AT: A is M-major
template <bool BF16, bool AT>
__device__ __forceinline__ constexpr uint32_t idesc() {
    return (1u << 4) | ((BF16 ? 1u : 0u) << 7) | ((BF16 ? 1u : 0u) << 10) | ((AT ? 1u : 0u) << 15) |
           ((128u >> 3) << 17) | ((128u >> 4) << 24);
}

__device__ __forceinline__ void st4(uint32_t a, const uint32_t *v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3])
                 : "memory");
}
__device__ __forceinline__ void sts16(uint32_t a, const uint32_t *v) {
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
                 : "memory");
}

// The thread block: 16 warps of 512 data threads and one that issues the MMAs
// (the tensor core takes a few MMAs at a time, so the issuing thread spends
// its time waiting for it).  They meet on mbarriers: ready[s] (16 warps) says
// that stage s + 1's operands are stored and its last results read, done[s]
// that its MMAs are complete.
// The MMA warp has a warpgroup to itself and hands its registers to the data
// warps: launched with 640 x 96 = 61440, then 512 x 104 + 128 x 56 = 60416.
constexpr int kData = 512, kThreads = kData + 128;

struct Bars {
    uint32_t ready[2], done[2];
    uint32_t watch[2];      // what the data warps wait on: done, or (test switch) one nothing arrives on
};

__device__ __forceinline__ void arrive(uint32_t bar) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0)
        asm volatile("{\n.reg .b64 t;\nmbarrier.arrive.shared::cta.b64 t, [%0];\n}" ::"r"(bar) : "memory");
}

// A data warp's bounded wait for stage g + 1's MMAs: one lane polls.  False
// once it ran out (recorded; the warp then leaves).
__device__ __forceinline__ bool wait_done(const Bars &b, int g, uint32_t &phase, long long limit, int *status) {
    bool ok = true;
    if ((threadIdx.x & 31) == 0) {
        ok = tc::poll(b.watch[g], (phase >> g) & 1u, limit);
        if (!ok) atomicOr(status, kStatusWaitExpired);
    }
    ok = __all_sync(0xffffffffu, ok);
    phase ^= 1u << g;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return ok;
}

// The 24 MMAs of stage 1 (A in TMEM, buffer b) or stage 2 (A in shared memory)
// and their commit (unrolled: in a loop the issue took 164 cycles per MMA, the
// tensor core takes 64).  The two products with a low part come first: the tensor core
// truncates each partial sum to FP32, and while the accumulator holds only them
// that costs 2^-11 of what it would after hi B_hi (whole convolution 6.8e-7;
// 2.8e-6 with hi B_hi first).
template <int STAGE, bool BF16>
__device__ __forceinline__ void issue(uint32_t sm, uint32_t done, int b) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("" : "+r"(sm));     // descriptors are formed here, not hoisted into registers the warp has not got
    const uint64_t bm = desc(sm), am = desc(sm + kSmemA);
#pragma unroll
    for (int i = 0; i < 24; ++i) {
        const int term = i / 8, kk = i % 8;                      // lo hi, hi lo, hi hi
        const uint64_t bd = bm + (uint64_t)(((term == 1 ? kMat : 0) + kk * 4096) >> 4);
        const uint64_t ad = am + (uint64_t)(((term == 0 ? kMat : 0) + kk * 4096) >> 4);
        const uint32_t a = 128u * (uint32_t)b + (term == 0 ? 64u : 0u) + 8u * kk, acc = i > 0;
        if constexpr (STAGE == 1)
            asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                         "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(kD1),
                         "r"(a), "l"(bd), "r"(idesc<BF16, false>()), "r"(acc)
                         : "memory");
        else
            asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                         "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(kD2),
                         "l"(ad), "l"(bd), "r"(idesc<BF16, true>()), "r"(acc)
                         : "memory");
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(done) : "memory");
}

// This thread's 16 complex points of stage g + 1's result (columns 16 q .. of
// the real and of the imaginary half).
__device__ __forceinline__ void load_d(float2 *x, uint32_t lane, int g, int q) {
    float re[16], im[16];
    const uint32_t d = lane + (g == 0 ? kD1 : kD2) + 16u * (uint32_t)q;
    tmem::ld16(d, re);
    tmem::ld16(d + 64, im);
    tmem::wait_ld16(re);
    tmem::wait_ld16(im);
#pragma unroll
    for (int j = 0; j < 16; ++j) x[j] = make_float2(re[j], im[j]);
}

// Half h of a thread's stage-1 operand: words (Re x_2w, Re x_2w+1), (Im ..), hi and lo.
__device__ __forceinline__ void store_a1(uint32_t lane, int b, int q, int h, const uint32_t *rh, const uint32_t *ih,
                                         const uint32_t *rl, const uint32_t *il) {
    const uint32_t a = lane + 128u * (uint32_t)b + 8u * (uint32_t)q + 4u * (uint32_t)h;
    st4(a, rh);
    st4(a + 32, ih);
    st4(a + 64, rl);
    st4(a + 96, il);
}

template <bool BF16>
__device__ __forceinline__ void split8(const float2 *x, uint32_t *rh, uint32_t *ih, uint32_t *rl, uint32_t *il) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        tc::split2<BF16>(x[2 * w].x, x[2 * w + 1].x, rh[w], rl[w]);
        tc::split2<BF16>(x[2 * w].y, x[2 * w + 1].y, ih[w], il[w]);
    }
}

// Twiddle stage 1's result (row r, points n2 = 16 q ..) and store it as stage 2's operand.
template <bool BF16>
__device__ __forceinline__ void store_a2(const float2 *z, uint32_t sm, const float4 *tw, int q, int row) {
    const int r = row & 63;
    const uint32_t a = sm + kSmemA + (uint32_t)((row >> 6) * 8 + 2 * q) * 128u +
                       (uint32_t)(r >> 3) * 2048u + (uint32_t)(r & 7) * 16u;   // k = r; imaginary part: k = 64 + r
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float2 v[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 w = tw[(4 * h + i) * 256 + 64 * q + r];
            v[2 * i] = cmul(z[8 * h + 2 * i], make_float2(w.x, w.y));
            v[2 * i + 1] = cmul(z[8 * h + 2 * i + 1], make_float2(w.z, w.w));
        }
        uint32_t rh[4], ih[4], rl[4], il[4];
        split8<BF16>(v, rh, ih, rl, il);
        sts16(a + 128 * h, rh);
        sts16(a + 128 * h + 8 * 2048, ih);
        sts16(a + 128 * h + kMat, rl);
        sts16(a + 128 * h + kMat + 8 * 2048, il);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

}  // namespace tc64

template <bool BF16, bool PRE>
__global__ void __launch_bounds__(tc64::kThreads, 1)
ols_tc64_kernel(const float2 *__restrict__ sig, const uint32_t *__restrict__ sig_hi, const uint32_t *__restrict__ sig_lo,
                long long Ns, const float4 *__restrict__ Hk, const uint4 *__restrict__ tables, float2 *__restrict__ y,
                int M, int F, long long L, long long nseg, long long Nout, long long total, int *status,
                long long wait_limit, int wait_never) {
    using namespace tc64;
    extern __shared__ float4 smem_raw[];
    __shared__ __align__(8) uint64_t mbar[6];       // ready[2], done[2], all MMAs done, one that nothing arrives on
    __shared__ uint32_t tbase;
    const uint32_t sm = tc::smem_u32(smem_raw);
    Bars bars;
    for (int g = 0; g < 2; ++g) {
        bars.ready[g] = tc::smem_u32(&mbar[g]);
        bars.done[g] = tc::smem_u32(&mbar[2 + g]);
        bars.watch[g] = wait_never ? tc::smem_u32(&mbar[5]) : bars.done[g];
    }
    // B hi, B lo and the twiddles
    for (int i = threadIdx.x; i < 2 * kMat / 16; i += kThreads) reinterpret_cast<uint4 *>(smem_raw)[i] = tables[i];
    for (int i = threadIdx.x; i < 4096 * 8 / 16; i += kThreads)
        reinterpret_cast<uint4 *>(smem_raw)[kSmemTw / 16 + i] = tables[2 * kMat / 16 + i];
    if (threadIdx.x == 0)
        for (int i = 0; i < 6; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_u32(&mbar[i])), "r"(i < 2 ? 16 : 1)
                         : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // the CTA owns all 512 columns, so they start at column 0: TMEM addresses are constants
    if (threadIdx.x / 32 == kData / 32) tmem::alloc(&tbase, 512);
    tmem::fence_before_sync();
    __syncthreads();
    tmem::fence_after_sync();

    // this CTA's share of the (segment pair, filter) steps
    const long long each = total / gridDim.x, more = total % gridDim.x, bi = blockIdx.x;
    const long long s0 = each * bi + (bi < more ? bi : more);
    long long todo = each + (bi < more ? 1 : 0);
    long long pair = s0 / F;
    int f = (int)(s0 - pair * F);

    if (threadIdx.x >= kData) {
        // the MMA warp: one thread follows the data warps' order
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (threadIdx.x == kData) {
            uint32_t phase = 0;
            bool ok = true;
            auto step = [&](int g, int b) {
                ok = ok && tc::poll(bars.ready[g], (phase >> g) & 1u, wait_limit);
                phase ^= 1u << g;
                if (!ok) return;
                if (g == 0) issue<1, BF16>(sm, bars.done[0], b);
                else issue<2, BF16>(sm, bars.done[1], 0);
            };
            for (; todo > 0 && ok; f = 0) {
                const int nf = F - f < todo ? F - f : (int)todo;
                todo -= nf;
                step(0, 0);                                  // the segments' forward transform
                step(1, 0);
                for (int it = 0; it <= nf && ok; ++it) {
                    if (it < nf) step(0, it & 1);
                    if (it >= 1) step(1, 0);
                }
            }
            if (!ok) atomicOr(status, kStatusWaitExpired);
            // everything issued is complete before the memory goes (bounded)
            const uint32_t all = tc::smem_u32(&mbar[4]);
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(all)
                         : "memory");
            tc::poll(all, 0, tc::kWaitLimit);
        }
        __syncwarp();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        const int row = threadIdx.x & 127, q = threadIdx.x >> 7, r = row & 63;
        const float4 *tw = reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(smem_raw) + kSmemTw);
        const uint32_t lane = tmem::lane_bits();
        float4 *const xs = smem_raw + kSmemX / 16 + threadIdx.x; // this thread's 16 points of the spectrum
        const int v0 = 1024 * q + r - (M - 1);                   // output v0 + 64 j of the segment
        uint32_t phase = 0;
        bool ok = true;
        for (; todo > 0 && ok; ++pair, f = 0) {
            const long long seg = 2 * pair + (row >> 6);
            const bool active = seg < nseg;
            const long long start = active ? seg * L : 0;
            const int nf = F - f < todo ? F - f : (int)todo;
            todo -= nf;
            {
                // forward: samples start + 64 (16 q + j) + r, conjugated
                const long long avail = active ? Ns - start : 0;
                const int lim = (int)(avail < 4096 ? avail : 4096);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t rh[4], ih[4], rl[4], il[4];
                    if constexpr (PRE) {
                        uint32_t a[8], b[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int n = 64 * (16 * q + 8 * h + j) + r;
                            const bool in = n < lim && in_bounds(start + n < Ns, status);
                            a[j] = in ? __ldg(sig_hi + start + n) : 0u;
                            b[j] = in ? __ldg(sig_lo + start + n) : 0u;
                        }
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            rh[w] = __byte_perm(a[2 * w], a[2 * w + 1], 0x5410);
                            ih[w] = __byte_perm(a[2 * w], a[2 * w + 1], 0x7632) ^ 0x80008000u;
                            rl[w] = __byte_perm(b[2 * w], b[2 * w + 1], 0x5410);
                            il[w] = __byte_perm(b[2 * w], b[2 * w + 1], 0x7632) ^ 0x80008000u;
                        }
                    } else {
                        float2 x[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int n = 64 * (16 * q + 8 * h + j) + r;
                            x[j] = (n < lim && in_bounds(start + n < Ns, status)) ? __ldg(sig + start + n)
                                                                                  : make_float2(0.f, 0.f);
                            x[j].y = -x[j].y;
                        }
                        split8<BF16>(x, rh, ih, rl, il);
                    }
                    store_a1(lane, 0, q, h, rh, ih, rl, il);
                }
                tmem::wait_st();
                tmem::fence_before_sync();
                arrive(bars.ready[0]);
                float2 X[16];
                ok = wait_done(bars, 0, phase, wait_limit, status);
                if (!ok) break;
                load_d(X, lane, 0, q);
                store_a2<BF16>(X, sm, tw, q, row);
                tmem::fence_before_sync();
                arrive(bars.ready[1]);
                ok = wait_done(bars, 1, phase, wait_limit, status);
                if (!ok) break;
                load_d(X, lane, 1, q);
                // conjugate back, x 16: the spectrum's scale
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    xs[512 * i] = make_float4(X[2 * i].x * 16.f, X[2 * i].y * -16.f, X[2 * i + 1].x * 16.f,
                                              X[2 * i + 1].y * -16.f);
            }
            const long long rem = active ? Nout - start : 0;
            const int span = (int)(rem < L ? rem : L);
            for (int it = 0; it < nf + 2; ++it) {
                if (it < nf) {                          // stage 1 of filter f + it
                    const float4 *hp = Hk + (size_t)(f + it) * 2048 + 64 * q + r;
                    float4 h4[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) h4[i] = load_spectrum(hp + 256 * i);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float2 x[8];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float4 w = h4[4 * h + i], X = xs[512 * (4 * h + i)];
                            x[2 * i] = cmul(make_float2(X.x, X.y), make_float2(w.x, w.y));
                            x[2 * i + 1] = cmul(make_float2(X.z, X.w), make_float2(w.z, w.w));
                        }
                        uint32_t rh[4], ih[4], rl[4], il[4];
                        split8<BF16>(x, rh, ih, rl, il);
                        store_a1(lane, it & 1, q, h, rh, ih, rl, il);
                    }
                }
                const bool mid = it >= 1 && it <= nf;   // filter f + it - 1 between its stages
                float2 z[16];
                if (mid) {
                    ok = wait_done(bars, 0, phase, wait_limit, status);
                    if (!ok) break;
                    load_d(z, lane, 0, q);
                }
                if (it < nf) {                          // D1 is read: stage 1 of filter f + it may follow
                    tmem::wait_st();
                    tmem::fence_before_sync();
                    arrive(bars.ready[0]);
                }
                if (it >= 2) {                          // filter f + it - 2 done
                    ok = wait_done(bars, 1, phase, wait_limit, status);
                    if (!ok) break;
                }
                if (mid) store_a2<BF16>(z, sm, tw, q, row);
                if (it >= 2) load_d(z, lane, 1, q);
                if (mid) {                              // D2 is read: stage 2 of filter f + it - 1 may follow
                    tmem::fence_before_sync();
                    arrive(bars.ready[1]);
                }
                if (it >= 2) {
                    float2 *dst = y + (size_t)(f + it - 2) * (size_t)Nout + (start + v0);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if ((unsigned)(v0 + 64 * j) < (unsigned)span && in_bounds(start + v0 + 64 * j < Nout, status))
                            __stcs(dst + 64 * j, make_float2(z[j].x * 0.0625f, z[j].y * 0.0625f));
                }
            }
        }
    }
    tmem::fence_before_sync();
    __syncthreads();
    tmem::fence_after_sync();
    if (threadIdx.x / 32 == kData / 32) tmem::dealloc(tbase, 512);
}

template <bool BF16, bool PRE>
static cudaError_t tc64_prepare_one() {
    return cudaFuncSetAttribute(ols_tc64_kernel<BF16, PRE>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc64::kSmem);
}
cudaError_t tc64_prepare(bool bf16) {
    cudaError_t e = bf16 ? tc64_prepare_one<true, false>() : tc64_prepare_one<false, false>();
    if (e == cudaSuccess) e = bf16 ? tc64_prepare_one<true, true>() : tc64_prepare_one<false, true>();
    return e;
}

template <bool BF16, bool PRE>
static cudaError_t tc64_launch_one(const ols_plan_s &p, const TcSignal &sg, int64_t Ns, float2 *y, int64_t L,
                                   int64_t nseg, int64_t Nout, cudaStream_t st) {
    const long long total = (nseg + 1) / 2 * p.F;
    const int grid = (int)(total < p.sm_count ? total : p.sm_count);
    ols_tc64_kernel<BF16, PRE><<<grid, tc64::kThreads, tc64::kSmem, st>>>(
        sg.s, sg.hi, sg.lo, Ns, reinterpret_cast<const float4 *>(p.Hk), reinterpret_cast<const uint4 *>(p.tc_bmat), y,
        p.M, p.F, L, nseg, Nout, total, p.d_status, p.tc_wait_limit, p.tc_wait_never ? 1 : 0);
    return cudaGetLastError();
}
cudaError_t tc64_launch(const ols_plan_s &p, const TcSignal &sg, int64_t Ns, float2 *y, int64_t L, int64_t nseg,
                        int64_t Nout, cudaStream_t st) {
    const bool bf16 = (p.flags & OLS_FLAG_TC_BF16SPLIT) != 0, pre = sg.hi != nullptr;
    if (bf16) return pre ? tc64_launch_one<true, true>(p, sg, Ns, y, L, nseg, Nout, st)
                         : tc64_launch_one<true, false>(p, sg, Ns, y, L, nseg, Nout, st);
    return pre ? tc64_launch_one<false, true>(p, sg, Ns, y, L, nseg, Nout, st)
               : tc64_launch_one<false, false>(p, sg, Ns, y, L, nseg, Nout, st);
}

}  // namespace ols
