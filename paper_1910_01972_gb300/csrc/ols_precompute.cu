// ols_precompute.cu -- plan-time FP64 kernels: the twiddle table W_N^m and
// the filter spectra (Algorithms 1 and 2, "forward FFT of the filters",
// done once before the convolution kernel; Fig. 1's first step).
//
// FP64 is used only here, off the convolution path: every exponent is
// reduced exactly in integers before the table lookup, and each spectrum
// value is an FP64 FFT's, rounded once to FP32.
#include <cuda_runtime.h>
#include <cstdint>

#include "ols_internal.h"

namespace ols {

__global__ void tw64_kernel(double2 *tw64, int N) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= N) return;
    double sn, cs;
    sincospi(2.0 * (double)m / (double)N, &sn, &cs);   // argument exact: N is a power of two
    tw64[m] = make_double2(cs, -sn);                     // exp(-2 pi i m / N)
}

// H[f][nu] = (1/N) sum_{k<M} h_f[k] W_N^{nu k}, written at storage position q
// (nu = nu_tab[q]) in the kernel's register layout: thread t = q / 16 holds
// register j = q % 16, and registers (2i, 2i+1) of all threads of a segment
// are interleaved so one 16-byte load fetches a pair.  Ht (adjoint; may be
// null): the spectrum of conj(h_f[M-1-k]), which is W_N^{nu (M-1)} conj(H).
//
// The zero-padded filter's spectrum at the frequencies nu = r + 16 k of one
// residue r is the P = N/16-point FFT of
//   u_r[n] = sum_j h[n + j P] W_N^{r (n + j P)},  n < P,
// and is exactly the block [r P, (r + 1) P) of storage positions (the forward
// FFT's first pass).  One group of P/2 threads per (filter, residue): the
// taps once (M cos/sin products in all), then log2 P radix-2 stages in shared
// memory, all in FP64 with exactly reduced exponents.  Bound by the FP64 unit
// (two multiply-adds per clock and SM): 4 M / P + 4 log2 P operations per point
// and table against the direct sum's 4 M (each of M = 129 .. 1025 taps for
// every frequency), and 16 F blocks even for small banks.  Both tables, before /
// after: F = 8, M = 65, N = 512 62 -> 9 us; 16, 129, 1024 116 -> 9; 32, 257, 2048
// 435 -> 13; 64, 512, 4096 2962 -> 33; 24, 1025, 8192 5098 -> 31 us.
__global__ void spectra_kernel(const float2 *__restrict__ h, int M, int log2N, const int32_t *__restrict__ nu_tab,
                               const double2 *__restrict__ tw64, float2 *__restrict__ Hk, float2 *__restrict__ Htk,
                               int layout) {
    extern __shared__ double2 smem64[];
    const int N = 1 << log2N, P = N / 16, lp = log2N - 4, TR = P / 2;
    const int grp = threadIdx.x / TR, i = threadIdx.x % TR;      // residue group of the block, its butterfly
    const int per_block = blockDim.x / TR;
    const int blocks = 16 / per_block;                           // blocks per filter
    const int f = blockIdx.x / blocks, r = (blockIdx.x % blocks) * per_block + grp;
    double2 *u = smem64 + grp * P;
    const float2 *hf = h + (size_t)f * M;
    double2 x[2];                                                // u_r[i], u_r[i + P/2]
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        double ar = 0.0, ai = 0.0;
        for (int k = i + e * TR; k < M; k += P) {
            const double2 w = tw64[((long long)r * k) & (N - 1)];
            const float2 hk = hf[k];
            ar = fma((double)hk.x, w.x, fma(-(double)hk.y, w.y, ar));
            ai = fma((double)hk.x, w.y, fma((double)hk.y, w.x, ai));
        }
        x[e] = make_double2(ar, ai);
    }
    // decimation in frequency: stage s pairs (p, p + s); U[k] ends at bit-reversed k
    for (int s = TR; s >= 1; s >>= 1) {
        const int m = i & (s - 1), p = ((i & ~(s - 1)) << 1) | m;
        if (s < TR) {
            x[0] = u[p];
            x[1] = u[p + s];
        }
        const double2 w = tw64[(long long)m * (N / (2 * s))];
        const double dr = x[0].x - x[1].x, di = x[0].y - x[1].y;
        u[p] = make_double2(x[0].x + x[1].x, x[0].y + x[1].y);
        u[p + s] = make_double2(fma(dr, w.x, -di * w.y), fma(dr, w.y, di * w.x));
        __syncthreads();
    }
    const double inv = 1.0 / (double)N;
    const int T = N / 16;
    for (int e = i; e < P; e += TR) {                            // e: (j, t) with t fastest
        const int tl = e & (P / 16 - 1), j = e / (P / 16);
        const int t = r * (P / 16) + tl;
        const int nu = nu_tab[16 * t + j], k = nu >> 4;
        const double2 v = u[__brev((unsigned)k) >> (32 - lp)];
        const size_t idx = (size_t)f * N + (size_t)(j >> 1) * (2 * T) + 2 * t + (j & 1);
        size_t hidx = idx;
        if (layout != LAYOUT_STD) {
            const int q = layout_pos(layout, nu);
            hidx = (size_t)f * N + (size_t)((q & 15) >> 1) * (2 * T) + 2 * (q >> 4) + (q & 1);
        }
        Hk[hidx] = make_float2((float)(v.x * inv), (float)(v.y * inv));
        if (Htk) {
            const double2 w = tw64[((long long)nu * (M - 1)) & (N - 1)];
            const double cr = fma(w.x, v.x, w.y * v.y), ci = fma(w.y, v.x, -w.x * v.y);   // w conj(v)
            Htk[idx] = make_float2((float)(cr * inv), (float)(ci * inv));
        }
    }
}

// Natural-order copy of the plan's spectra: H[f][nu_tab[q]] = Hk[f][layout(q)].
__global__ void spectra_natural_kernel(const float2 *__restrict__ Hk, int F, int log2N,
                                       const int32_t *__restrict__ nu_tab, float2 *__restrict__ H, int layout) {
    const int N = 1 << log2N;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long long)F * N) return;
    const int f = (int)(gid >> log2N);
    const int q = (int)(gid & (N - 1));
    const int T = N / 16, t = q >> 4, j = q & 15;
    const size_t idx = (size_t)f * N + (size_t)(j >> 1) * (2 * T) + 2 * t + (j & 1);
    H[(size_t)f * N + (layout == LAYOUT_STD ? nu_tab[q] : layout_freq(layout, q))] = Hk[idx];
}

cudaError_t launch_tw64(double2 *tw64, int N, cudaStream_t st) {
    tw64_kernel<<<(N + 255) / 256, 256, 0, st>>>(tw64, N);
    return cudaGetLastError();
}

cudaError_t launch_spectra(const float2 *h, int M, int F, int log2N, const int32_t *nu,
                           const double2 *tw64, float2 *Hk, float2 *Htk, int layout, cudaStream_t st) {
    const int P = (1 << log2N) / 16, block = P / 2 > 32 ? P / 2 : 32;
    const int per_block = block / (P / 2);
    const long long grid = (long long)F * (16 / per_block);
    if (grid > 0x7fffffffll) return cudaErrorInvalidValue;
    spectra_kernel<<<(unsigned)grid, block, sizeof(double2) * (size_t)(P * per_block), st>>>(h, M, log2N, nu, tw64, Hk,
                                                                                            Htk, layout);
    return cudaGetLastError();
}

cudaError_t launch_spectra_natural(const float2 *Hk, int F, int log2N, const int32_t *nu, float2 *H,
                                   int layout, cudaStream_t st) {
    const long long total = (long long)F << log2N;
    spectra_natural_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(Hk, F, log2N, nu, H, layout);
    return cudaGetLastError();
}

}  // namespace ols
