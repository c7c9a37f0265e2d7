// Shell sums of the energy spectrum (kbc_spectrum in include/kbc.h).
#pragma once

#include <cuda_runtime.h>

namespace kbc {

// z = ux + i uy.  One complex transform of z serves both components:
// |Z(k)|^2 + |Z(-k)|^2 = 2 (|ux_hat(k)|^2 + |uy_hat(k)|^2), and k and -k lie in
// the same shell, so the shell sums of |Z|^2 / 2 are those of both energies.
// 4096^2: 3.1 ms against 4.3 ms for two real transforms.
__global__ void __launch_bounds__(256)
spectrum_pack(const double* __restrict__ u, long long nn, double2* __restrict__ z)
{
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < nn; q += (long long)gridDim.x * blockDim.x)
        z[q] = make_double2(u[q], u[nn + q]);
}

// round(sqrt(m)): the single-precision root, put right by s^2 - s < m <= s^2 + s
__device__ __forceinline__ int shell_of(int m)
{
    int s = (int)(sqrtf((float)m) + 0.5f);
    if (s > 0 && m <= s * s - s) --s;  // m = 0 is shell 0
    if (m > s * s + s) ++s;
    return s;
}

// Adds |Z|^2 scale / 2 of every coefficient (row = y, column = x wavenumber in
// FFT order) to its shell sum E[round(|k|)], shells >= nbins left out.  scale =
// 1 / n^4 turns |FFT|^2 into that of coefficients normalised by the node count.
// A thread sums runs of eight columns and adds to the histogram where the
// shell changes; a warp in one shell adds once.  (One atomic addition and one
// double square root per coefficient took as long as a transform.)  With
// smem != 0 a block sums in a shared histogram of nbins doubles first.
// HALF: z is the half spectrum of a real field, columns 0 .. n/2, of which those
// between stand for their Hermitian partners as well.
constexpr int kShellRun = 8;

template <bool HALF>
__global__ void __launch_bounds__(256)
spectrum_bin(const double2* __restrict__ z, int n, int nbins, double scale, double* __restrict__ E, int smem)
{
    extern __shared__ double hist[];
    double* sum = smem ? hist : E;
    if (smem) {
        for (int b = threadIdx.x; b < nbins; b += blockDim.x) hist[b] = 0.0;
        __syncthreads();
    }
    auto put = [&](int shell, double v) {
        if (shell < nbins) atomicAdd(sum + shell, v * (0.5 * scale));
    };
    const int w = HALF ? n / 2 + 1 : n;  // columns
    const int lane = threadIdx.x & 31, chunks = (w + 32 * kShellRun - 1) / (32 * kShellRun);
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (long long t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < (long long)n * chunks; t += warps) {
        const int ky = (int)(t / chunks), x0 = ((int)(t - (long long)ky * chunks) * 32 + lane) * kShellRun;
        const int fy = 2 * ky < n ? ky : ky - n;
        const double2* row = z + (long long)ky * w;
        double acc = 0.0;
        int cur = -1;
        bool moved = false;
#pragma unroll
        for (int j = 0; j < kShellRun; ++j) {
            const int kx = x0 + j;
            if (kx >= w) break;
            const int fx = 2 * kx < n ? kx : kx - n;
            const int shell = shell_of(fx * fx + fy * fy);
            if (shell != cur && cur >= 0) {
                put(cur, acc);
                acc = 0.0;
                moved = true;
            }
            cur = shell;
            const double2 c = row[kx];
            if constexpr (HALF) acc = fma(kx == 0 || 2 * kx == n ? 1.0 : 2.0, fma(c.x, c.x, c.y * c.y), acc);
            else acc = fma(c.x, c.x, fma(c.y, c.y, acc));
        }
        const int first = __shfl_sync(0xffffffffu, cur, 0);
        if (__all_sync(0xffffffffu, !moved && cur == first)) {
            for (int d = 16; d > 0; d >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, d);
            if (lane == 0 && cur >= 0) put(cur, acc);
        } else if (cur >= 0) {
            put(cur, acc);
        }
    }
    if (smem) {
        __syncthreads();
        for (int b = threadIdx.x; b < nbins; b += blockDim.x)
            if (hist[b] != 0.0) atomicAdd(&E[b], hist[b]);
    }
}

// Z(k) = (2 pi k / n)^2 E(k): the enstrophy density of shell k.
__global__ void spectrum_enstrophy(const double* __restrict__ E, double* __restrict__ Z, int nbins,
                                   int n)
{
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nbins; b += gridDim.x * blockDim.x) {
        const double k = 6.283185307179586 * (double)b / (double)n;
        Z[b] = k * k * E[b];
    }
}

}  // namespace kbc
