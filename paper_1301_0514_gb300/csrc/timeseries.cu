// Light-curve time analysis (Sect. 5): the time power spectrum of each curve,
// whose slope breaks near 1/t_ref, and the correlation of curves taken along
// parallel tracks (two telescopes a distance apart).
//
// Periodogram P_k = |sum_s (c_s - mean c) e^{-2 pi i k s / n}|^2 / n, k = 0..n/2:
// a team of n/16 threads holds one curve (16 values per thread), removes the
// curve's mean (FP64 sum) before the FP32 transform so that the rounding of
// a large mean does not leak into the weak bins, and writes |X_k|^2 / n.
// Correlation: one block per pair, mean then centred sums, FP64; pairs come in
// groups that share one row of a (a reference curve against its parallels).
#include "dispatch.cuh"
#include "fft.cuh"
#include "kernels.cuh"

namespace scint {

template <int N> __host__ __device__ constexpr int ps_lines() {
    return N >= kTileRow32 ? 1 : (kTileRow32 / N < 64 ? kTileRow32 / N : 64);
}

template <int N>
__global__ void __launch_bounds__(ps_lines<N>() * FftPlan<N>::T)
power_spectrum_kernel(const float* curves, int n_curves, float* power, const float2* tw) {
    using Pl = FftPlan<N>;
    constexpr int T = Pl::T, E = Pl::E, B = ps_lines<N>(), NW = (T + 31) / 32;
    extern __shared__ __align__(16) float2 ps_smem[];
    __shared__ double wsum[B][NW];
    const int team = threadIdx.x / T, t = threadIdx.x % T;
    const int c = blockIdx.x * B + team;
    const bool live = c < n_curves;
    const float* src = curves + (size_t)(live ? c : 0) * N;
    float x[E];
    double s = 0.0;
#pragma unroll
    for (int m = 0; m < E; ++m) {
        x[m] = live ? src[t + m * T] : 0.0f;
        s += x[m];
    }
    // team sum: warps of the team, then the team's warps in order
    if constexpr (T >= 32) {
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 31) == 0) wsum[team][t >> 5] = s;
    } else {
        // teams smaller than a warp: T lanes of one team are contiguous in the warp
        for (int o = T / 2; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, T);
        if (t == 0) wsum[team][0] = s;
    }
    __syncthreads();
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) tot += wsum[team][w];
    const float mean = (float)(tot / N);
    float2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = make_float2(x[m] - mean, 0.0f);
    fft_line<float2, N, -1, 16, 1, 0, 1>(v, ps_smem + team * Pl::BUF, t, tw);
    if (live) {
        float* out = power + (size_t)c * (N / 2 + 1);
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int k = t + m * T;
            if (k <= N / 2) out[k] = k == 0 ? 0.0f : fmaf(v[m].x, v[m].x, v[m].y * v[m].y) * (1.0f / N);
        }
    }
}

cudaError_t launch_power_spectrum(const float* curves, int n_curves, int n, float* power, const float2* tw,
                                  cudaStream_t s) {
    if (n_curves <= 0) return cudaSuccess;
    return dispatch_n(n, [&](auto nc) -> cudaError_t {
        constexpr int N = decltype(nc)::value;
        if constexpr (N > 8192) {
            return cudaErrorNotSupported;
        } else {
            constexpr int B = ps_lines<N>();
            constexpr size_t smem = (size_t)B * FftPlan<N>::BUF * sizeof(float2);
            cudaError_t e = set_smem(power_spectrum_kernel<N>, smem);
            if (e != cudaSuccess) return e;
            power_spectrum_kernel<N><<<(n_curves + B - 1) / B, B * FftPlan<N>::T, smem, s>>>(curves, n_curves,
                                                                                              power, tw);
            return cudaGetLastError();
        }
    });
}

// FP64 block sum (blockDim.x == 256), result in every thread
__device__ double block_sum_all(double v) {
    __shared__ double part[8];
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += part[w];
    __syncthreads();
    return t;
}

// U samples of a thread as doubles, through their bits unless one of them is unusual:
// on GB300's narrow FP64 pipe a conversion costs as much as two additions.
template <int U>
SCINT_DEV void load_widened(const float* x, int step, double (&d)[U]) {
    float v[U];
    bool odd = false;
#pragma unroll
    for (int k = 0; k < U; ++k) {
        v[k] = x[(size_t)k * step];
        odd |= f2d_unusual(v[k]);
    }
    if (!odd) {
#pragma unroll
        for (int k = 0; k < U; ++k) d[k] = f2d_bits(v[k]);
    } else {
#pragma unroll
        for (int k = 0; k < U; ++k) d[k] = (double)v[k];
    }
}
// f(k, x_s, y_s) for this thread's samples s: U at a time (k = 0..U - 1), the rest one by one (k = 0)
template <int U, typename F>
SCINT_DEV void for_samples(const float* x, const float* y, int n, F&& f) {
    const int step = blockDim.x;
    int s = threadIdx.x;
    if constexpr (U > 1) {
        for (; n - s > (U - 1) * step; s += U * step) {
            double xv[U], yv[U];
            load_widened(x + s, step, xv);
            load_widened(y + s, step, yv);
#pragma unroll
            for (int k = 0; k < U; ++k) f(k, xv[k], yv[k]);
        }
    }
#pragma unroll 1
    for (; s < n; s += step) {
        double xv[1], yv[1];
        load_widened(x + s, step, xv);
        load_widened(y + s, step, yv);
        f(0, xv[0], yv[0]);
    }
}

// The FP64 pipe bounds it (384 pairs of 4096 samples: 61 -> 54 us, 85 % busy before): U samples of a
// thread at a time, each with sums of its own, so that the additions do not wait for one another.
template <int U>
SCINT_DEV double block_total(const double (&v)[U]) {
    if constexpr (U == 4) return block_sum_all((v[0] + v[1]) + (v[2] + v[3]));
    else return block_sum_all(v[0]);
}
template <int U>
__global__ void __launch_bounds__(256) correlation_kernel(const float* a, int group, long long a_stride,
                                                          const float* b, int n, double* r) {
    const int i = blockIdx.x;
    const float* x = a + (size_t)(i / group) * a_stride;
    const float* y = b + (size_t)i * n;
    double ax[U] = {}, ay[U] = {};
    for_samples<U>(x, y, n, [&](int k, double xv, double yv) {
        ax[k] += xv;
        ay[k] += yv;
    });
    const double mx = block_total(ax) / n, my = block_total(ay) / n;
    double axy[U] = {}, axx[U] = {}, ayy[U] = {};
    for_samples<U>(x, y, n, [&](int k, double xv, double yv) {
        const double dx = xv - mx, dy = yv - my;
        axy[k] = fma(dx, dy, axy[k]);
        axx[k] = fma(dx, dx, axx[k]);
        ayy[k] = fma(dy, dy, ayy[k]);
    });
    const double sxy = block_total(axy), sxx = block_total(axx), syy = block_total(ayy);
    if (threadIdx.x == 0) r[i] = sxy / sqrt(sxx * syy);
}

cudaError_t launch_correlation(const float* a, int a_rows, long long a_stride, const float* b, int n_pairs, int n,
                               double* r, cudaStream_t s) {
    if (n_pairs <= 0) return cudaSuccess;
    // four samples at a time from four samples per thread on; below, one by one in fewer registers (10000 pairs of
    // 256 samples: 620 us with four sums of which three stay zero, 464 without)
    if (n >= 4 * 256) correlation_kernel<4><<<n_pairs, 256, 0, s>>>(a, n_pairs / a_rows, a_stride, b, n, r);
    else correlation_kernel<1><<<n_pairs, 256, 0, s>>>(a, n_pairs / a_rows, a_stride, b, n, r);
    return cudaGetLastError();
}

}  // namespace scint
