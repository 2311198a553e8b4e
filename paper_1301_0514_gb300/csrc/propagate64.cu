// Fresnel propagation of one screen at one wavelength entirely in FP64 (the paper's
// plain method, Eq. hxy, with the edge taper of Sect. 3.2.1): the reference-precision
// form of the FP32 passes in propagate.cu, for grids up to 4096^2.
//
// Row pass:    A_in = SF(x) SF(y) exp(i phi s) (FP64 sine and cosine of phi s), FFT_x,
//              times H_x(kx)/N, IFFT_x -> field (complex128, row-major).
// Column pass: field column -> FFT_y -> H_y(ky)/N -> IFFT_y -> |A|^2 (FP64 map).
// H(k) = exp(-i pi lambda z k^2) with k = m/L: the phase in turns is c m^2 with
// c = lambda z / (2 L^2); c is split as c_hi + c_lo with c_hi holding 31 significant
// bits, so that c_hi m^2 is exact in FP64 for |m| <= 2048 and its fractional part
// carries no rounding; c_lo m^2 adds the rest.
#include <cmath>

#include "dispatch.cuh"
#include "fft.cuh"
#include "kernels.cuh"

namespace scint {

// taper at pixel centre i + 1/2 (raised sine over the margin, 1 inside), FP64
SCINT_DEV double taper64(int i, int n, double margin_px) {
    if (margin_px <= 0.0) return 1.0;
    const double u = fmin((double)i + 0.5, (double)n - (double)i - 0.5);
    if (u > margin_px) return 1.0;
    const double sn = sinpi(u / (2.0 * margin_px));
    return sn * sn;
}

// H(m)/n for the signed frequency index m: exp(-2 pi i frac(c m^2)) / n
SCINT_DEV double2 transfer64(const Prop64Args& a, int i) {
    const int n = a.n;
    const long long m = i < n / 2 ? i : i - n;
    const double m2 = (double)(m * m);
    const double hi = a.c_hi * m2;                  // exact: 31 + 22 bits
    double turns = (hi - floor(hi)) + a.c_lo * m2;
    turns -= floor(turns);
    double sn, cs;
    sincospi(-2.0 * turns, &sn, &cs);
    return make_double2(cs / n, sn / n);
}

// H(m)/n for m = 0..n/2 and the taper of one half of a line (both are even), one value per thread:
// in the passes themselves they had been a sincospi per element of every line, and in the margin a
// sinpi too.  With the tables, twiddles kept between calls and four values per thread at 256^2 both
// passes took 83 -> 37 us there (FP64 pipe 33 -> 63 % busy), 168 -> 101 us at 512^2, 587 -> 346 us at 1024^2.
__global__ void prop64_tables_kernel(Prop64Args a, double2* h, double* sf) {
    begin_after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, half = a.n / 2;
    if (i <= half) h[i] = transfer64(a, i);
    if (i < half) sf[i] = taper64(i, a.n, a.margin_px);
}
template <int N, bool TAB>
SCINT_DEV double2 transfer_of(const Prop64Args& a, int i) {
    if constexpr (TAB) return a.h[i <= N / 2 ? i : N - i];
    else return transfer64(a, i);
}
template <int N, bool TAB>
SCINT_DEV double taper_of(const Prop64Args& a, int i) {
    if constexpr (TAB) return a.sf[i < N / 2 ? i : N - 1 - i];
    else return taper64(i, N, a.margin_px);
}

template <int N> __host__ __device__ constexpr size_t p64_smem() { return (size_t)FftPlan<N>::BUF * sizeof(double2); }
// values per thread: 4 at N = 128 and 256 (a line has two warps or one; with eight values per thread
// and 256 lines the SMs had one or two warps each, and the FP64 pipe was 33 % busy), 8 up to
// N = 1024 (four were 4 % slower at 512: more FP64 operations, and the lines fill the SMs).  Below 128 what
// has a plan: 4 at 64, 16 at 32 (eight values of 32- and 64-point lines leave stages that fft_stage refuses), 8 at 16.
template <int N> __host__ __device__ constexpr int p64_ept() {
    return N >= 64 && N <= 256 ? 4 : (N == 32 || N > 1024 ? 16 : 8);
}

template <int N, bool TAB>
__global__ void __launch_bounds__(FftPlan<N, p64_ept<N>()>::T) prop64_rows_kernel(Prop64Args a) {
    begin_pass<N>();
    constexpr int EPT = p64_ept<N>();
    using Pl = FftPlan<N, EPT>;
    constexpr int T = Pl::T, E = Pl::E;
    extern __shared__ double2 smem64[];
    const int y = blockIdx.x, t = threadIdx.x;
    const double sfy = taper_of<N, TAB>(a, y);
    double2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int x = t + m * T;
        double sn, cs;
        sincos(a.phi[(size_t)y * N + x] * a.scale, &sn, &cs);
        const double w = sfy * taper_of<N, TAB>(a, x);
        v[m] = make_double2(w * cs, w * sn);
    }
    fft_line<double2, N, -1, EPT, 1, 0>(v, smem64, t, a.tw);
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = cmul(v[m], transfer_of<N, TAB>(a, t + m * T));
    fft_line<double2, N, +1, EPT, 1, 0>(v, smem64, t, a.tw);
#pragma unroll
    for (int m = 0; m < E; ++m) a.field[(size_t)y * N + t + m * T] = v[m];
}

template <int N, bool TAB>
__global__ void __launch_bounds__(FftPlan<N, p64_ept<N>()>::T) prop64_cols_kernel(Prop64Args a) {
    begin_pass<N>();
    constexpr int EPT = p64_ept<N>();
    using Pl = FftPlan<N, EPT>;
    constexpr int T = Pl::T, E = Pl::E;
    extern __shared__ double2 smem64[];
    const int x = blockIdx.x, t = threadIdx.x;
    double2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = a.field[(size_t)(t + m * T) * N + x];
    fft_line<double2, N, -1, EPT, 1, 0>(v, smem64, t, a.tw);
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = cmul(v[m], transfer_of<N, TAB>(a, t + m * T));
    fft_line<double2, N, +1, EPT, 1, 0>(v, smem64, t, a.tw);
#pragma unroll
    for (int m = 0; m < E; ++m) a.intensity[(size_t)(t + m * T) * N + x] = v[m].x * v[m].x + v[m].y * v[m].y;
}

template <int N, bool TAB>
cudaError_t launch_passes64(const Prop64Args& a, cudaStream_t s) {
    cudaError_t e = set_smem(prop64_rows_kernel<N, TAB>, p64_smem<N>());
    if (e == cudaSuccess) e = set_smem(prop64_cols_kernel<N, TAB>, p64_smem<N>());
    if (e != cudaSuccess) return e;
    constexpr int T = FftPlan<N, p64_ept<N>()>::T;
    if constexpr (TAB) {
        e = launch_pass<N>(1, prop64_rows_kernel<N, TAB>, dim3(N), dim3(T), p64_smem<N>(), s, a);
    } else {    // the kernel before may be the one that fills the twiddles (begin_after_previous)
        prop64_rows_kernel<N, TAB><<<N, T, p64_smem<N>(), s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    return launch_pass<N>(1, prop64_cols_kernel<N, TAB>, dim3(N), dim3(T), p64_smem<N>(), s, a);
}

cudaError_t launch_prop64(const Prop64Args& args, void* tables, cudaStream_t s) {
    return dispatch_n(args.n, [&](auto nc) -> cudaError_t {
        constexpr int N = decltype(nc)::value;
        if constexpr (N > kMax64N) {
            return cudaErrorNotSupported;
        } else {
            Prop64Args a = args;
            if (!tables) return launch_passes64<N, false>(a, s);
            double2* h = static_cast<double2*>(tables);
            double* sf = reinterpret_cast<double*>(h + N / 2 + 1);
            static_assert((N / 2 + 1) * sizeof(double2) + N / 2 * sizeof(double) <= N * sizeof(double2), "tables fit");
            const cudaError_t e = launch_next(prop64_tables_kernel, dim3((N / 2 + 32) / 32), dim3(32), 0, s, a, h, sf);
            if (e != cudaSuccess) return e;
            a.h = h;
            a.sf = sf;
            return launch_passes64<N, true>(a, s);
        }
    });
}

}  // namespace scint
