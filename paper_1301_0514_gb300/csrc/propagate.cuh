// Block shapes and layouts shared by the propagation passes and their adjoints.
#pragma once

#include "fft.cuh"
#include "kernels.cuh"

namespace scint {

constexpr int kColEPT = 16;   // values per thread in the column passes
constexpr size_t kMaxSmem = 227 * 1024;

// Lines longer than one block's shared memory (N = 16384) go to a cluster of two
// blocks, split by one radix-2 step: each block transforms one parity, as two half lines (prop_*_split_kernel in
// propagate.cu) or as a whole N/2-point line (conj_*_split_kernel there, adj_*_split_kernel in adjoint.cu).
// The kernels below are the unsplit passes.
template <int N> __host__ __device__ constexpr int pcs() { return N >= kSplitN ? 2 : 1; }

// rows per row-pass block, columns per column-pass block (all lines of a block
// are transformed together); threads are per block
template <int N> __host__ __device__ constexpr int prow_lines() { return N >= kTileRow32 ? 1 : (kTileRow32 / N < N ? kTileRow32 / N : N); }
template <int N> __host__ __device__ constexpr int prow_threads() { return prow_lines<N>() * FftPlan<N>::T; }
// Column-pass blocks take 256 threads (two blocks per SM, so a stage barrier idles
// half the SM, not all of it) wherever a block still holds two or more columns of
// a strip; at N = 4096 that would leave one column (a quarter of every 32-byte
// sector read), so there a block holds two columns in 512 threads.
template <int N> __host__ __device__ constexpr int pcol_lines() {
    return N >= 8192 ? 1 : (N >= 4096 ? 2 : (4096 / N < N ? 4096 / N : N));
}
template <int N> __host__ __device__ constexpr int pcol_threads() { return pcol_lines<N>() * FftPlan<N, kColEPT>::T; }
// Strip width of the intermediate: at least 4 columns, so that every row of the
// row pass writes whole 32-byte sectors; a column block then reads its
// pcol_lines() columns out of one strip (sibling blocks share the sectors in L2).
template <int N> __host__ __device__ constexpr int pstrip() { return pcol_lines<N>() >= 4 ? pcol_lines<N>() : (N >= 4 ? 4 : N); }

template <int N> constexpr size_t ptws_bytes(int twm) { return twm == 1 ? (size_t)FftPlan<N>::TWS * sizeof(float2) : 0; }
template <int N> constexpr size_t prow_smem() {
    return (size_t)prow_lines<N>() * (FftPlan<N>::BUF * sizeof(float2) + N * sizeof(long long));
}
// Transfer-function column blocks of these sizes give each column a team of threads with a barrier and a line buffer
// of its own, so that one column's line exchanges run beside another's butterflies; in smaller
// blocks (and at 8192, one column per block) the columns are interleaved across the lanes and share
// the block's barriers.
template <int N> __host__ __device__ constexpr bool col_teams() { return N >= 512 && N <= 4096; }
// column pass: line buffers and, without teams, the twiddle table when it fits
template <int N> __host__ __device__ constexpr size_t pcol_base_bytes() {
    return (size_t)pcol_lines<N>() * FftPlan<N>::BUF * sizeof(float2);
}
// Twiddles of the column passes (fft.cuh): register bases and their products (2) in the teams, which share no barrier
// that a table's making could use, and where the table does not fit; else the block's shared table (1).  The row passes take bases.
template <int N, bool CONJ> __host__ __device__ constexpr int pcol_twm() {
    return (!CONJ && col_teams<N>()) || pcol_base_bytes<N>() + (size_t)FftPlan<N>::TWS * sizeof(float2) > kMaxSmem ? 2 : 1;
}
// Below 512 a block's columns evaluate H_x once per block and wavelength into shared memory: with two tables there,
// and no barrier of their own, that is less than the latency of a table's loads behind the forward transform, which few
// blocks and warps hide (32 wavelengths at 64^2, the whole call: 145 us with tables in memory, 143 when each element
// took its own hardware sine, 133 so; at 256^2 149, 148 and 140).
template <int N, bool CONJ> __host__ __device__ constexpr bool own_transfer() { return !CONJ && N < 512; }
template <int N> __host__ __device__ constexpr int own_entries() { return N / 2 + 1; }
template <int N, bool CONJ = false> constexpr size_t pcol_smem() {
    return pcol_base_bytes<N>() + ptws_bytes<N>(pcol_twm<N, CONJ>()) +
           (own_transfer<N, CONJ>() ? 2 * own_entries<N>() * sizeof(float2) : 0);
}

// signed FFT frequency index of bin i
SCINT_DEV int sfreq(int i, int n) { return i < n / 2 ? i : i - n; }

// element (y, x) of a strip-layout field
template <int WL> SCINT_DEV size_t strip_index(int y, int x, int n) {
    return (size_t)(x / WL) * n * WL + (size_t)y * WL + (x % WL);
}

// phi (radians) -> 64-bit fixed-point turns, P = round(phi 2^32 / 2 pi)
SCINT_DEV long long phase_fixed(double phi) { return __double2ll_rn(phi * (4294967296.0 / (2.0 * kPi))); }
// The same for E values of a thread, P(m) = phase_fixed(phi(m)).  Below 2^21 rad the product is
// rounded to an integer by the one FP64 addition of 1.5 2^52 it is fused with, and the integer is read
// from the sum's bits: one instruction on the narrow FP64 pipe instead of a product and a conversion
// (16 cycles of an SM per warp each; the row pass at one wavelength 0.142 -> 0.110 ms at 4096^2).
// Rounded once instead of twice, the two differ next to a tie only, by 2^-32 turns.
template <int E, typename Load, typename Store>
SCINT_DEV void phases_fixed(Load&& load, Store&& store) {
    double f[E];
    unsigned top = 0;
#pragma unroll
    for (int m = 0; m < E; ++m) {
        f[m] = load(m);
        top = max(top, (unsigned)__double2hiint(f[m]) & 0x7FFFFFFFu);
    }
    if (top < 0x41400000u) {    // |phi| < 2^21 for every value
        const double k = 4294967296.0 / (2.0 * kPi), magic = 0x1.8p52;
#pragma unroll
        for (int m = 0; m < E; ++m) store(m, __double_as_longlong(fma(f[m], k, magic)) - 0x4338000000000000ll);
    } else {                    // large phases, infinities, NaN
#pragma unroll
        for (int m = 0; m < E; ++m) store(m, phase_fixed(f[m]));
    }
}

// exp(i (phi s + add 2^-64 turns)) from P and S = round(s 2^32): the low 64
// bits of P S are the fractional turns of phi s times 2^64 (exact reduction
// mod 2 pi); the angle in [-pi, pi) goes to the hardware sine/cosine (abs.
// error ~4e-7 there).
SCINT_DEV float2 unit_phasor(long long P, unsigned long long S, unsigned long long add = 0ull) {
    const unsigned long long prod = (unsigned long long)P * S + add;   // + extra turns 2^-64
    const float ang = (float)(int)(prod >> 32) * (float)(2.0 * kPi * 0x1.0p-32);
    float sn, cs;
    __sincosf(ang, &sn, &cs);
    return make_float2(cs, sn);
}

// H_x(k) = exp(-i pi lambda z k^2) at FFT index i, from C = frac(-lambda z / 2L^2) 2^64:
// the phase C m^2 mod 2^64 (m the signed frequency index) is exact in fixed-point turns.
SCINT_DEV float2 transfer_phasor(unsigned long long C, int i, int n) {
    const long long m = sfreq(i, n);
    return unit_phasor(0, 0ull, C * (unsigned long long)(m * m));
}
// The same for the signed index m, |m| < 2^15: the upper 32 bits of C m^2 mod 2^64 are all that the
// angle takes, so 32-bit products do (the same bits).  The row passes up to 8192 evaluate H_x so: their
// load/store pipe is the busier one, and a table in shared memory had cost 2-4 % of them with 32
// wavelengths (8192, from global memory: 12 %).
SCINT_DEV float2 transfer_fast(unsigned long long C, int m) {
    const unsigned mm = (unsigned)(m * m);
    const unsigned hi = __umulhi((unsigned)C, mm) + (unsigned)(C >> 32) * mm;
    float sn, cs;
    __sincosf((float)(int)hi * (float)(2.0 * kPi * 0x1.0p-32), &sn, &cs);
    return make_float2(cs, sn);
}
// The same to FP32 accuracy, for the column passes' tables and the 16384-point lines (TableArgs; ~25
// instructions where there is no table): the turns are reduced to an eighth of a turn around a quarter turn
// before the sine and cosine.  The hardware sine's absolute error of 4e-7, once for the screen
// and once for each axis, is the larger part of the passes' error; without it on one axis the
// intensities' error against 64 bits is below what it was with twiddles from the exact table in the
// columns and one factorisation less in the long lines (one wavelength at 4096^2: 8.9e-7 -> 8.2e-7, 48 screens 8.0e-7 -> 7.1e-7).
SCINT_DEV float2 transfer_signed(unsigned long long C, int m) {
    const unsigned mm = (unsigned)(m * m);
    const int turns = (int)(__umulhi((unsigned)C, mm) + (unsigned)(C >> 32) * mm);
    const unsigned q = ((unsigned)turns + 0x20000000u) >> 30;
    float sn, cs;
    sincospif((float)(int)((unsigned)turns - (q << 30)) * 0x1.0p-31f, &sn, &cs);
    const float re = q & 1u ? sn : cs, im = q & 1u ? cs : sn;    // times i^q
    return make_float2(q == 1u || q == 2u ? -re : re, q >= 2u ? -im : im);
}
// signed frequency index of element t + m T of a line of N = E T values, t < T
template <int N, int E> SCINT_DEV int signed_index(int t, int m) {
    return t + m * (N / E) - (2 * m >= E ? N : 0);
}
// its entry in a half table, |signed_index|
template <int N, int E> SCINT_DEV int half_index(int t, int m) {
    return 2 * m >= E ? N - (t + m * (N / E)) : t + m * (N / E);
}
// H_x(k)/n (the inverse transform's normalisation)
SCINT_DEV float2 transfer_at(unsigned long long C, int i, int n) { return transfer_phasor(C, i, n) * (1.0f / n); }

// One-FFT mode: chirp |x_1|^2 / (2 R_F^2) with x_1 = (i - n/2) Delta in fixed-point
// turns, C (i - n/2)^2 mod 2^64 (exact), plus half a turn for odd i: the factor
// (-1)^i that centres the transform on the optical axis (the sum over
// (i - n/2)(k - n/2) is the plain DFT times (-1)^(i + k) and a constant).
SCINT_DEV unsigned long long chirp_turns(unsigned long long C, int i, int n) {
    const long long d = (long long)i - n / 2;
    return C * (unsigned long long)(d * d) + ((unsigned long long)(i & 1) << 63);
}

}  // namespace scint
