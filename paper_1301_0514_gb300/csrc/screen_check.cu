// Screen check of Sect. 3.1.1: the phase spectrum and structure function
// recomputed from the generated F_phi, and R_diff^rec.
//
//   S_rec(q_j) = sum_{annulus j} |F|^2 / (count_j L^2), annulus j = bins with
//                j - 1/2 <= |m| < j + 1/2 (nearest integer to |m|);
//   D_rec(r)   = 2 (xi_rec(0) - xi_rec(r)) with Eq. crec on the annuli,
//              = 4 pi dq sum_{j=1}^{J} q_j S_rec(q_j) (1 - J0(2 pi q_j r)),
//                q_j = j dq, dq = 1/L, J = min(n_bins - 1, N/2) (q_max = 1/(2 Delta));
//   R_diff^rec = root of D_rec(R) = 1, bisection on (0, L/2].
//
// The annulus sums run as one persistent pass: each block keeps a histogram of
// every annulus in shared memory, its warps walk one octant of the spectrum (radial_kernel
// below), and the block adds its histogram into the global one at the end.  The sums are 64-bit
// fixed point (see annulus_shift), hence exact and independent of the order of the additions;
// outside the FP64 square the loop has no FP64 operation (GB300's FP64 pipe is narrow).  The noise is
// regenerated per bin (spectrum.cuh), never stored.  The root takes a few launches (bisect_kernel);
// within one the blocks' partial sums are combined in a fixed order by the
// last block to finish, so the result does not depend on scheduling.
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>
#include <math_constants.h>

#include "dispatch.cuh"
#include "kernels.cuh"
#include "spectrum.cuh"

namespace scint {

// Nearest integer to sqrt(m2), exactly: j with j^2 - j + 1 <= m2 <= j^2 + j.
// m2 <= 2 (N/2)^2 < 2^31 for N <= 32768, so 32-bit integers suffice (64-bit
// conversions would run on the narrow FP64 pipe).
SCINT_DEV int annulus_of(int m2) {
    // any estimate within +-1 will do: the integer tests below make j exact
    const float f = (float)m2;
    int j = m2 > 0 ? __float2int_rn(f * rsqrtf(f)) : 0;
    while (j * j + j < m2) ++j;
    while (j > 0 && j * j - j + 1 > m2) --j;
    return j;
}

// Annulus sums in 64-bit fixed point.  Annulus j's values are scaled by 2^s_j
// with s_j chosen so that the expected bin power amp^2 j^-beta lands in
// [2^36, 2^37); a bin holds at most ~120 times that (the -2 ln u tail and the
// spread of |m| within an annulus) and an annulus at most ~1.5e5 bins, so a sum
// stays below 2^62.  Truncating each value to the fixed-point grid costs at
// most 2^-36 of the annulus' scale per bin.  Integer sums are exact, so the
// result does not depend on the order of the additions.
// Any shift near the target range is valid as long as the sums and the final
// normalisation use the same one, so the fast hardware log2 serves (the same
// j gives the same shift in every kernel).
SCINT_DEV int annulus_shift(const SynthArgs& a, int j) {
    const float l2 = 2.0f * __log2f(a.amp32) + 4.0f * a.neg_beta_4_32 * __log2f((float)max(j, 1));
    return 36 - (int)floorf(l2);
}
// v 2^s truncated to an integer, from the bits of a positive normal float / double
SCINT_DEV unsigned long long to_fixed(float v, int s) {
    const uint32_t b = __float_as_uint(v);
    if ((b >> 23) == 0u) return 0ull;
    const int e = (int)(b >> 23) - 150 + s;
    const unsigned long long m = (b & 0x7FFFFFu) | 0x800000u;
    return e >= 0 ? m << e : (e > -24 ? m >> -e : 0ull);
}
SCINT_DEV unsigned long long to_fixed(double v, int s) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if ((b >> 52) == 0ull) return 0ull;
    const int e = (int)(b >> 52) - 1075 + s;
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    return e >= 0 ? m << e : (e > -53 ? m >> -e : 0ull);
}

// The bins of one octant, 0 <= ax <= ay <= n/2 (a = |m|), stand for the whole grid: up to eight
// bins (+-ax, +-ay), (+-ay, +-ax) share |m|^2 and so the annulus, its shift and the amplitude
// (one index search, one powf and one log2 per eight bins; the noise of each bin stays its own).
// A warp takes 32 R cells of a spectral row ay, each lane R of them in a row, in the
// direction in which the annulus changes slowly (at most 0.71 per cell), and adds a run of
// cells of one annulus in a register before it goes to the block's shared histogram.  The sums
// are the same integers as bin by bin.  At n = 14000: sums 2.16 -> 1.14 ms (328 -> 176 warp
// instructions per 32 bins; Philox and the two branches of -ln u remain, issue 76 %), counts
// 0.35 -> 0.07 ms, against whole rows per block and a powf and an annulus search per bin.  The rows ay <= low_k,
// drawn in FP64, go first and cell by cell (radial_square).
// R = 4, or 1 while that leaves warps without a task (1000^2: 51 -> 38 us).
constexpr int kRun = 4;

// number of (row, segment) tasks of rows 0..h
template <int R> __host__ __device__ constexpr int radial_tasks(int h) {
    constexpr int kSeg = 32 * R;
    const int G = h / kSeg;
    return kSeg * (G * (G + 1) / 2) + (h + 1 - G * kSeg) * (G + 1);
}
// task -> (row ay, first cell): rows [g kSeg, (g + 1) kSeg), kSeg = 32 R, have g + 1 segments each
template <int R> SCINT_DEV void radial_task(int task, int& ay, int& ax0) {
    constexpr int kSeg = 32 * R;
    int g = (int)((sqrtf(8.0f * ((float)task / kSeg) + 1.0f) - 1.0f) * 0.5f);
    while (kSeg * ((g + 1) * (g + 2) / 2) <= task) ++g;
    while (kSeg * (g * (g + 1) / 2) > task) --g;
    const int rem = task - kSeg * (g * (g + 1) / 2);
    ay = g * kSeg + rem / (g + 1);
    ax0 = (rem % (g + 1)) * kSeg;
}

// The octant's rows 0..min(low_k, n/2), whose bins are drawn in FP64: a cell per group of G lanes (1, 2, 4 or 8),
// which share its up to eight draws.  In runs of four cells per lane the chain of 32 logarithms took 50 us, longer
// than the whole sums of a small grid.
__host__ __device__ constexpr int square_cells(int rows) { return rows * (rows + 1) / 2; }
// Lanes per cell: a draw costs about 30 instructions on the FP64 pipe and a cell's amplitude 70, repeated by each
// of its lanes; so many lanes while latency counts, one when the pipe is full.
inline int square_lanes(int cells) { return cells <= 4096 ? 8 : (cells <= 12288 ? 4 : (cells <= 16384 ? 2 : 1)); }
SCINT_DEV void radial_square(const SynthArgs& a, int rows, int n_hist, int G, unsigned long long* hs) {
    const int n = a.n, h = n / 2, cells = square_cells(rows);
    const int lane = threadIdx.x & 31, g = lane & (G - 1);
    const int step = (int)gridDim.x * (kRadialThreads / 32) * (32 / G);
#pragma unroll 1
    for (int c0 = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * (32 / G); c0 < cells; c0 += step) {
        const int c = c0 + lane / G;
        unsigned long long acc = 0ull;
        int j = n_hist;
        if (c < cells) {
            int ay = (int)((sqrtf(8.0f * (float)c + 1.0f) - 1.0f) * 0.5f);
            while (square_cells(ay + 1) <= c) ++ay;
            while (square_cells(ay) > c) --ay;
            const int ax = c - square_cells(ay), m2 = ax * ax + ay * ay;
            j = annulus_of(m2);
            if (j < n_hist && m2 > 0) {
                const int shift = annulus_shift(a, j);
                const double sig = amplitude_low(a, m2), sig2 = sig * sig;
#pragma unroll 1
                for (int d = g; d < 8; d += G) {
                    // (ax, ay) or (ay, ax), then the mirror bins in y (d & 2) and x (d & 1): 0 and -n/2 have none
                    const int px = d < 4 ? ax : ay, py = d < 4 ? ay : ax;
                    if ((d >= 4 && ax == ay) || ((d & 2) && (py == 0 || py == h)) || ((d & 1) && (px == 0 || px == h))) continue;
                    const u32x4 w = bin_words(a, d & 1 ? n - px : px, d & 2 ? n - py : py);
                    acc += to_fixed(sig2 * (2.0 * neg_log_ua64(w)), shift);
                }
            }
        }
        for (int o = 1; o < G; o *= 2) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (g == 0 && j < n_hist) atomicAdd(hs + j, acc);
    }
}

// COUNT: bins per annulus.  Otherwise: fixed-point sums of |F|^2 (high bins from
// their FP32 value, low bins from their FP64 value, as the synthesis draws them).
template <bool COUNT, int R>
__global__ void __launch_bounds__(kRadialThreads)
radial_kernel(SynthArgs a, int n_hist, int square_group, unsigned long long* sums, unsigned long long* counts) {
    extern __shared__ __align__(16) unsigned char radial_smem[];
    unsigned long long* hs = reinterpret_cast<unsigned long long*>(radial_smem);
    unsigned* hc = reinterpret_cast<unsigned*>(radial_smem);
    for (int j = threadIdx.x; j < n_hist; j += blockDim.x) {
        if (COUNT) hc[j] = 0u;
        else hs[j] = 0ull;
    }
    __syncthreads();
    const int n = a.n, h = n / 2;
    // row ay has no annulus below ay
    const int top = min(h, n_hist), square = min(a.low_k, top);
    const int tasks = radial_tasks<R>(top), lane = threadIdx.x & 31;
    const int warps = gridDim.x * (kRadialThreads / 32);
    if (!COUNT) radial_square(a, square + 1, n_hist, square_group, hs);
    const int first = COUNT ? 0 : radial_tasks<R>(square);    // the rows above the square
#pragma unroll 1
    for (int task = first + (threadIdx.x >> 5) * gridDim.x + blockIdx.x; task < tasks; task += warps) {
        int ay, ax0;
        radial_task<R>(task, ay, ax0);
        ax0 += lane * R;
        int cur = -1, shift = 0;
        unsigned long long acc = 0ull;
        unsigned cnt = 0u;
        // frequency -h and its mirror are one bin, and so is 0
        const bool two_y = ay != 0 && ay != h;
#pragma unroll 1
        for (int i = 0; i < R; ++i) {
            const int ax = ax0 + i;
            if (ax > ay) break;
            const int m2 = ax * ax + ay * ay;
            const int j = annulus_of(m2);
            if (j != cur) {
                if (cur >= 0 && cur < n_hist) {
                    if (COUNT) atomicAdd(hc + cur, cnt);
                    else atomicAdd(hs + cur, acc);
                }
                cur = j;
                acc = 0ull;
                cnt = 0u;
                if (!COUNT) shift = annulus_shift(a, j);
            }
            const bool two_x = ax != 0 && ax != h;
            if (COUNT) {
                cnt += (two_x ? 2u : 1u) * (two_y ? 2u : 1u) * (ax != ay ? 2u : 1u);
            } else if (j < n_hist) {
                const float sig = amplitude_high(a, m2), sig2 = sig * sig;
                // (ax, ay) and, off the diagonal, (ay, ax); each with both signs of both
#pragma unroll 1
                for (int q = 0; q < (ax != ay ? 4 : 2); ++q) {
                    const int px = q < 2 ? ax : ay, py = q < 2 ? ay : ax;
                    const bool two_px = q < 2 ? two_x : two_y, two_py = q < 2 ? two_y : two_x;
                    if ((q & 1) && !two_py) continue;
                    const uint32_t ky = (uint32_t)((q & 1) ? n - py : py);
                    const u32x4 w = philox4x32_10(u32x4{(uint32_t)px, ky, a.screen_id, 0u}, a.key0, a.key1);
                    const u32x4 v = philox4x32_10(u32x4{(uint32_t)(n - px), ky, a.screen_id, 0u}, a.key0, a.key1);
                    acc += to_fixed(sig2 * (2.0f * neg_log_ua32(w)), shift);
                    if (two_px) acc += to_fixed(sig2 * (2.0f * neg_log_ua32(v)), shift);
                }
            }
        }
        if (cur >= 0 && cur < n_hist) {
            if (COUNT) atomicAdd(hc + cur, cnt);
            else atomicAdd(hs + cur, acc);
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < n_hist; j += blockDim.x) {
        if (COUNT) {
            if (hc[j]) atomicAdd(counts + j, (unsigned long long)hc[j]);
        } else {
            if (hs[j]) atomicAdd(sums + j, hs[j]);
        }
    }
}

// s_rec holds the fixed-point sums on entry (as integers); S_rec = sum 2^-s_j / count / L^2
__global__ void radial_finish_kernel(SynthArgs a, int n_hist, double inv_l2, double* s,
                                     const unsigned long long* counts) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_hist) return;
    const unsigned long long fx = reinterpret_cast<const unsigned long long*>(s)[j];
    s[j] = counts[j] ? ldexp((double)fx, -annulus_shift(a, j)) / (double)counts[j] * inv_l2 : 0.0;
}

template <int R>
static cudaError_t launch_radial(const SynthArgs& a, int n_hist, unsigned long long* sums, unsigned long long* counts,
                                 int blocks, cudaStream_t s) {
    const size_t bytes_s = (size_t)n_hist * sizeof(unsigned long long), bytes_c = (size_t)n_hist * sizeof(unsigned);
    cudaError_t e;
    if ((e = set_smem(radial_kernel<false, R>, bytes_s)) != cudaSuccess) return e;
    if ((e = set_smem(radial_kernel<true, R>, bytes_c)) != cudaSuccess) return e;
    const int group = square_lanes(square_cells(std::min(a.low_k, std::min(a.n / 2, n_hist)) + 1));
    radial_kernel<true, R><<<blocks, kRadialThreads, bytes_c, s>>>(a, n_hist, 0, sums, counts);
    radial_kernel<false, R><<<blocks, kRadialThreads, bytes_s, s>>>(a, n_hist, group, sums, counts);
    return cudaGetLastError();
}

cudaError_t launch_radial_spectrum(const SynthArgs& a, double inv_l2, int n_hist, double* s_rec,
                                   unsigned long long* counts, int blocks, cudaStream_t s) {
    unsigned long long* fx = reinterpret_cast<unsigned long long*>(s_rec);
    const bool runs = radial_tasks<kRun>(std::min(a.n / 2, n_hist)) >= blocks * (kRadialThreads / 32);
    const cudaError_t e = runs ? launch_radial<kRun>(a, n_hist, fx, counts, blocks, s) : launch_radial<1>(a, n_hist, fx, counts, blocks, s);
    if (e != cudaSuccess) return e;
    radial_finish_kernel<<<(n_hist + 255) / 256, 256, 0, s>>>(a, n_hist, inv_l2, s_rec, counts);
    return cudaGetLastError();
}

// ---- Eq. crec ------------------------------------------------------------------
// sum_{j = j0 + 1, j0 + 1 + stride, ...} q_j S_j (1 - J0(2 pi q_j r)) for this thread
SCINT_DEV double crec_terms(const double* __restrict__ s, int J, double dq, double r, int first, int stride) {
    double acc = 0.0;
    for (int j = first; j <= J; j += stride) {
        const double q = j * dq;
        acc += q * s[j] * (1.0 - j0(2.0 * kPi * q * r));
    }
    return acc;
}

// block sum in a fixed order (the result is the same on every run)
SCINT_DEV double block_sum_fixed(double v, double* red) {
    red[threadIdx.x] = v;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const double t = red[0];
    __syncthreads();
    return t;
}

// A lag's terms in kCrecParts parts: thread t of part k takes j = 1 + 256 k + t, then every 2048th.  The parts'
// sums are added in the order of k, whichever blocks formed them, so a lag's bits do not depend on the call's
// other lags.  One block per lag, or a cluster when the lags leave SMs idle (launch_crec).
__global__ void __launch_bounds__(kCrecThreads) crec_kernel(CrecArgs a, const double* r_km, double* d) {
    static_assert(kCrecThreads == 32 * kCrecParts, "a warp per part");
    __shared__ double red[kCrecParts][kCrecThreads];
    __shared__ double part[kCrecParts];
    auto cl = cooperative_groups::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank(), i = (int)blockIdx.x / C;
    const int t = threadIdx.x;
    const int parts = min(kCrecParts, (a.J + kCrecThreads - 1) / kCrecThreads);    // the others have no term
    const double r = r_km[i];
#pragma unroll 1
    for (int k = rank; k < parts; k += C)
        red[k][t] = crec_terms(a.s, a.J, a.dq, r, 1 + k * kCrecThreads + t, kCrecParts * kCrecThreads);
    __syncthreads();
    // warp w adds up part w (reducing after every part was 6 % slower with 2048 terms)
    const int w = t / 32, lane = t % 32;
    if (w < parts && w % C == rank) {
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < kCrecThreads / 32; ++k) v += red[w][32 * k + lane];
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) part[w] = v;
    }
    if (C > 1) cl.sync();
    else __syncthreads();
    if (rank == 0 && t == 0) {
        double tot = 0.0;
        for (int k = 0; k < parts; ++k) tot += C > 1 ? *cl.map_shared_rank(&part[k], k % C) : part[k];
        d[i] = 4.0 * kPi * a.dq * tot;
    }
    if (C > 1) cl.sync();    // no block leaves before its parts are read
}

// Blocks per lag.  7000 J0 terms keep one SM's narrow FP64 pipe busy for 0.14 ms, so up to two lags per three
// SMs go to a cluster of as many blocks as there are parts with terms (at most 8).  From there on the lags fill
// the SMs by themselves, and the idle threads and barriers of a cluster cost more than the spread gives.  One block /
// a cluster of eight, us: 48 lags of 7000 terms 146 / 56, 152 lags 146 / 194; 1000 lags of 128 terms 31 / 140.
cudaError_t launch_crec(const CrecArgs& a, const double* r_km, int n_r, double* d, cudaStream_t s) {
    int dev = 0, sms = 0, cs = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (n_r <= sms * 2 / 3)
        while (cs < kCrecParts && cs * kCrecThreads < a.J) cs *= 2;
    return launch_k(crec_kernel, cs, dim3(n_r * cs), dim3(kCrecThreads), 0, s, a, r_km, d);
}

// ---- R_diff^rec: bisection of D_rec(R) = 1 on (0, L/2] ------------------------------
// Round by round.  A bisection round evaluates D_rec at the midpoint of the bracket and at both
// midpoints that may follow, each over its share of the blocks, and then takes two bisection
// steps: the decisions are those of one step at a time.  Once the bracket is so narrow that every
// term is smooth over it (q_max times its half width below pi/64 rad), a last round
// evaluates D_rec at the eight Chebyshev nodes of the bracket and bisects the polynomial
// through them (interpolation error below (pi/64)^8 / (8! 2^7) < 1e-17 of D's terms) down to
// the resolution of the 64 steps.  At n = 14000: 9 rounds and the last, 13 us each, where one launch
// per bisection step with a serial sum of its blocks' partials took 65 x 16 us.  More steps per round
// do not pay: a D_rec costs the whole GPU's FP64 pipes 1 us (J = 7000), a round's latency is 10.
constexpr int kNodes = 8;
struct NodeCos { double c[4 * kNodes]; };    // cos(pi j / 16)

// The first round also evaluates D_rec(L/2), which decides whether there is a root.
template <bool LAST>
__global__ void __launch_bounds__(kCrecThreads) bisect_kernel(CrecArgs a, BisectState* st, int first, int points,
                                                            int iterations, NodeCos nc, double* out) {
    __shared__ double red[kCrecThreads];
    __shared__ double D[kNodes];
    __shared__ bool is_last;
    const double lo = first ? 0.0 : st->lo, hi = first ? a.half_L : st->hi;
    const bool none = first ? false : st->no_root != 0;
    if (none) {    // uniform across the grid: nothing left to do
        if (LAST && blockIdx.x == 0 && threadIdx.x == 0) *out = CUDART_NAN;
        return;
    }
    const double mid = 0.5 * (lo + hi), half = 0.5 * (hi - lo);
    const int per = gridDim.x / points, pt = blockIdx.x / per, b = blockIdx.x % per;
    double r;
    if (LAST) r = fma(half, nc.c[2 * pt + 1], mid);
    else r = pt == 0 ? 0.5 * (lo + mid) : (pt == 1 ? mid : (pt == 2 ? 0.5 * (mid + hi) : a.half_L));
    const double acc = crec_terms(a.s, a.J, a.dq, r, 1 + b * (int)blockDim.x + (int)threadIdx.x, per * (int)blockDim.x);
    const double t = block_sum_fixed(acc, red);
    if (threadIdx.x == 0) {
        st->partial[blockIdx.x] = t;
        __threadfence();
        is_last = atomicAdd(&st->arrived, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    // warp w adds the partials of point w (fixed order)
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w < points) {
        double v = 0.0;
        for (int k = lane; k < per; k += 32) v += __ldcg(&st->partial[w * per + k]);
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) D[w] = 4.0 * kPi * a.dq * v;
    }
    __syncthreads();
    if (w != 0) return;
    if constexpr (!LAST) {
        if (lane == 0) {
            double l = lo, h = hi;
            if (D[1] < 1.0) {
                l = mid;
                if (D[2] < 1.0) l = 0.5 * (mid + hi);
                else h = 0.5 * (mid + hi);
            } else {
                h = mid;
                if (D[0] < 1.0) l = 0.5 * (lo + mid);
                else h = 0.5 * (lo + mid);
            }
            st->lo = l;
            st->hi = h;
            if (first) st->no_root = D[3] < 1.0;
            st->arrived = 0u;
        }
    } else {
        // Chebyshev coefficients of D over the bracket, then 5 bisection steps at a time: lane j holds
        // the polynomial at the j-th of 32 equal parts of the bracket (u in [-1, 1])
        double c[kNodes];
#pragma unroll
        for (int k = 0; k < kNodes; ++k) {
            double v = 0.0;
#pragma unroll
            for (int i = 0; i < kNodes; ++i) v = fma(D[i], nc.c[(k * (2 * i + 1)) % (4 * kNodes)], v);
            c[k] = v * (k == 0 ? 1.0 / kNodes : 2.0 / kNodes);
        }
        double ul = -1.0, uh = 1.0;
#pragma unroll 1
        for (int k = 0; k < iterations; k += 5) {
            const double u = fma(uh - ul, lane * 0.03125, ul);
            double b1 = 0.0, b2 = 0.0;     // Clenshaw's recurrence
#pragma unroll
            for (int q = kNodes - 1; q >= 1; --q) {
                const double b0 = fma(2.0 * u, b1, c[q] - b2);
                b2 = b1;
                b1 = b0;
            }
            const unsigned below = __ballot_sync(0xffffffffu, fma(u, b1, c[0] - b2) < 1.0);
            int l = 0, h = 32;
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                const int m = (l + h) / 2;
                if ((below >> m) & 1u) l = m;
                else h = m;
            }
            const double d = uh - ul, base = ul;
            ul = fma(d, l * 0.03125, base);
            uh = fma(d, h * 0.03125, base);
        }
        if (lane == 0) *out = fma(half, 0.5 * (ul + uh), mid);
    }
}

// bisection steps before the last round: the bracket's half width is then L/4 2^-steps with
// 2^steps >= 16 n (two steps per round)
static int bisect_steps(int n) {
    int steps = 0;
    while ((1ll << steps) < 16ll * n) ++steps;
    return steps + (steps & 1);
}
int bisect_launches(int n) { return bisect_steps(n) / 2 + 1; }

cudaError_t launch_bisect(const CrecArgs& a, BisectState* st, int n, int iterations, double* out, cudaStream_t s) {
    NodeCos nc;
    for (int j = 0; j < 4 * kNodes; ++j) nc.c[j] = std::cos(kPi * j / (2.0 * kNodes));
    const int steps = bisect_steps(n);
    cudaError_t e = cudaMemsetAsync(st, 0, sizeof(BisectState), s);
    for (int k = 0; k < steps && e == cudaSuccess; k += 2) {
        const int points = k == 0 ? 4 : 3;
        bisect_kernel<false><<<kBisectBlocks / points * points, kCrecThreads, 0, s>>>(a, st, k == 0, points, 0, nc, out);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    bisect_kernel<true><<<kBisectBlocks / kNodes * kNodes, kCrecThreads, 0, s>>>(a, st, 0, kNodes, iterations - steps, nc, out);
    return cudaGetLastError();
}

}  // namespace scint
