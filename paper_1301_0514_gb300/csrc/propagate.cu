// Fresnel propagation of a phase screen by the transfer function (Eq. hxy)
// with the edge taper of Sect. 3.2.1 and passband co-addition (Sect. 3.2.4).
//
// The transfer function H(k) = exp(-i pi lambda z (kx^2 + ky^2)) factors into
// H_x(kx) H_y(ky), so the 2D propagator is a 1D propagator along x followed by
// one along y.  Each 1D propagator is FFT -> multiply -> inverse FFT on a line
// held in registers and shared memory, so a wavelength costs two HBM passes:
//   row pass:    phi (read once per wavelength group) -> exact phase reduction
//                -> sin/cos -> taper -> FFT_x -> H_x/N -> IFFT_x -> field (write);
//                H_x and H_y come from one scalar per wavelength (no table
//                loads), their phases exact in fixed-point turns like the screen phase
//   column pass: field (read) -> FFT_y -> H_y/N -> IFFT_y -> w |A|^2, summed over
//                the group in registers -> intensity (one write per group)
//
// Phase reduction: phi is converted once per pixel to 64-bit fixed point in
// turns, P = round(phi 2^32 / 2 pi); for each wavelength the low 64 bits of
// P * round(s 2^32) (s = lambda_ref / lambda) are the fractional turns of
// phi s scaled by 2^64, so the reduction modulo 2 pi is exact integer
// arithmetic (error |phi s| 2^-33 / 2 pi turns from rounding s) and only the
// reduced angle goes to the FP32 sine/cosine.
#include <algorithm>

#include "dispatch.cuh"
#include "prop_body.cuh"
#include "propagate.cuh"
#include "stream.cuh"

namespace scint {

// ---- tables ---------------------------------------------------------------------
// raised-sine taper SF at the pixel centre (i + 1/2), symmetric about the centre
// (Sect. 3.2.1), and the transfer function
__global__ void prop_tables_kernel(const __grid_constant__ TableArgs a) {
    begin_after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int l = blockIdx.y, n = a.n, entries = transfer_entries(n);
    if (a.h && i < entries) {
        int m = i;    // the entry's frequency
        if (n > 4096) {
            if (n >= kSplitN) m = i < n / 2 ? 2 * i : 2 * (i - n / 2) + 1;
            if (m >= n / 2) m -= n;
        }
        a.h[(size_t)l * entries + i] = transfer_signed(a.h_fx[l], m);
    }
    if (i >= n) return;
    const double lm = a.margin_px[l];
    double sf = 1.0;
    if (lm > 0.0) {
        const double u = fmin((double)i + 0.5, (double)n - (double)i - 0.5);
        if (u <= lm) {
            const double sn = sinpi(u / (2.0 * lm));
            sf = sn * sn;
        }
    }
    a.sf[(size_t)l * n + i] = (float)sf;
}

cudaError_t launch_prop_tables(const TableArgs& a, cudaStream_t s) {
    dim3 grid((std::max(a.n, a.h ? transfer_entries(a.n) : 0) + 255) / 256, a.count);
    return launch_next(prop_tables_kernel, grid, dim3(256), 0, s, a);
}

template <int N, bool CONJ>
__global__ void __launch_bounds__(prow_threads<N>(), (prow_threads<N>() <= 256 ? 2 : 1))
prop_rows_kernel(PropArgs a) {
    extern __shared__ float2 smem32[];
    begin_pass<N>();
    prop_rows_body<N, CONJ>(a, blockIdx.x, threadIdx.x, smem32);
}

template <int N, bool CONJ>
__global__ void __launch_bounds__(pcol_threads<N>(), (pcol_threads<N>() <= 256 ? 2 : 1))
prop_cols_kernel(PropArgs a) {
    extern __shared__ float2 smem32[];
    begin_pass<N>();
    prop_cols_body<N, CONJ>(a, blockIdx.x, threadIdx.x, smem32);
}

// ---- streamed passes (rows, and columns of the transfer function, 512 to 4096) -------------
// The same arithmetic with the inputs of the next wavelength or line on their way while this one is
// transformed: without it every warp of a block waited for its loads at the same time, at the
// head of each wavelength.  The copies need neither registers nor load instructions (a copy by
// cp.async had cost more than it hid, on the load/store pipe that the line exchanges keep
// 60 % busy).  The passes are bound by issue slots (105-120 instructions per pixel and wavelength)
// and by the load/store pipe of the exchanges; per-launch times before and after (event pairs, which keep the launches
// apart), ms:
//                  32 wavelengths                          one wavelength
//          rows           columns               rows             columns
//   512    0.102 -> 0.080   0.084 -> 0.078      0.0112 -> 0.0111  0.0097 -> 0.0097
//   1024   0.176 -> 0.155   0.159 -> 0.139      0.0172 -> 0.0152  0.0139 -> 0.0142
//   2048   0.625 -> 0.573   0.573 -> 0.491      0.0449 -> 0.0317  0.0405 -> 0.0351
//   4096   2.504 -> 2.382   2.563 -> 2.519      0.1657 -> 0.1075  0.1619 -> 0.1308
// A whole call at one wavelength in a graph: 512^2 14.5 -> 13.2 us, 1024^2 24.6 -> 22.3.  There the former columns
// (interleaved lines, a shared twiddle table) with early launches take 13.4 and 22.1 us: no rule for that.
// The one-FFT columns keep plain loads: with half the transforms per value the copies of 16-byte
// rows became their bound (4096^2, 8 wavelengths: 0.493 ms, streamed 0.531).
//   Row pass: the block's phases by one bulk copy into the array that keeps their fixed-point
//   form (converted in place, each thread its own entries), the taper of each wavelength by
//   another; both are issued once the forward transform's barriers show that the block has read
//   what they overwrite.
//   Column pass: the block's columns of one wavelength as boxes of 16-byte rows, dense, into a stage
//   of their own; a team of threads per column (col_teams), twiddles from register bases, whose
//   products cost less than the table's loads once the columns do not share barriers (2048^2: 0.559 ms
//   with the table).
// With few wavelengths the blocks walk lines (walk_blocks).
template <int N> __host__ __device__ constexpr bool row_stream() { return N >= 512 && N <= 4096; }
template <int N> constexpr size_t prow_stream_smem() {
    return (size_t)prow_lines<N>() * (FftPlan<N>::BUF * sizeof(float2) + N * sizeof(long long)) + N * sizeof(float) + 24;
}

template <int N, bool CONJ>
__global__ void __launch_bounds__(prow_threads<N>(), (prow_threads<N>() <= 256 ? 2 : 1))
prop_rows_stream_kernel(PropArgs a, int bulk) {
    using Pl = FftPlan<N>;
    constexpr int T = Pl::T, E = Pl::E, B = prow_lines<N>(), W = pstrip<N>(), BUFL = Pl::BUF;
    extern __shared__ float2 smem32[];
    begin_pass<N>();
    const int team = threadIdx.x / T, t = threadIdx.x % T;
    float2* buf = smem32 + team * BUFL;
    long long* Pall = reinterpret_cast<long long*>(smem32 + B * BUFL);
    long long* P = Pall + team * N + t;
    float* sfs = reinterpret_cast<float*>(Pall + B * N);
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(sfs + N);    // phases, taper
    unsigned* reads = reinterpret_cast<unsigned*>(bar + 2);    // rows that have read the taper
    // below 2048 a row is a team with a barrier of its own (512^2: 3 % faster; at 2048 2 % slower)
    constexpr int SUB = N < 2048 ? T : 0;
    const int count = a.lam.count, tiles = N / B;
    auto load_phi = [&](int tile) {
        tile_expect(bar, B * N * sizeof(double));
        bulk_load(Pall, a.phi + (size_t)tile * (B * N), B * N * sizeof(double), bar);
    };
    auto load_sf = [&](int l) {
        tile_expect(bar + 1, N * sizeof(float));
        bulk_load(sfs, a.sf + (size_t)l * N, N * sizeof(float), bar + 1);
    };
    if (threadIdx.x == 0) {
        tile_init(bar);
        tile_init(bar + 1);
        *reads = 0u;
        tile_init_fence();
        if (bulk) load_phi(blockIdx.x);
        load_sf(0);
    }
    TwiddleRegs<float2, N, 16> tr;
    tr.load(a.tw, t);
    __syncthreads();
    unsigned phase = 0;    // bits: parity of the phases' copy, of the taper's
    bool ok = true;
#pragma unroll 1
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int y = tile * B + team;
        if (bulk) {
            ok = ok && wait_tile(bar, phase & 1);
            phase ^= 1;
            phases_fixed<E>([&](int m) { return __longlong_as_double(P[m * T]); }, [&](int m, long long p) { P[m * T] = p; });
            tile_reuse_fence();
        } else {
            phases_fixed<E>([&](int m) { return a.phi[(size_t)y * N + t + m * T]; }, [&](int m, long long p) { P[m * T] = p; });
        }
#pragma unroll 1
        for (int l = 0; l < count; ++l) {
            if (count > 1 || tile == (int)blockIdx.x) {
                ok = ok && wait_tile(bar + 1, phase >> 1);
                phase ^= 2;
            }
            const unsigned long long S = a.lam.scale_fx[l];
            // 1/N of the inverse transform on the taper of the row (prop_rows_body); NaN if a copy is missing
            const float sfy = ok ? (CONJ ? sfs[y] : sfs[y] * (1.0f / N)) : __int_as_float(0x7FFFFFFF);
            float2 v[E];
            if constexpr (CONJ) {
                const unsigned long long C = a.conj.chirp_fx[l];
                const unsigned long long cy = chirp_turns(C, y, N);
#pragma unroll
                for (int m = 0; m < E; ++m)
                    v[m] = unit_phasor(P[m * T], S, cy + chirp_turns(C, t + m * T, N)) * (sfy * sfs[t + m * T]);
            } else {
#pragma unroll
                for (int m = 0; m < E; ++m) v[m] = unit_phasor(P[m * T], S) * (sfy * sfs[t + m * T]);
            }
            fft_line_tr<float2, N, -1, 16, 1, 1, SUB>(v, buf, t, tr);
            // the row is past its first exchange, hence done with this wavelength's taper, and with the
            // phases at the last wavelength; the last row to get here sends for the next ones
            if (SUB == 0 ? threadIdx.x == 0 : t == 0) {
                __threadfence_block();
                if (SUB == 0 || atomicAdd(reads, 1u) % B == B - 1) {
                    const bool last = l + 1 == count, more = tile + (int)gridDim.x < tiles;
                    if (count > 1 && (!last || more)) load_sf(last ? 0 : l + 1);
                    if (bulk && last && more) load_phi(tile + gridDim.x);
                }
            }
            if constexpr (!CONJ) {
                const unsigned long long hc = a.lam.h_fx[l];
#pragma unroll
                for (int m = 0; m < E; ++m) v[m] = cmul(v[m], transfer_fast(hc, signed_index<N, E>(t, m)));
                fft_line_tr<float2, N, +1, 16, 1, 1, SUB>(v, buf, t, tr);
            }
            static_assert(T % W == 0, "whole strips between a thread's values");
            float2* dst = a.work + (size_t)l * N * N + strip_index<W>(y, t, N);
#pragma unroll
            for (int m = 0; m < E; ++m) dst[(size_t)(m * T) * N] = v[m];
        }
    }
    if (!ok) {    // nothing in flight may outlive the block: wait again, with the same limit
        for (int k = 0; k < 4; ++k) wait_tile(bar + (k >> 1), k & 1);
    }
}

// W consecutive values of a row of the map, o (+)= r; wide: o is aligned to min(4 W, 16) bytes
template <int W>
SCINT_DEV void store_row(float* o, float (&r)[W], int wide, int accumulate) {
    if (accumulate) {
#pragma unroll
        for (int k = 0; k < W; ++k) r[k] += o[k];
    }
    if (!wide) {
#pragma unroll
        for (int k = 0; k < W; ++k) o[k] = r[k];
    } else if constexpr (W == 2) {
        *reinterpret_cast<float2*>(o) = make_float2(r[0], r[1]);
    } else {
        static_assert(W % 4 == 0, "two columns or quadruples");
#pragma unroll
        for (int k = 0; k < W; k += 4) *reinterpret_cast<float4*>(o + k) = make_float4(r[k], r[k + 1], r[k + 2], r[k + 3]);
    }
}

// TAB: H_x by a copy from the group's tables.  A workspace without room for them has the block evaluate the
// half table itself, two tables in turn, one barrier between its making and its use (32 wavelengths in one group, with
// tables / so / with an evaluation per element: 1075 / 1144 / 1281 us at 2048^2, 4.91 / 5.12 / 5.36 ms at 4096^2).
template <int N, bool TAB> __host__ __device__ constexpr int stream_entries() { return TAB ? transfer_entries(N) : 2 * own_entries<N>(); }
template <int N, bool TAB> constexpr size_t pcol_stream_smem() {
    return col_stage_bytes<N>() + (size_t)(pcol_lines<N>() * FftPlan<N>::BUF + stream_entries<N, TAB>()) * sizeof(float2) + 24;
}

template <int N, bool TAB>
__global__ void __launch_bounds__(pcol_threads<N>(), (pcol_threads<N>() <= 256 ? 2 : 1))
prop_cols_stream_kernel(PropArgs a, const __grid_constant__ CUtensorMap tm, int wide) {
    using Pl = FftPlan<N, kColEPT>;
    constexpr int T = Pl::T, E = Pl::E, W = pcol_lines<N>();
    extern __shared__ float2 smem32[];
    begin_pass<N>();
    const int w = threadIdx.x / T, t = threadIdx.x % T;    // a team per column
    float2* stage = smem32;
    float2* bufs = stage + N * W;
    float2* buf = bufs + w * Pl::BUF;
    constexpr int HT = transfer_entries(N);
    float2* hs = bufs + W * Pl::BUF;
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(hs + stream_entries<N, TAB>());    // stage, H
    unsigned* reads = reinterpret_cast<unsigned*>(bar + 2);    // teams that have read the stage, H
    const int count = a.lam.count;
    auto load_h = [&](int l) {
        tile_expect(bar + 1, HT * sizeof(float2));
        bulk_load(hs, a.h + (size_t)l * HT, HT * sizeof(float2), bar + 1);
    };
    if (threadIdx.x == 0) {
        tile_init(bar);
        tile_init(bar + 1);
        reads[0] = reads[1] = 0u;
        tile_init_fence();
        issue_columns<N>(stage, &tm, 0, blockIdx.x * W, bar);
        if (TAB) load_h(0);
    }
    TwiddleRegs<float2, N, 16> tr;
    tr.load(a.tw, t);
    __syncthreads();
    unsigned parity = 0;    // bits: the stage's, H's
    bool ok = true;
#pragma unroll 1
    for (int x0 = blockIdx.x * W; x0 < N; x0 += gridDim.x * W) {
        float acc[E];
#pragma unroll
        for (int m = 0; m < E; ++m) acc[m] = 0.0f;
#pragma unroll 1
        for (int l = 0; l < count; ++l) {
            const bool new_h = count > 1 || x0 == (int)blockIdx.x * W;
            float2* h = TAB ? hs : hs + (l & 1) * own_entries<N>();
            if (!TAB && new_h) {
                for (int i = threadIdx.x; i < own_entries<N>(); i += pcol_threads<N>()) h[i] = transfer_signed(a.lam.h_fx[l], i);
            }
            ok = ok && wait_tile(bar, parity & 1);
            parity ^= 1;
            float2 v[E];
            const float2* col = stage + (w / kBoxCols) * N * kBoxCols + w % kBoxCols;
#pragma unroll
            for (int m = 0; m < E; ++m) v[m] = col[(t + m * T) * kBoxCols];
            fft_line_tr<float2, N, -1, kColEPT, 1, 1, T>(v, buf, t, tr);
            // the team is past its first exchange, hence done with the stage; the last team to get here
            // sends for the next columns
            if (t == 0) {
                __threadfence_block();
                if (atomicAdd(reads, 1u) % W == W - 1) {
                    const bool last = l + 1 == count;
                    const int nx = last ? x0 + (int)gridDim.x * W : x0;
                    if (nx < N) issue_columns<N>(stage, &tm, last ? 0 : l + 1, nx, bar);
                }
            }
            const bool more = x0 + (int)gridDim.x * W < N;
            if (TAB && new_h) {
                ok = ok && wait_tile(bar + 1, parity >> 1);
                parity ^= 2;
            } else if (!TAB && new_h) {
                __syncthreads();    // this table is whole; the other one's readers are past it
            }
#pragma unroll
            for (int m = 0; m < E; ++m) v[m] = cmul(v[m], h[half_index<N, E>(t, m)]);
            fft_line_tr<float2, N, +1, kColEPT, 1, 1, T>(v, buf, t, tr);
            if (TAB && count > 1 && t == 0) {    // the same for H
                __threadfence_block();
                if (atomicAdd(reads + 1, 1u) % W == W - 1 && (l + 1 < count || more)) load_h(l + 1 < count ? l + 1 : 0);
            }
            // 1/N of H_y, squared, on the weight (prop_cols_body); NaN if a copy is missing
            const float wl = ok ? a.lam.weight[l] * (1.0f / ((float)N * (float)N)) : __int_as_float(0x7FFFFFFF);
#pragma unroll
            for (int m = 0; m < E; ++m) acc[m] = fmaf(wl, fmaf(v[m].x, v[m].x, v[m].y * v[m].y), acc[m]);
        }
        // the columns side by side through the line buffers, one store of W values per row (a value of
        // one column per thread and row had cost 0.05 ms at 4096^2: one 4-byte sector write each)
        float* own = reinterpret_cast<float*>(buf);
#pragma unroll
        for (int m = 0; m < E; ++m) own[t + m * T] = acc[m];
        __syncthreads();
#pragma unroll 2
        for (int y = threadIdx.x; y < N; y += pcol_threads<N>()) {
            float r[W];
#pragma unroll
            for (int k = 0; k < W; ++k) r[k] = reinterpret_cast<const float*>(bufs + k * Pl::BUF)[y];
            store_row<W>(a.intensity + (size_t)y * N + x0, r, wide, a.accumulate);
        }
        __syncthreads();
    }
    if (!ok) {
        for (int k = 0; k < (TAB ? 4 : 2); ++k) wait_tile(bar + (k >> 1), k & 1);
    }
}
template <int N, bool TAB>
cudaError_t launch_cols_stream(const PropArgs& a, const CUtensorMap& tm, cudaStream_t s) {
    constexpr size_t smem = pcol_stream_smem<N, TAB>();
    static_assert(smem <= kMaxSmem, "streamed column pass does not fit");
    auto k = prop_cols_stream_kernel<N, TAB>;
    cudaError_t e = set_smem(k, smem);
    int blocks = 0;
    if (e == cudaSuccess) e = walk_blocks(k, pcol_threads<N>(), smem, N / pcol_lines<N>(), a.lam.count, &blocks);
    if (e != cudaSuccess) return e;
    constexpr int align = pcol_lines<N>() == 2 ? 8 : 16;
    return launch_pass<N>(a.lam.count, k, dim3(blocks), dim3(pcol_threads<N>()), smem, s, a, tm,
                          (int)(reinterpret_cast<uintptr_t>(a.intensity) % align == 0));
}

// ---- lines of 8192 points: two half lines per team (fft_long) ----------------------------
// Per launch against 512 threads with sixteen values each: rows 3.70 -> 3.06 ms (8 wavelengths), 0.797 ->
// 0.496 (one); columns 3.95 -> 2.9 to 3.2 and 1.08 -> 0.56.
// Row pass: 256 threads per row, two rows per SM; the phases by bulk copy as above, the taper
// from its table (no room beside two rows' phases).
// Column pass: 256 threads and one column per block, two blocks per SM, so that one column's
// loads run behind the other's transforms; the passband sums in shared memory (the values take
// the registers).  Clusters of four blocks share a strip and put their four columns' sums
// side by side through distributed shared memory: one 16-byte store per row and cluster instead
// of a 4-byte one per row and column.
template <int N> __host__ __device__ constexpr bool long_lines() { return N == 8192; }
template <int N> constexpr size_t prow_long_smem() { return (size_t)LongPlan<N>::BUF * sizeof(float2) + N * sizeof(long long) + 16; }

// a and b times H at the frequencies 2k and 2k + 1, k = t + m T (TAB: from the table)
template <int N, bool TAB>
SCINT_DEV void long_transfer(float2 (&a)[16], float2 (&b)[16], const PropArgs& p, int l, int t) {
    constexpr int T = LongPlan<N>::T;
    if constexpr (TAB) {
        const float4* h = reinterpret_cast<const float4*>(p.h + (size_t)l * N) + t;
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const float4 q = __ldg(h + m * T);
            a[m] = cmul(a[m], make_float2(q.x, q.y));
            b[m] = cmul(b[m], make_float2(q.z, q.w));
        }
    } else {
        const unsigned long long hc = p.lam.h_fx[l];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int f = 2 * signed_index<N / 2, 16>(t, m);
            a[m] = cmul(a[m], transfer_signed(hc, f));
            b[m] = cmul(b[m], transfer_signed(hc, f + 1));
        }
    }
}

template <int N, bool CONJ>
__global__ void __launch_bounds__(LongPlan<N>::T, 2) prop_rows_long_kernel(PropArgs a, int bulk) {
    using Pl = LongPlan<N>;
    constexpr int T = Pl::T, H = Pl::H, W = pstrip<N>();
    extern __shared__ float2 smem32[];
    const int t = threadIdx.x;
    float2* buf = smem32;
    long long* Pall = reinterpret_cast<long long*>(smem32 + Pl::BUF);
    long long* P = Pall + t;
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(Pall + N);
    auto load_phi = [&](int y) {
        tile_expect(bar, N * sizeof(double));
        bulk_load(Pall, a.phi + (size_t)y * N, N * sizeof(double), bar);
    };
    if (t == 0) {
        tile_init(bar);
        tile_init_fence();
        if (bulk) load_phi(blockIdx.x);
    }
    TwiddleRegs<float2, N / 2, 16, 4> tr;
    tr.load(a.tw, t, 2);
    const float2 w0 = __ldg(a.tw + t);
    __syncthreads();
    unsigned parity = 0;
    bool ok = true;
#pragma unroll 1
    for (int y = blockIdx.x; y < N; y += gridDim.x) {
        if (bulk) {
            ok = ok && wait_tile(bar, parity);
            parity ^= 1;
            phases_fixed<2 * H>([&](int m) { return __longlong_as_double(P[m * T]); }, [&](int m, long long p) { P[m * T] = p; });
            tile_reuse_fence();
        } else {
            phases_fixed<2 * H>([&](int m) { return a.phi[(size_t)y * N + t + m * T]; }, [&](int m, long long p) { P[m * T] = p; });
        }
#pragma unroll 1
        for (int l = 0; l < a.lam.count; ++l) {
            const unsigned long long S = a.lam.scale_fx[l];
            const float* sf = a.sf + (size_t)l * N;
            // 1/N of the inverse transform on the taper of the row; NaN if a copy is missing
            const float sfy = ok ? (CONJ ? sf[y] : sf[y] * (1.0f / N)) : __int_as_float(0x7FFFFFFF);
            float2 va[H], vb[H];
            if constexpr (CONJ) {
                const unsigned long long C = a.conj.chirp_fx[l];
                const unsigned long long cy = chirp_turns(C, y, N);
#pragma unroll
                for (int m = 0; m < H; ++m) {
                    const int x = t + m * T, z = x + N / 2;
                    va[m] = unit_phasor(P[m * T], S, cy + chirp_turns(C, x, N)) * (sfy * __ldg(sf + x));
                    vb[m] = unit_phasor(P[m * T + N / 2], S, cy + chirp_turns(C, z, N)) * (sfy * __ldg(sf + z));
                }
            } else {
#pragma unroll
                for (int m = 0; m < H; ++m) {
                    const int x = t + m * T, z = x + N / 2;
                    va[m] = unit_phasor(P[m * T], S) * (sfy * __ldg(sf + x));
                    vb[m] = unit_phasor(P[m * T + N / 2], S) * (sfy * __ldg(sf + z));
                }
            }
            // the one-FFT method has no accurate H to make up for the products' rounding: its factors come from the table
            // (rms error of 3 wavelengths at 8192^2: 3.41e-7 with products, 3.30e-7 before there were half lines)
            fft_long<N, -1, CONJ>(va, vb, buf, t, tr, w0, a.tw);
            // every thread is past an exchange, hence done with the phases at the last wavelength
            if (bulk && t == 0 && l + 1 == a.lam.count && y + (int)gridDim.x < N) load_phi(y + gridDim.x);
            float2* dst = a.work + (size_t)l * N * N + strip_index<W>(y, CONJ ? 2 * t : t, N);
            if constexpr (CONJ) {
                // the frequencies 2k and 2k + 1 are neighbours in the strip
#pragma unroll
                for (int m = 0; m < H; ++m)
                    *reinterpret_cast<float4*>(dst + (size_t)(2 * m * T) * N) =
                        make_float4(va[m].x, va[m].y, vb[m].x, vb[m].y);
            } else {
                const unsigned long long hc = a.lam.h_fx[l];
#pragma unroll
                for (int m = 0; m < H; ++m) {
                    const int f = 2 * signed_index<N / 2, H>(t, m);
                    va[m] = cmul(va[m], transfer_fast(hc, f));
                    vb[m] = cmul(vb[m], transfer_fast(hc, f + 1));
                }
                fft_long<N, +1>(va, vb, buf, t, tr, w0);
#pragma unroll
                for (int m = 0; m < H; ++m) {
                    dst[(size_t)(m * T) * N] = va[m];
                    dst[(size_t)(m * T + N / 2) * N] = vb[m];
                }
            }
        }
    }
    if (!ok) {
        wait_tile(bar, 0);
        wait_tile(bar, 1);
    }
}

constexpr int kLongCluster = 4;
template <int N> constexpr size_t pcol_long_smem() { return (size_t)LongPlan<N>::BUF * sizeof(float2) + N * sizeof(float); }

template <int N, bool TAB>
__global__ void __launch_bounds__(LongPlan<N>::T, 2) prop_cols_long_kernel(PropArgs a, int wide) {
    using Pl = LongPlan<N>;
    constexpr int T = Pl::T, H = Pl::H, WL = pstrip<N>(), C = kLongCluster;
    static_assert(WL == C, "a cluster per strip");
    extern __shared__ float2 smem32[];
    auto cl = cooperative_groups::this_cluster();
    const int t = threadIdx.x, r = (int)cl.block_rank();
    float2* buf = smem32;
    float* acc = reinterpret_cast<float*>(smem32 + Pl::BUF);    // own entries until the end
    TwiddleRegs<float2, N / 2, 16, 4> tr;
    tr.load(a.tw, t, 2);
    const float2 w0 = __ldg(a.tw + t);
    const int x0 = (int)blockIdx.x / C * C;
    const float2* col = a.work + (size_t)x0 * N + r;
#pragma unroll 1
    for (int l = 0; l < a.lam.count; ++l) {
        const float2* src = col + (size_t)l * N * N;
        float2 va[H], vb[H];
#pragma unroll
        for (int m = 0; m < H; ++m) {
            va[m] = __ldcg(src + (size_t)(t + m * T) * WL);
            vb[m] = __ldcg(src + (size_t)(t + m * T + N / 2) * WL);
        }
        fft_long<N, -1>(va, vb, buf, t, tr, w0);
        long_transfer<N, TAB>(va, vb, a, l, t);
        fft_long<N, +1>(va, vb, buf, t, tr, w0);
        // 1/N of H_y, squared, on the weight (prop_cols_body)
        const float wl = a.lam.weight[l] * (1.0f / ((float)N * (float)N));
#pragma unroll
        for (int m = 0; m < H; ++m) {
            float* p = acc + t + m * T;
            float* q = p + N / 2;
            const float pa = l ? *p : 0.0f, qa = l ? *q : 0.0f;
            *p = fmaf(wl, fmaf(va[m].x, va[m].x, va[m].y * va[m].y), pa);
            *q = fmaf(wl, fmaf(vb[m].x, vb[m].x, vb[m].y * vb[m].y), qa);
        }
    }
    cl.sync();
    // rank r stores its quarter of the rows, the cluster's four columns side by side
    const float* part[C];
#pragma unroll
    for (int k = 0; k < C; ++k) part[k] = cl.map_shared_rank(acc, k);
#pragma unroll 4
    for (int y = r * (N / C) + t; y < (r + 1) * (N / C); y += T) {
        float s[C];
#pragma unroll
        for (int k = 0; k < C; ++k) s[k] = part[k][y];
        store_row<C>(a.intensity + (size_t)y * N + x0, s, wide, a.accumulate);
    }
    cl.sync();    // no block leaves before its sums are read
}

bool field_map(CUtensorMap* tm, const float2* work, int n, int count, int strip) {
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<Encode>(f);
    }();
    if (!encode || reinterpret_cast<uintptr_t>(work) % 16) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)(2 * strip), (cuuint64_t)count * (n / strip) * n};
    const cuuint64_t strides[1] = {(cuuint64_t)strip * sizeof(float2)};
    const cuuint32_t box[2] = {2 * kBoxCols, kBoxRows}, step[2] = {1, 1};
    return encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float2*>(work), dims, strides, box, step,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---- lines split over a two-block cluster (N = 16384) -------------------------------
// One radix-2 step on each side of the line transforms divides them between the two
// blocks of a cluster (n < N/2, W = exp(-2 pi i / N)):
//   forward, decimation in frequency: a_n = x_n + x_{n+N/2}, b_n = (x_n - x_{n+N/2}) W^n,
//     X_{2k} = FFT_{N/2}(a)_k, X_{2k+1} = FFT_{N/2}(b)_k;
//   inverse, decimation in time: A' = IFFT_{N/2}(Y_{2k}), B' = IFFT_{N/2}(Y_{2k+1}),
//     y_n = A'_n + W^{-n} B'_n, y_{n+N/2} = A'_n - W^{-n} B'_n.
// Block r takes the parity-r half-problem, an 8192-point line of two half lines (fft_long: 256
// threads, two blocks per SM), and H at the frequencies 2k + r.  It reads and writes the
// line at its quarters n in [r N/4, (r + 1) N/4) and n + N/2 only: each input is read, and each
// phasor formed, by one block, which keeps its parity's a_n or b_n and hands the other to its
// partner through shared memory; the same exchange before the last step brings what the block's
// outputs need.  Per wavelength the halves meet twice, each time a full cluster barrier after the
// values are published and a split one after they are read.
// Block 1's quarter is the upper half of its half-problem, so it runs fft_long with the halves
// swapped: W_{N/2}^n changes sign, and array a is always the part the block keeps.
// Measured per 16384^2 pass at one wavelength, against 512 threads with sixteen values each, one
// block per SM, whole lines read by both blocks: rows 4.24 -> 3.07 ms, columns 3.09 -> 2.75 ms (with the transpose).
template <int N> __host__ __device__ constexpr int psplit_threads() { return FftPlan<N / 2>::T; }
template <int N> constexpr size_t conj_row_split_smem() {
    return (size_t)FftPlan<N / 2>::BUF * sizeof(float2) + (size_t)N * sizeof(long long);
}
template <int N> constexpr size_t conj_col_split_smem() {
    return (size_t)(FftPlan<N / 2>::BUF + FftPlan<N / 2>::TWS) * sizeof(float2);
}
template <int N> __host__ __device__ constexpr int lsplit_threads() { return LongPlan<N / 2>::T; }
template <int N> constexpr size_t prow_split_smem() {
    return (size_t)LongPlan<N / 2>::BUF * sizeof(float2) + (size_t)(N / 2) * sizeof(long long) + 16;
}
template <int N> constexpr size_t pcol_split_smem() {
    return (size_t)LongPlan<N / 2>::BUF * sizeof(float2) + (size_t)(N / 2) * sizeof(float);
}

// W_N^(n0 + m N/64) from W_N^n0, m < 16
template <int M> SCINT_DEV float2 quarter_twiddle(float2 w0) {
    if constexpr (M == 0) return w0;
    else return cmul(w0, make_float2((float)cos64q(M), (float)-cos64q(16 - M)));
}
// The forward exchange: (x0, x1) = x at n = r N/4 + t + m T and n + N/2 (m < 16) become this block's
// parity: a the part at its own quarter, b the partner's.  Begins by waiting for the partner's last
// read of buf, ends with a split arrive: wait before buf is written again.
template <int N, int M = 0>
SCINT_DEV void quarter_split(float2* x0, float2* x1, float2* out, int r, float2 wq) {
    if constexpr (M < 16) {
        const float2 sum = x0[M] + x1[M], dif = cmul(x0[M] - x1[M], quarter_twiddle<M>(wq));
        x0[M] = r == 0 ? sum : dif;
        out[pad16(M * LongPlan<N / 2>::T)] = r == 0 ? dif : sum;    // T is a multiple of 16
        quarter_split<N, M + 1>(x0, x1, out, r, wq);
    }
}
template <int N>
SCINT_DEV void exchange_forward(float2 (&a)[16], float2 (&b)[16], float2* buf, int t, int r, float2 wq) {
    constexpr int T = LongPlan<N / 2>::T;
    cluster_wait();
    quarter_split<N>(a, b, buf + pad16(t), r, wq);
    line_sync<2>();
    const unsigned pb = cluster_addr(buf, (unsigned)(r ^ 1)) + (unsigned)(pad16(t) * sizeof(float2));
#pragma unroll
    for (int m = 0; m < 16; ++m) b[m] = ld_cluster<float2>(pb + (unsigned)(m * (T + T / 16) * sizeof(float2)));
    cluster_arrive();
}
// The inverse exchange: a = this block's parity at its own quarter, b at the partner's; on exit
// a = y_n and b = y_{n+N/2} at its own quarter.  Same barriers.
template <int N, int M = 0>
SCINT_DEV void quarter_join(float2* a, float2* q, int r, float2 wq) {
    if constexpr (M < 16) {
        const float2 A = r == 0 ? a[M] : q[M], B = r == 0 ? q[M] : a[M];
        const float2 y = cfma(B, conjc(quarter_twiddle<M>(wq)), A);
        q[M] = twice_minus(A, y);
        a[M] = y;
        quarter_join<N, M + 1>(a, q, r, wq);
    }
}
template <int N>
SCINT_DEV void exchange_inverse(float2 (&a)[16], float2 (&b)[16], float2* buf, int t, int r, float2 wq) {
    constexpr int T = LongPlan<N / 2>::T;
    float2* out = buf + pad16(t);
#pragma unroll
    for (int m = 0; m < 16; ++m) out[m * (T + T / 16)] = b[m];
    line_sync<2>();
    const unsigned pb = cluster_addr(buf, (unsigned)(r ^ 1)) + (unsigned)(pad16(t) * sizeof(float2));
#pragma unroll
    for (int m = 0; m < 16; ++m) b[m] = ld_cluster<float2>(pb + (unsigned)(m * (T + T / 16) * sizeof(float2)));
    cluster_arrive();
    quarter_join<N>(a, b, r, wq);
}
// a and b times H at the frequencies 2k + r of fft_long's k (a: k = 2 (t + m T), b: the next)
// (TAB: from the table)
template <int N, bool TAB>
SCINT_DEV void split_transfer(float2 (&a)[16], float2 (&b)[16], const PropArgs& p, int l, int t, int r) {
    constexpr int T = LongPlan<N / 2>::T;
    if constexpr (TAB) {
        const float4* h = reinterpret_cast<const float4*>(p.h + (size_t)l * N + r * (N / 2)) + t;
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const float4 q = __ldg(h + m * T);
            a[m] = cmul(a[m], make_float2(q.x, q.y));
            b[m] = cmul(b[m], make_float2(q.z, q.w));
        }
    } else {
        const unsigned long long hc = p.lam.h_fx[l];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int f = 4 * signed_index<N / 4, 16>(t, m) + r;
            a[m] = cmul(a[m], transfer_signed(hc, f));
            b[m] = cmul(b[m], transfer_signed(hc, f + 2));
        }
    }
}

template <int N, bool TAB>
__global__ void __launch_bounds__(lsplit_threads<N>(), 2) prop_rows_split_kernel(PropArgs a, int bulk) {
    constexpr int H2 = N / 2, M = N / 4;
    using Pl = LongPlan<H2>;
    constexpr int T = Pl::T, W = pstrip<N>();
    extern __shared__ float2 smem32[];
    const int r = (int)cooperative_groups::this_cluster().block_rank();
    const int t = threadIdx.x, n0 = r * M + t;
    float2* buf = smem32;
    long long* Pall = reinterpret_cast<long long*>(smem32 + Pl::BUF);    // this block's quarters
    long long* P = Pall + t;
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(Pall + H2);
    auto load_phi = [&](int y) {
        const double* phi = a.phi + (size_t)y * N + r * M;
        tile_expect(bar, H2 * sizeof(double));
        bulk_load(Pall, phi, M * sizeof(double), bar);
        bulk_load(Pall + M, phi + H2, M * sizeof(double), bar);
    };
    if (t == 0) {
        tile_init(bar);
        tile_init_fence();
        if (bulk) load_phi(blockIdx.x / 2);
    }
    TwiddleRegs<float2, M, 16, 4> tr;
    tr.load(a.tw, t, 4);    // the N-point table at every fourth index
    const float2 wq = __ldg(a.tw + n0), w1 = __ldg(a.tw + 2 * t), w0 = r ? make_float2(-w1.x, -w1.y) : w1;
    __syncthreads();
    cluster_arrive();
    unsigned parity = 0;
    bool ok = true;
    // persistent: the cluster takes rows y, y + clusters, ...
#pragma unroll 1
    for (int y = blockIdx.x / 2; y < N; y += gridDim.x / 2) {
        if (bulk) {
            ok = ok && wait_tile(bar, parity);
            parity ^= 1;
            phases_fixed<32>([&](int m) { return __longlong_as_double(P[m * T]); }, [&](int m, long long p) { P[m * T] = p; });
            tile_reuse_fence();
        } else {
            const double* phi = a.phi + (size_t)y * N + n0;
            phases_fixed<32>([&](int m) { return phi[m * T + (m < 16 ? 0 : H2 - M)]; },
                             [&](int m, long long p) { P[m * T] = p; });
        }
#pragma unroll 1
        for (int l = 0; l < a.lam.count; ++l) {
            const unsigned long long S = a.lam.scale_fx[l];
            const float* sf = a.sf + (size_t)l * N;
            // 1/N of the inverse transform on the taper of the row; NaN if a copy is missing
            const float sfy = ok ? sf[y] * (1.0f / N) : __int_as_float(0x7FFFFFFF);
            float2 va[16], vb[16];
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                va[m] = unit_phasor(P[m * T], S) * (sfy * __ldg(sf + n0 + m * T));
                vb[m] = unit_phasor(P[m * T + M], S) * (sfy * __ldg(sf + n0 + m * T + H2));
            }
            exchange_forward<N>(va, vb, buf, t, r, wq);
            // every thread is past a barrier, hence done with the phases at the last wavelength
            if (bulk && t == 0 && l + 1 == a.lam.count && y + (int)gridDim.x / 2 < N) load_phi(y + gridDim.x / 2);
            cluster_wait();
            fft_long<H2, -1>(va, vb, buf, t, tr, w0);
            split_transfer<N, TAB>(va, vb, a, l, t, r);
            fft_long<H2, +1>(va, vb, buf, t, tr, w0);
            exchange_inverse<N>(va, vb, buf, t, r, wq);
            float2* dst = a.work + (size_t)l * N * N + strip_index<W>(y, n0, N);
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                dst[(size_t)(m * T) * N] = va[m];
                dst[(size_t)(m * T + H2) * N] = vb[m];
            }
        }
    }
    cluster_wait();    // no block leaves before its buffer is read
    if (!ok) {
        wait_tile(bar, 0);
        wait_tile(bar, 1);
    }
}

template <int N, bool TAB>
__global__ void __launch_bounds__(lsplit_threads<N>(), 2) prop_cols_split_kernel(PropArgs a) {
    constexpr int H2 = N / 2, M = N / 4;
    using Pl = LongPlan<H2>;
    constexpr int T = Pl::T, WL = pstrip<N>();
    extern __shared__ float2 smem32[];
    const int r = (int)cooperative_groups::this_cluster().block_rank();
    const int t = threadIdx.x, n0 = r * M + t;
    float2* buf = smem32;
    float* acc = reinterpret_cast<float*>(smem32 + Pl::BUF) + t;    // own entries
    TwiddleRegs<float2, M, 16, 4> tr;
    tr.load(a.tw, t, 4);
    const float2 wq = __ldg(a.tw + n0), w1 = __ldg(a.tw + 2 * t), w0 = r ? make_float2(-w1.x, -w1.y) : w1;
    cluster_arrive();
    // persistent: the cluster takes columns x, x + clusters, ...
#pragma unroll 1
    for (int x = blockIdx.x / 2; x < N; x += gridDim.x / 2) {
#pragma unroll 1
        for (int l = 0; l < a.lam.count; ++l) {
            const float2* src = a.work + (size_t)l * N * N + (size_t)(x / WL) * N * WL + (x % WL) + (size_t)n0 * WL;
            float2 va[16], vb[16];
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                va[m] = __ldcg(src + (size_t)(m * T) * WL);
                vb[m] = __ldcg(src + (size_t)(m * T + H2) * WL);
            }
            exchange_forward<N>(va, vb, buf, t, r, wq);
            cluster_wait();
            fft_long<H2, -1>(va, vb, buf, t, tr, w0);
            split_transfer<N, TAB>(va, vb, a, l, t, r);
            fft_long<H2, +1>(va, vb, buf, t, tr, w0);
            exchange_inverse<N>(va, vb, buf, t, r, wq);
            // 1/N of H_y, squared, on the weight (prop_cols_body); the last sum goes out column-major, so that
            // the stores coalesce (transpose_add_kernel puts it in place)
            const float wl = a.lam.weight[l] * (1.0f / ((float)N * (float)N));
            const bool last = l + 1 == a.lam.count;
            float* col = last ? a.scratch + (size_t)x * N + n0 : acc;
            const int half = last ? H2 : M;
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                const float p = l ? acc[m * T] : 0.0f, q = l ? acc[m * T + M] : 0.0f;
                col[m * T] = fmaf(wl, fmaf(va[m].x, va[m].x, va[m].y * va[m].y), p);
                col[m * T + half] = fmaf(wl, fmaf(vb[m].x, vb[m].x, vb[m].y * vb[m].y), q);
            }
        }
    }
    cluster_wait();
}

// One-FFT mode (Eq. intens, Eq. Gxy) at N = 16384: forward transforms only, so the
// decimation-in-frequency split alone divides them (block r makes the frequencies
// 2k + r).  The row pass copies the partner's half of the row's phases once per row
// (split arrive/wait around the next row's fill) and writes X(2k + r); the column pass
// needs nothing from its partner: both blocks read the whole column (the second read
// from L2) and each writes its parity's pattern rows, column-major.
template <int N>
__global__ void __launch_bounds__(psplit_threads<N>(), 1) conj_rows_split_kernel(PropArgs a) {
    constexpr int H2 = N / 2;
    using Pl = FftPlan<H2>;
    constexpr int T = Pl::T, E = Pl::E, W = pstrip<N>();
    extern __shared__ float2 smem32[];
    const int r = (int)cooperative_groups::this_cluster().block_rank();
    const int t = threadIdx.x;
    float2* buf = smem32;
    long long* P = reinterpret_cast<long long*>(smem32 + Pl::BUF);
    TwiddleRegs<float2, H2, 16> tr;
    tr.load(a.tw, t, 2);
    bool first = true;
#pragma unroll 1
    for (int y = blockIdx.x / 2; y < N; y += gridDim.x / 2) {
        if (!first) cluster_wait();     // the partner has copied this block's previous phases
        first = false;
        const double* phi = a.phi + (size_t)y * N + r * H2;
        phases_fixed<E>([&](int m) { return phi[t + m * T]; }, [&](int m, long long p) { P[r * H2 + t + m * T] = p; });
        line_sync<2>();
        const unsigned pp = cluster_addr(P, (unsigned)(r ^ 1)) + (unsigned)(((r ^ 1) * H2 + t) * sizeof(long long));
#pragma unroll
        for (int m = 0; m < E; ++m)
            P[(r ^ 1) * H2 + t + m * T] = ld_cluster<long long>(pp + (unsigned)(m * T * sizeof(long long)));
        cluster_arrive();
#pragma unroll 1
        for (int l = 0; l < a.lam.count; ++l) {
            const unsigned long long S = a.lam.scale_fx[l], C = a.conj.chirp_fx[l];
            const float* sf = a.sf + (size_t)l * N;
            const float sfy = sf[y];
            const unsigned long long cy = chirp_turns(C, y, N);
            float2 v[E];
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const int e = t + m * T;
                // G = SF SF exp(i (phi s + |x_1|^2 / 2 R_F^2)) (-1)^(x + y), Eq. Gxy
                const float2 x0 = unit_phasor(P[e], S, cy + chirp_turns(C, e, N)) * (sfy * __ldg(sf + e));
                const float2 x1 = unit_phasor(P[e + H2], S, cy + chirp_turns(C, e + H2, N)) * (sfy * __ldg(sf + e + H2));
                v[m] = split_dif(x0, x1, r, e, a.tw);
            }
            fft_line_tr<float2, H2, -1, 16, 1>(v, buf, t, tr);
            float2* dst = a.work + (size_t)l * N * N;
#pragma unroll
            for (int m = 0; m < E; ++m) dst[strip_index<W>(y, 2 * (t + m * T) + r, N)] = v[m];
        }
    }
    if (!first) cluster_wait();
}

template <int N>
__global__ void __launch_bounds__(psplit_threads<N>(), 1) conj_cols_split_kernel(PropArgs a) {
    constexpr int H2 = N / 2;
    using Pl = FftPlan<H2>;
    constexpr int T = Pl::T, E = Pl::E, WL = pstrip<N>();
    extern __shared__ float2 smem32[];
    const int r = (int)cooperative_groups::this_cluster().block_rank();
    const int t = threadIdx.x;
    float2* buf = smem32;
    float2* tws = smem32 + Pl::BUF;
    fill_twiddle_table<float2, H2>(tws, a.tw, t, T, 2);
    __syncthreads();
#pragma unroll 1
    for (int x = blockIdx.x / 2; x < N; x += gridDim.x / 2) {
        float acc[E];
#pragma unroll
        for (int m = 0; m < E; ++m) acc[m] = 0.0f;
#pragma unroll 1
        for (int l = 0; l < a.lam.count; ++l) {
            const float2* src = a.work + (size_t)l * N * N + (size_t)(x / WL) * N * WL + (x % WL);
            float2 v[E];
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const int e = t + m * T;
                v[m] = split_dif(src[(size_t)e * WL], src[(size_t)(e + H2) * WL], r, e, a.tw);
            }
            fft_line<float2, H2, -1, 16, 1, 1, 1>(v, buf, t, tws);
            // h = (Delta^2 / lambda z)^2 |FT G|^2 on the pattern grid of this wavelength (Eq. intens)
            const float nrm = a.conj.norm[l];
            if (a.conj.direct) {
                const float wn = a.lam.weight[l] * nrm;
#pragma unroll
                for (int m = 0; m < E; ++m) acc[m] = fmaf(wn, fmaf(v[m].x, v[m].x, v[m].y * v[m].y), acc[m]);
            } else {
                float* pat = a.conj.pattern + (size_t)l * N * N + (size_t)x * N;
#pragma unroll
                for (int m = 0; m < E; ++m) pat[2 * (t + m * T) + r] = nrm * fmaf(v[m].x, v[m].x, v[m].y * v[m].y);
            }
        }
        if (a.conj.direct) {
            // column-major, transposed into place by transpose_add_kernel
            float* col = a.scratch + (size_t)x * N;
#pragma unroll
            for (int m = 0; m < E; ++m) col[2 * (t + m * T) + r] = acc[m];
        }
    }
}

// intensity (+)= the transpose of the column-major map src, in 32 x 32 tiles through
// shared memory (reads and writes both coalesced); n is a multiple of 32
__global__ void __launch_bounds__(256) transpose_add_kernel(const float* __restrict__ src, float* dst, int n,
                                                            int accumulate) {
    __shared__ float tile[32][33];
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
#pragma unroll
    for (int k = ty; k < 32; k += 8) tile[k][tx] = src[(size_t)(x0 + k) * n + y0 + tx];   // [x][y]
    __syncthreads();
#pragma unroll
    for (int k = ty; k < 32; k += 8) {
        float* o = dst + (size_t)(y0 + k) * n + x0 + tx;
        const float v = tile[tx][k];
        *o = accumulate ? *o + v : v;
    }
}

template <bool CONJ>
cudaError_t launch_rows(const PropArgs& a, cudaStream_t s) {
    return dispatch_n(a.n, [&](auto nc) -> cudaError_t {
        constexpr int N = decltype(nc)::value;
        if constexpr (pcs<N>() == 2 && CONJ) {
            static_assert(conj_row_split_smem<N>() <= kMaxSmem, "split row pass does not fit");
            auto k = conj_rows_split_kernel<N>;
            cudaError_t e = set_smem(k, conj_row_split_smem<N>());
            int nc = 0;
            if (e == cudaSuccess) e = active_clusters(k, 2, psplit_threads<N>(), conj_row_split_smem<N>(), &nc);
            if (e != cudaSuccess) return e;
            return launch_k(k, 2, dim3(2 * std::min(nc, N)), dim3(psplit_threads<N>()), conj_row_split_smem<N>(), s, a);
        } else if constexpr (pcs<N>() == 2) {
            static_assert(2 * (prow_split_smem<N>() + 1024) <= 228 * 1024, "two blocks per SM");
            auto k = a.h ? prop_rows_split_kernel<N, true> : prop_rows_split_kernel<N, false>;
            cudaError_t e = set_smem(k, prow_split_smem<N>());
            int nc = 0;
            if (e == cudaSuccess) e = active_clusters(k, 2, lsplit_threads<N>(), prow_split_smem<N>(), &nc);
            if (e != cudaSuccess) return e;
            return launch_k(k, 2, dim3(2 * std::min(nc, N)), dim3(lsplit_threads<N>()), prow_split_smem<N>(), s, a,
                            (int)(reinterpret_cast<uintptr_t>(a.phi) % 16 == 0));
        } else if constexpr (prow_smem<N>() > kMaxSmem || pcol_smem<N, true>() > kMaxSmem) {
            return cudaErrorNotSupported;
        } else {
            if constexpr (long_lines<N>()) {
                static_assert(2 * (prow_long_smem<N>() + 1024) <= 228 * 1024, "two rows per SM");
                auto k = prop_rows_long_kernel<N, CONJ>;
                cudaError_t e = set_smem(k, prow_long_smem<N>());
                int blocks = 0;
                if (e == cudaSuccess) e = walk_blocks(k, LongPlan<N>::T, prow_long_smem<N>(), N, a.lam.count, &blocks);
                if (e != cudaSuccess) return e;
                k<<<blocks, LongPlan<N>::T, prow_long_smem<N>(), s>>>(a, reinterpret_cast<uintptr_t>(a.phi) % 16 == 0);
                return cudaGetLastError();
            } else if constexpr (row_stream<N>()) {
                static_assert(prow_stream_smem<N>() <= kMaxSmem, "streamed row pass does not fit");
                auto k = prop_rows_stream_kernel<N, CONJ>;
                cudaError_t e = set_smem(k, prow_stream_smem<N>());
                int blocks = 0;
                if (e == cudaSuccess)
                    e = walk_blocks(k, prow_threads<N>(), prow_stream_smem<N>(), N / prow_lines<N>(), a.lam.count, &blocks);
                if (e != cudaSuccess) return e;
                // a bulk copy starts on a 16-byte boundary: phases elsewhere are read by plain loads
                return launch_pass<N>(a.lam.count, k, dim3(blocks), dim3(prow_threads<N>()), prow_stream_smem<N>(), s, a,
                                      (int)(reinterpret_cast<uintptr_t>(a.phi) % 16 == 0));
            } else {
                cudaError_t e = set_smem(prop_rows_kernel<N, CONJ>, prow_smem<N>());
                if (e != cudaSuccess) return e;
                return launch_pass<N>(a.lam.count, prop_rows_kernel<N, CONJ>, dim3(N / prow_lines<N>()),
                                      dim3(prow_threads<N>()), prow_smem<N>(), s, a);
            }
        }
    });
}

template <bool CONJ>
cudaError_t launch_cols(const PropArgs& a, cudaStream_t s) {
    return dispatch_n(a.n, [&](auto nc) -> cudaError_t {
        constexpr int N = decltype(nc)::value;
        if constexpr (pcs<N>() == 2) {
            const bool to_scratch = !CONJ || a.conj.direct;    // intensity through the transpose
            if (to_scratch && !a.scratch) return cudaErrorInvalidValue;
            constexpr size_t smem = CONJ ? conj_col_split_smem<N>() : pcol_split_smem<N>();
            constexpr int threads = CONJ ? psplit_threads<N>() : lsplit_threads<N>();
            static_assert(smem <= kMaxSmem, "split column pass does not fit");
            auto k = CONJ ? conj_cols_split_kernel<N> : (a.h ? prop_cols_split_kernel<N, true> : prop_cols_split_kernel<N, false>);
            cudaError_t e = set_smem(k, smem);
            int nc = 0;
            if (e == cudaSuccess) e = active_clusters(k, 2, threads, smem, &nc);
            if (e != cudaSuccess) return e;
            e = launch_k(k, 2, dim3(2 * std::min(nc, N)), dim3(threads), smem, s, a);
            if (e != cudaSuccess || !to_scratch) return e;
            transpose_add_kernel<<<dim3(N / 32, N / 32), 256, 0, s>>>(a.scratch, a.intensity, N, a.accumulate);
            return cudaGetLastError();
        } else if constexpr (prow_smem<N>() > kMaxSmem || pcol_smem<N, true>() > kMaxSmem) {
            return cudaErrorNotSupported;
        } else {
            if constexpr (!CONJ && long_lines<N>()) {
                static_assert(2 * (pcol_long_smem<N>() + 1024) <= 228 * 1024, "two columns per SM");
                auto k = a.h ? prop_cols_long_kernel<N, true> : prop_cols_long_kernel<N, false>;
                const cudaError_t e = set_smem(k, pcol_long_smem<N>());
                if (e != cudaSuccess) return e;
                return launch_k(k, kLongCluster, dim3(N), dim3(LongPlan<N>::T), pcol_long_smem<N>(), s, a,
                                (int)(reinterpret_cast<uintptr_t>(a.intensity) % 16 == 0));
            } else {
                if constexpr (!CONJ && col_stream<N>()) {
                    CUtensorMap tm;
                    if (field_map(&tm, a.work, N, a.lam.count, pstrip<N>()))
                        return a.h ? launch_cols_stream<N, true>(a, tm, s) : launch_cols_stream<N, false>(a, tm, s);
                }
                constexpr size_t smem = pcol_smem<N, CONJ>();
                cudaError_t e = set_smem(prop_cols_kernel<N, CONJ>, smem);
                if (e != cudaSuccess) return e;
                return launch_pass<N>(a.lam.count, prop_cols_kernel<N, CONJ>, dim3(N / pcol_lines<N>()), dim3(pcol_threads<N>()), smem,
                                      s, a);
            }
        }
    });
}

cudaError_t launch_prop_rows(const PropArgs& a, bool conj, cudaStream_t s) {
    return conj ? launch_rows<true>(a, s) : launch_rows<false>(a, s);
}
cudaError_t launch_prop_cols(const PropArgs& a, bool conj, cudaStream_t s) {
    return conj ? launch_cols<true>(a, s) : launch_cols<false>(a, s);
}

// ---- passband of one-FFT patterns --------------------------------------------------
// Output pixel (X, Y) samples pattern l at (X - n/2) r_l + n/2 and (Y - n/2) r_l + n/2
// pattern pixels; the products are exact in 32.32 fixed point (|X - n/2| r_l < 2^47).
// Patterns are column-major (element (x, y) at x n + y).
struct Sample {
    int i0;       // integer part, not yet wrapped
    float f;      // fraction
};
SCINT_DEV Sample sample_at(int X, int n, long long r_fx) {
    const long long u = (long long)(X - n / 2) * r_fx + ((long long)(n / 2) << 32);
    return Sample{(int)(u >> 32), (float)(unsigned)(u & 0xFFFFFFFFll) * 0x1.0p-32f};
}

// Tiled form: a block makes a 32 x 32 output tile and keeps it in registers over
// all wavelengths.  Lanes take consecutive output rows of one column, so the
// four bilinear taps of a warp read consecutive elements of two pattern columns
// (patterns are column-major); the tile goes out through shared memory as rows.
// The taps' places of the tile's 32 columns and 32 rows are worked out once per kResLambda wavelengths,
// by one thread each, and read from shared memory (in place, per pixel and wavelength, their
// 64-bit products were half of the 49 instructions: 4096^2, 8 wavelengths 0.292 -> 0.193 ms).
constexpr int kResTile = 32, kResLambda = 16;
struct Tap {
    int i0;      // wrapped
    float f;
};
SCINT_DEV Tap tap_at(int X, int n, long long r_fx) {
    const Sample s = sample_at(X, n, r_fx);
    return Tap{s.i0 & (n - 1), s.f};
}
__global__ void __launch_bounds__(256) resample_tiled_kernel(const __grid_constant__ ResampleArgs a) {
    __shared__ float tile[kResTile][kResTile + 1];   // [x][y]
    __shared__ Tap tx[kResLambda][kResTile], ty[kResLambda][kResTile];
    const int n = a.n;
    const int X0 = blockIdx.x * kResTile, Y0 = blockIdx.y * kResTile;
    const int ly = threadIdx.x % kResTile, lx = threadIdx.x / kResTile;   // lx in [0, 8)
    float acc[kResTile / 8] = {};
    for (int l0 = 0; l0 < a.count; l0 += kResLambda) {
        const int g = min(kResLambda, a.count - l0);
        __syncthreads();
        for (int i = threadIdx.x; i < 2 * kResTile * g; i += 256) {
            const int l = i / (2 * kResTile), k = i % kResTile;
            const long long r = a.r_fx[l0 + l];
            if (i % (2 * kResTile) < kResTile) tx[l][k] = tap_at(X0 + k, n, r);
            else ty[l][k] = tap_at(Y0 + k, n, r);
        }
        __syncthreads();
#pragma unroll 1
        for (int l = 0; l < g; ++l) {
            const float* h = a.pattern + (size_t)(l0 + l) * n * n;
            const Tap sy = ty[l][ly];
            const int y0 = sy.i0, y1 = (y0 + 1) & (n - 1);
            const float wl = a.weight[l0 + l];
            float h00[kResTile / 8], h01[kResTile / 8], h10[kResTile / 8], h11[kResTile / 8], fx[kResTile / 8];
#pragma unroll
            for (int q = 0; q < kResTile / 8; ++q) {
                const Tap sx = tx[l][lx + 8 * q];
                const float* c0 = h + (size_t)sx.i0 * n;
                const float* c1 = h + (size_t)((sx.i0 + 1) & (n - 1)) * n;
                fx[q] = sx.f;
                h00[q] = __ldg(c0 + y0);
                h01[q] = __ldg(c0 + y1);
                h10[q] = __ldg(c1 + y0);
                h11[q] = __ldg(c1 + y1);
            }
#pragma unroll
            for (int q = 0; q < kResTile / 8; ++q) {
                const float left = fmaf(sy.f, h01[q] - h00[q], h00[q]), right = fmaf(sy.f, h11[q] - h10[q], h10[q]);
                acc[q] = fmaf(wl, fmaf(fx[q], right - left, left), acc[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < kResTile / 8; ++q) tile[lx + 8 * q][ly] = acc[q];
    __syncthreads();
    // rows out: lanes take consecutive x of one row
#pragma unroll
    for (int q = 0; q < kResTile / 8; ++q) {
        const int oy = lx + 8 * q, ox = ly;
        float* o = a.intensity + (size_t)(Y0 + oy) * n + X0 + ox;
        const float v = tile[ox][oy];
        *o = a.accumulate ? *o + v : v;
    }
}

// Plain form for grids below one tile.
__global__ void resample_kernel(ResampleArgs a) {
    const int n = a.n;
    const size_t total = (size_t)n * n;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int X = (int)(i % n), Y = (int)(i / n);
        float acc = 0.0f;
        for (int l = 0; l < a.count; ++l) {
            const Sample sx = sample_at(X, n, a.r_fx[l]), sy = sample_at(Y, n, a.r_fx[l]);
            const int x0 = sx.i0 & (n - 1), y0 = sy.i0 & (n - 1);
            const int x1 = (x0 + 1) & (n - 1), y1 = (y0 + 1) & (n - 1);
            const float* h = a.pattern + (size_t)l * total;
            const float h00 = __ldg(h + (size_t)x0 * n + y0), h10 = __ldg(h + (size_t)x1 * n + y0);
            const float h01 = __ldg(h + (size_t)x0 * n + y1), h11 = __ldg(h + (size_t)x1 * n + y1);
            const float top = fmaf(sx.f, h10 - h00, h00), bot = fmaf(sx.f, h11 - h01, h01);
            acc = fmaf(a.weight[l], fmaf(sy.f, bot - top, top), acc);
        }
        a.intensity[i] = a.accumulate ? a.intensity[i] + acc : acc;
    }
}

cudaError_t launch_resample(const ResampleArgs& a, cudaStream_t s) {
    const bool tiled = a.n >= kResTile;
    if (tiled) {
        resample_tiled_kernel<<<dim3(a.n / kResTile, a.n / kResTile), 256, 0, s>>>(a);
        return cudaGetLastError();
    }
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const size_t total = (size_t)a.n * a.n;
    const int blocks = (int)std::min<size_t>((total + 255) / 256, (size_t)sms * 8);
    resample_kernel<<<blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace scint
