// Asynchronous tile loads of the propagation passes: TMA copies into shared memory that
// complete on an mbarrier, issued by one thread of the block an item ahead of its use.
//
// The waits are bounded: wait_tile gives up after kTileWaitTries attempts (each suspends for
// a while in hardware; far longer than any copy takes) and reports it; the kernels then write
// NaN, so that a copy that never completes shows in the result instead of hanging the GPU.
#pragma once

#include <cuda.h>

#include "propagate.cuh"

namespace scint {

constexpr int kTileWaitTries = 1 << 20;

SCINT_DEV unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

SCINT_DEV void tile_init(unsigned long long* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
// make the initialised barriers visible to the asynchronous proxy (one thread, before the block barrier)
SCINT_DEV void tile_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// order this thread's (and, after a block barrier, the block's) earlier accesses to shared memory
// before the asynchronous writes issued next
SCINT_DEV void tile_reuse_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

SCINT_DEV void tile_expect(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// contiguous bytes (a multiple of 16, both addresses 16-byte aligned)
SCINT_DEV void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// the box of a 2D tensor at (x, y); x times the element size is a multiple of 16 bytes
SCINT_DEV void box_load(void* dst, const CUtensorMap* tm, int x, int y, unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<unsigned long long>(tm)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}
SCINT_DEV bool wait_tile(unsigned long long* bar, unsigned parity) {
    const unsigned addr = smem_u32(bar);
    for (int i = 0; i < kTileWaitTries; ++i) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// ---- columns of a strip-layout field ---------------------------------------------
// The fields of a wavelength group are one matrix of rows of pstrip<N>() values: row
// (l N / WL + strip) N + y.  A column block's W = pcol_lines<N>() columns are W/2 boxes of two
// values (16 bytes, the least a box may have) by N rows at its strip (boxes of 256 rows), dense
// in shared memory: value (y, w) at ((w / 2) N + y) 2 + w % 2.
template <int N> __host__ __device__ constexpr bool col_stream() { return col_teams<N>(); }
template <int N> __host__ __device__ constexpr size_t col_stage_bytes() { return (size_t)N * pcol_lines<N>() * sizeof(float2); }
constexpr int kBoxRows = 256, kBoxCols = 2;

template <int N>
SCINT_DEV void issue_columns(float2* stage, const CUtensorMap* tm, int l, int x0, unsigned long long* bar) {
    constexpr int W = pcol_lines<N>(), WL = pstrip<N>();
    static_assert(W % kBoxCols == 0 && N % kBoxRows == 0, "whole boxes");
    tile_expect(bar, (unsigned)col_stage_bytes<N>());
    const int row = (l * (N / WL) + x0 / WL) * N, c = (x0 % WL) * 2;    // c: a multiple of 4 floats
#pragma unroll 1
    for (int i = 0; i < W / kBoxCols * (N / kBoxRows); ++i) {
        const int q = i / (N / kBoxRows), r = i % (N / kBoxRows) * kBoxRows;
        box_load(stage + (size_t)(q * N + r) * kBoxCols, tm, c + q * 2 * kBoxCols, row + r, bar);
    }
}

// The tensor map of `count` fields of an n x n grid at work (the driver's encoder, looked up
// once); false when it is not to be had, and the caller takes the plain loads.
bool field_map(CUtensorMap* tm, const float2* work, int n, int count, int strip);

// Blocks of a pass over `items` independent lines or tiles, each of `count` wavelengths: one
// item per block when a block has several wavelengths to spread its start over, else as many
// blocks as are resident, each walking items (the start, the twiddles and the first load once
// per block, the next item's load behind this one's work).
constexpr int kWalkBelow = 8;
template <typename K>
inline cudaError_t walk_blocks(K kernel, int threads, size_t smem, int items, int count, int* blocks) {
    *blocks = items;
    if (count >= kWalkBelow) return cudaSuccess;
    int resident = 0;
    const cudaError_t e = resident_blocks(kernel, threads, smem, &resident);
    if (e == cudaSuccess) *blocks = resident < items ? resident : items;
    return e;
}

}  // namespace scint
