// Launchers of the batched probe kernels (see cht_ops.cuh).
#include <atomic>

#include "cht_grid.h"
#include "cht_ops.cuh"
#include "cht_per_device.h"

namespace cht {
namespace {

// Empties a table: zero cells, zero state.  One launch in the chain of
// overlapping ones (see pdl_enter) instead of two memsets between them, which
// break it: clear + insert + find on 2^20 cells 42.2 -> 36.0 us a pass.  Tables
// up to kClearLog2 only: this kernel's 32-byte stores reach 6.2 TB/s (2^22
// cells 10.6 us, two memsets 13.6; 2^24 43.0 and 39.8; 2^28 654 and 556), so
// larger ones are memset.
constexpr u32 kClearLog2 = 22;

__global__ void __launch_bounds__(256) clear_kernel(OpArgs a) {
    pdl_enter();
    const u64 pairs = (1ull << a.log2c) / 2, stride = u64(gridDim.x) * 256;
    for (u64 i = u64(blockIdx.x) * 256 + threadIdx.x; i < pairs; i += stride)
        asm volatile("st.global.v4.u64 [%0], {%1,%1,%1,%1};" ::"l"(a.cells + 2 * i), "l"(0ull) : "memory");
    if (blockIdx.x == 0 && threadIdx.x < sizeof(DevState) / 8) reinterpret_cast<u64*>(a.st)[threadIdx.x] = 0;
}
static_assert(sizeof(DevState) % 8 == 0 && sizeof(DevState) / 8 <= 256, "one word per thread");

template <int G, int V, int MODE, int kFlags = 0>
cudaError_t launch_one(const OpArgs& a, int ctas_per_sm, cudaStream_t s) {
    static std::atomic<int> occ{0};
    int per_sm = occ.load(std::memory_order_relaxed);
    if (per_sm == 0) {
        cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, op_kernel<G, V, MODE, kFlags>, kOpBlock, 0);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        occ.store(per_sm, std::memory_order_relaxed);
    }
    if (ctas_per_sm > 0 && ctas_per_sm < per_sm) per_sm = ctas_per_sm;
    u64 grid = u64(sm_count()) * u64(per_sm);
    const u64 need = (a.n + kOpBlock - 1) / kOpBlock;
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    const cudaError_t e = launch_overlapped(op_kernel<G, V, MODE, kFlags>, unsigned(grid), kOpBlock, 0, s, a);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Per-thread operations (group_width = -1), V = 2 or 4 cells per step.
template <int V, int MODE>
cudaError_t launch_thread_v(const OpArgs& a, int ctas_per_sm, cudaStream_t s) {
    static std::atomic<int> occ{0};
    int per_sm = occ.load(std::memory_order_relaxed);
    if (per_sm == 0) {
        cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, thread_kernel<V, MODE>, kThreadBlock, 0);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        occ.store(per_sm, std::memory_order_relaxed);
    }
    const u64 grid =
        thread_grid((a.n + kThreadBlock - 1) / kThreadBlock, u64(sm_count()), u64(per_sm), ctas_per_sm, MODE != kFind);
    const cudaError_t e = launch_overlapped(thread_kernel<V, MODE>, unsigned(grid), kThreadBlock, 0, s, a);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int MODE>
cudaError_t launch_thread(const OpArgs& a, int v, int ctas_per_sm, cudaStream_t s) {
    return v == 2 ? launch_thread_v<2, MODE>(a, ctas_per_sm, s) : launch_thread_v<4, MODE>(a, ctas_per_sm, s);
}

// Tables with tombstone reuse or the full key space: kernels exist for the
// automatic windows only -- 1 lane x 1 sector, 2 lanes x 2 sectors, 4 lanes x
// 1 or 2 sectors; any other configured window takes the nearest of these.
template <int MODE, int F>
cudaError_t launch_window(const OpArgs& a, int g, int v, int ctas_per_sm, cudaStream_t s) {
    if (g <= 1) return launch_one<1, 2, MODE, F>(a, ctas_per_sm, s);
    if (g == 2) return launch_one<2, 4, MODE, F>(a, ctas_per_sm, s);
    if (g == 4 && v != 4) return launch_one<4, 2, MODE, F>(a, ctas_per_sm, s);
    return launch_one<4, 4, MODE, F>(a, ctas_per_sm, s);
}

template <int MODE>
cudaError_t launch_flagged(const OpArgs& a, int g, int v, int flags, int ctas_per_sm, cudaStream_t s) {
    constexpr bool fills = mode_fills(MODE);
    switch (flags) {
        case kFlagReuse:
            if constexpr (fills) return launch_window<MODE, kFlagReuse>(a, g, v, ctas_per_sm, s);
            break;
        case kFlagFullKeys: return launch_window<MODE, kFlagFullKeys>(a, g, v, ctas_per_sm, s);
        case kFlagReuse | kFlagFullKeys:
            if constexpr (fills) return launch_window<MODE, kFlagReuse | kFlagFullKeys>(a, g, v, ctas_per_sm, s);
            break;
        default: break;
    }
    return cudaErrorInvalidValue;
}

// Up to 2^25 cells the finds of the two windows in use there store each result
// as it comes: L2 holds a good part of the table, its requests don't bound the
// finds, and the ring's instructions cost as much as it saves or more (load 0.7,
// direct against ring: 2^22 finds on 2^22 cells 108 and 116 us, 2^23 on 2^23 165
// and 188 us, 2^24 on 2^24 442 and 459 us, 2^24 on 2^25 535 and 541 us; for
// 2^26 cells see kRingOps).
constexpr u32 kDirectLog2 = 25;

// (group width G, cells per lane V): G = 1 always loads a whole sector.
template <int MODE>
cudaError_t launch_mode(const OpArgs& a, int g, int v, int ctas_per_sm, cudaStream_t s) {
    const int flags = ((mode_fills(MODE) && a.reuse) ? kFlagReuse : 0) | (a.full_keys ? kFlagFullKeys : 0);
    if (g < 0) {
        // the per-thread kernels: plain tables, the whole batch in one
        // grid-stride pass (in-order pieces take the 1-lane group loop)
        if (!flags && a.chunk == 0) return launch_thread<MODE>(a, v, ctas_per_sm, s);
        g = 1;
        if (v != 4) v = 2;
    }
    if (flags) return launch_flagged<MODE>(a, g, v, flags, ctas_per_sm, s);
    if (v == 4) {
        switch (g) {
            case 1:
                if constexpr (MODE == kFind)
                    if (a.log2c <= kDirectLog2) return launch_one<1, 4, MODE, kFlagDirect>(a, ctas_per_sm, s);
                return launch_one<1, 4, MODE>(a, ctas_per_sm, s);
            case 2:
                if constexpr (MODE == kFind)
                    if (a.log2c <= kDirectLog2) return launch_one<2, 4, MODE, kFlagDirect>(a, ctas_per_sm, s);
                return launch_one<2, 4, MODE>(a, ctas_per_sm, s);
            case 4: return launch_one<4, 4, MODE>(a, ctas_per_sm, s);
            case 8: return launch_one<8, 4, MODE>(a, ctas_per_sm, s);
            default: return cudaErrorInvalidValue;
        }
    }
    if (v == 2) {
        switch (g) {
            case 1: return launch_one<1, 2, MODE>(a, ctas_per_sm, s);
            case 2: return launch_one<2, 2, MODE>(a, ctas_per_sm, s);
            case 4: return launch_one<4, 2, MODE>(a, ctas_per_sm, s);
            case 8: return launch_one<8, 2, MODE>(a, ctas_per_sm, s);
            case 16: return launch_one<16, 2, MODE>(a, ctas_per_sm, s);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (g) {
        case 1: return launch_one<1, 2, MODE>(a, ctas_per_sm, s);
        case 2: return launch_one<2, 1, MODE>(a, ctas_per_sm, s);
        case 4: return launch_one<4, 1, MODE>(a, ctas_per_sm, s);
        case 8: return launch_one<8, 1, MODE>(a, ctas_per_sm, s);
        case 16: return launch_one<16, 1, MODE>(a, ctas_per_sm, s);
        case 32: return launch_one<32, 1, MODE>(a, ctas_per_sm, s);
        default: return cudaErrorInvalidValue;
    }
}

template <int MODE, bool RE, int BLOCK = kAggBlock>
cudaError_t launch_agg(const OpArgs& a, int ctas_per_sm, cudaStream_t s) {
    constexpr size_t smem = agg_smem_bytes<MODE, BLOCK>();
    static PerDevice known;
    int dev = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = known.get(dev, &per_sm, [&](int* n) {
        const auto fn = iou_agg_kernel<MODE, RE, BLOCK>;
        cudaError_t q = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        // as much of the unified L1 / shared memory as shared memory as the
        // kernel can use (38 KB per 256-thread CTA, 152 KB per 1024-thread CTA)
        if (q == cudaSuccess) q = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (q == cudaSuccess) q = cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, fn, BLOCK, smem);
        if (*n < 1) *n = 1;
        return q;
    });
    if (e != cudaSuccess) return e;
    if (ctas_per_sm > 0 && ctas_per_sm < per_sm) per_sm = ctas_per_sm;
    u64 grid = u64(sm_count()) * u64(per_sm);
    const u64 nwin = (a.n + 4 * BLOCK - 1) / (4 * BLOCK);
    if (grid > nwin) grid = nwin;
    if (grid < 1) grid = 1;
    e = launch_overlapped(iou_agg_kernel<MODE, RE, BLOCK>, unsigned(grid), BLOCK, smem, s, a);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_clear(Cell* cells, u32 log2c, DevState* st, cudaStream_t s) {
    if (log2c > kClearLog2) {
        const cudaError_t e = cudaMemsetAsync(cells, 0, (1ull << log2c) * sizeof(Cell), s);
        return e != cudaSuccess ? e : cudaMemsetAsync(st, 0, sizeof(DevState), s);
    }
    OpArgs a{};
    a.cells = cells;
    a.log2c = log2c;
    a.st = st;
    u64 grid = ((1ull << log2c) / 2 + 255) / 256;
    const u64 most = u64(sm_count()) * 8;
    if (grid > most) grid = most;
    const cudaError_t e = launch_overlapped(clear_kernel, unsigned(grid), 256, 0, s, a);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_iou_aggregated(Mode mode, const OpArgs& a, int ctas_per_sm, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    const bool re = a.reuse != 0;
    switch (mode) {
        case kIouAdd: return re ? launch_agg<kIouAdd, true>(a, ctas_per_sm, s) : launch_agg<kIouAdd, false>(a, ctas_per_sm, s);
        case kIouOverwrite:
            return re ? launch_agg<kIouOverwrite, true>(a, ctas_per_sm, s)
                      : launch_agg<kIouOverwrite, false>(a, ctas_per_sm, s);
        // update: equal keys fold the same way; no cell is filled, so tombstone
        // reuse does not apply
        case kUpdAdd: return launch_agg<kUpdAdd, false>(a, ctas_per_sm, s);
        case kUpdOverwrite: return launch_agg<kUpdOverwrite, false>(a, ctas_per_sm, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_iou_aggregated_wide(Mode mode, const OpArgs& a, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    const bool re = a.reuse != 0;
    if (mode == kIouAdd) return re ? launch_agg<kIouAdd, true, 1024>(a, 0, s) : launch_agg<kIouAdd, false, 1024>(a, 0, s);
    if (mode == kIouOverwrite)
        return re ? launch_agg<kIouOverwrite, true, 1024>(a, 0, s) : launch_agg<kIouOverwrite, false, 1024>(a, 0, s);
    return cudaErrorInvalidValue;
}

cudaError_t launch_op(Mode mode, const OpArgs& a, int group_width, int lane_cells, int ctas_per_sm,
                      cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    const int v = lane_cells;
    switch (mode) {
        case kFind: return launch_mode<kFind>(a, group_width, v, ctas_per_sm, s);
        case kInsert: return launch_mode<kInsert>(a, group_width, v, ctas_per_sm, s);
        case kIouAdd: return launch_mode<kIouAdd>(a, group_width, v, ctas_per_sm, s);
        case kIouOverwrite: return launch_mode<kIouOverwrite>(a, group_width, v, ctas_per_sm, s);
        case kErase: return launch_mode<kErase>(a, group_width, v, ctas_per_sm, s);
        case kUpdAdd: return launch_mode<kUpdAdd>(a, group_width, v, ctas_per_sm, s);
        case kUpdOverwrite: return launch_mode<kUpdOverwrite>(a, group_width, v, ctas_per_sm, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace cht
