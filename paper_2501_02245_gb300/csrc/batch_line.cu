// Batched persistent sweep of 1D lines: items are (solve, warp tile) pairs drawn
// from the ticket counter as in batch_kernel.cuh; a warp walks the line of its
// tile with the window of sweep_line.cuh, both passes (both passes' launches
// where walls need a refresh between them).
#include <algorithm>
#include "batch_kernel.cuh"
#include "sweep_line.cuh"

namespace gsis {

constexpr int LINE_WPB = 4;

// Z64: the FP64 members' items with Z64 planes per column (the others are passed
// over), 0: the FP32-arithmetic ones; one kernel for both would give every item the
// FP64 code's registers.
template <int Z64>
__global__ void __launch_bounds__(32 * LINE_WPB, Z64 ? 3 : 4) k_sweep_batch_line(const BatchSolve* __restrict__ solves,
                                                                                 const int2* __restrict__ items,
                                                                                 int n_items, int* __restrict__ ticket,
                                                                                 int pass0, int pass1) {
    constexpr bool F64 = Z64 > 0;
    // the solve's arguments, one copy per warp: registers are the limit of this
    // kernel's occupancy (in the single launch they sit in the constant bank)
    __shared__ SweepArgs args[LINE_WPB];
    __shared__ LineStage stages[F64 ? 1 : LINE_WPB];
    using T = typename std::conditional<F64, double, float>::type;
    __shared__ LineEnds<T, F64 ? Z64 : LINE_ZP32> ends[LINE_WPB];
    auto& end = ends[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    SweepArgs& a = args[threadIdx.x >> 5];
    LineStage* stage = &stages[F64 ? 0 : threadIdx.x >> 5];
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(ticket, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= n_items) return;   // the counter only grows: every warp leaves after at most n_items draws
        const int2 it = items[t];
        const BatchSolve& B = solves[it.x];
        const int dtype = B.dtype;
        if ((dtype == GSIS_F64) != F64) continue;
        __syncwarp();   // the previous item's last reads
        for (int w = lane; w < (int)(sizeof(SweepArgs) / sizeof(int)); w += 32)
            reinterpret_cast<int*>(&a)[w] = reinterpret_cast<const int*>(&B.a)[w];
        __syncwarp();
        if constexpr (F64) {
            line_tile<double, double, Z64>(a, (double*)B.f, B.cells, it.y, lane, pass0, pass1, stage, end);
        } else {
            if (dtype == GSIS_F32)
                line_tile<float, float, LINE_ZP32>(a, (float*)B.f, B.cells, it.y, lane, pass0, pass1, stage, end);
            else if (dtype == GSIS_BF16)
                line_tile<__nv_bfloat16, float, LINE_ZP32>(a, (__nv_bfloat16*)B.f, B.cells, it.y, lane, pass0, pass1, stage, end);
            else
                line_tile<__half, float, LINE_ZP32>(a, (__half*)B.f, B.cells, it.y, lane, pass0, pass1, stage, end);
        }
    }
}

template <int Z64>
static int grid_of() {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sweep_batch_line<Z64>, 32 * LINE_WPB, 0);
    return std::max(1, sms * std::max(1, per));
}

int batch_grid_line(int planes64) { return planes64 == 2 ? grid_of<2>() : (planes64 == 1 ? grid_of<1>() : grid_of<0>()); }

void batch_launch_line(const BatchSolve* s, const int2* i, int n, int* t, int grid, cudaStream_t st, int p0, int p1,
                       int planes64) {
    if (planes64 == 2) k_sweep_batch_line<2><<<grid, 32 * LINE_WPB, 0, st>>>(s, i, n, t, p0, p1);
    else if (planes64 == 1) k_sweep_batch_line<1><<<grid, 32 * LINE_WPB, 0, st>>>(s, i, n, t, p0, p1);
    else k_sweep_batch_line<0><<<grid, 32 * LINE_WPB, 0, st>>>(s, i, n, t, p0, p1);
}

}  // namespace gsis
