// Single-solve launch of the 1D line sweep (sweep_line.cuh): one warp per tile.
#include <algorithm>
#include "sweep_line.cuh"

namespace gsis {

template <typename S, typename T, int ZP>
__global__ void __launch_bounds__(128) k_sweep_line(SweepArgs a, S* __restrict__ f, int N, int ntiles, int pass) {
    __shared__ LineStage stages[std::is_same<T, double>::value ? 1 : 4];
    __shared__ LineEnds<T, ZP> ends[4];
    const int w = threadIdx.x >> 5, tile = blockIdx.x * 4 + w;   // four warps: one per SM sub-partition
    if (tile < ntiles)   // pass 1: backward, step 0
        line_tile<S, T, ZP>(a, f, N, tile, threadIdx.x & 31, 1 - pass, 2 - pass,
                            &stages[std::is_same<T, double>::value ? 0 : w], ends[w]);
}

// One cell per hyperplane, every cell kinetic, no periodic wrap: row k is cell
// k and its neighbours are rows k - 1 and k + 1.  (The kernels keep a row's
// bytes in 32 bits.)
bool line_ok(const gsis_ctx* c) {
    return c->normal_components == 1 && c->m.nj == 1 && c->m.nk == 1 && c->m.bc_type[0] != GSIS_BC_PERIODIC &&
           c->Nd == c->m.N && c->Nd > 0 && (double)c->vg.Nv * vdf_elem_bytes(c->p.vdf_dtype) < 2147483648.0;
}

static int tiles(const gsis_ctx* c, int zp) { return (c->vg.nx * c->vg.ny + 31) / 32 * ((c->vg.nz + zp - 1) / zp); }
int line_tiles(const gsis_ctx* c, int planes64) { return tiles(c, c->p.vdf_dtype == GSIS_F64 ? planes64 : LINE_ZP32); }

int fp64_pipes() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return 4 * std::max(1, sms);
}

// Planes per column of an FP64 line alone, 0 for the general sweep.  One plane and the
// general sweep take 18 FP64 operations per point, two planes 15.  One plane wins while no
// sub-partition has two warps (30 cells, 1,800 velocities, 63 tiles on 608 sub-partitions:
// 74 us against 85; 200 cells, 15,360 velocities, 480 tiles: 405 against 476).  With two
// planes the busiest sub-partition's warps set the time, 0.46 ms for each on 200 cells; the
// general sweep has twice the tiles and evens out at 0.56 ms for each warp of two planes that a
// sub-partition would have in the mean.  So two planes are taken where the most is at most 1.2
// times the mean: 1,296 tiles (3 and 2.1) 1.39 ms against 1.20, 1,728 (3 and 2.8) 1.39
// against 1.58, 2,304 (4 and 3.8) 1.85 against 2.25, 4,096 (7 and 6.7) 3.22 against 3.71.  Below
// two warps each the general sweep's five-value loads cost nothing (27,648 velocities: 0.52
// ms against 0.62).
static int line_planes64(const gsis_ctx* c) {
    const int n = tiles(c, 2), pipes = fp64_pipes(), most = (n + pipes - 1) / pipes;
    if (n >= 2 * pipes) return 5LL * most * pipes <= 6LL * n ? 2 : 0;
    return tiles(c, 1) <= pipes ? 1 : 0;
}

bool line_alone(const gsis_ctx* c) {
    return line_ok(c) && (c->p.vdf_dtype != GSIS_F64 || line_planes64(c) > 0);
}

template <typename S, typename T, int ZP>
static void launch(gsis_ctx* c, const SweepArgs& a, int pass) {
    const int nt = tiles(c, ZP);
    k_sweep_line<S, T, ZP><<<(nt + 3) / 4, 128, 0, c->stream>>>(a, (S*)c->f, (int)c->Nd, nt, pass);
}

void launch_sweep_line(gsis_ctx* c, const SweepArgs& a, int pass) {
    switch (c->p.vdf_dtype) {
        case GSIS_F64:
            if (line_planes64(c) == 2) launch<double, double, 2>(c, a, pass);
            else launch<double, double, 1>(c, a, pass);
            break;
        case GSIS_F32: launch<float, float, LINE_ZP32>(c, a, pass); break;
        case GSIS_BF16: launch<__nv_bfloat16, float, LINE_ZP32>(c, a, pass); break;
        default: launch<__half, float, LINE_ZP32>(c, a, pass); break;
    }
}

}  // namespace gsis
