// Single-solve launch of the 1D line sweep (sweep_line.cuh): one warp per tile.
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
int line_tiles(const gsis_ctx* c) { return tiles(c, c->p.vdf_dtype == GSIS_F64 ? LINE_ZP64 : LINE_ZP32); }

// Planes per column of an FP64 line alone, 0 for the general sweep.  Two planes
// take 15 FP64 operations per point, one plane and the general sweep 18.  A single
// warp fills only 60 % of its sub-partition's FP64 pipe, so two planes need two
// warps for each of the 608 sub-partitions; one plane wins while no sub-partition
// has two warps (30 cells, 1,800 velocities: 74 us against 83); between them
// the general sweep's five-value loads cost nothing (200 cells, 27,648
// velocities: 518 us against 622).
static int line_planes64(const gsis_ctx* c) { return tiles(c, 2) >= 1216 ? 2 : (tiles(c, 1) <= 608 ? 1 : 0); }

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
