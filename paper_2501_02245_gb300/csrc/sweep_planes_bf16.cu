// Pair sweep of two planes (sweep_planes.cuh), BF16 storage.
#include "sweep_planes.cuh"

namespace gsis {

void launch_sweep_planes_bf16(gsis_ctx* c, const SweepArgs& a, int pass, int shape) {
    launch_planes<__nv_bfloat16>(c, a, pass, shape);
}

}  // namespace gsis
