// Pair sweep of two planes (sweep_planes.cuh), F32 storage.
#include "sweep_planes.cuh"

namespace gsis {

void launch_sweep_planes_f32(gsis_ctx* c, const SweepArgs& a, int pass, int shape) {
    launch_planes<float>(c, a, pass, shape);
}

}  // namespace gsis
