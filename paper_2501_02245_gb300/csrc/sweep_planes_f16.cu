// Pair sweep of two planes (sweep_planes.cuh), F16 storage.
#include "sweep_planes.cuh"

namespace gsis {

void launch_sweep_planes_f16(gsis_ctx* c, const SweepArgs& a, int pass, int shape) {
    launch_planes<__half>(c, a, pass, shape);
}

}  // namespace gsis
