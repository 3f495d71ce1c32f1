// Host side of the batched persistent sweep: the candidate tile shapes, the
// grid size of each (resident CTAs per SM x SMs) and the launch.  The kernel
// is in batch_kernel.cuh, instantiated in batch_nc1.cu and batch_nc3.cu.
#include "batch_kernel.cuh"

namespace gsis {

// ---------------------------------------------------------------------------- candidates
struct TileShape {
    int vpt, cb, wpb;
    int kind;    // 0: single velocities; 1: velocity pairs with packed FP32 arithmetic (FP32/BF16/FP16 members with an even nx only);
                 // 2: 1D lines (sweep_line.cuh; every member a line), vpt: planes per column of the FP64 members
    const char* name;
};

static const TileShape kShapes[] = {
    {1, 1, 4, 0, "vpt1_cb1_w4"}, {2, 1, 4, 0, "vpt2_cb1_w4"}, {4, 1, 4, 0, "vpt4_cb1_w4"},
    {2, 1, 8, 0, "vpt2_cb1_w8"}, {2, 2, 4, 0, "vpt2_cb2_w4"}, {4, 2, 2, 0, "vpt4_cb2_w2"},
    {1, 1, 4, 1, "pair1_cb1_w4"}, {2, 1, 4, 1, "pair2_cb1_w4"}, {1, 1, 8, 1, "pair1_cb1_w8"},
    {2, 0, 4, 2, "line_w4"}, {1, 0, 4, 2, "line1_w4"},
};
constexpr int kNumShapes = sizeof(kShapes) / sizeof(kShapes[0]);

int batch_num_shapes() { return kNumShapes; }
const char* batch_shape_name(int s) { return (s >= 0 && s < kNumShapes) ? kShapes[s].name : "?"; }
int batch_shape_vtile(int s) { return (kShapes[s].kind == 1 ? 64 : 32) * kShapes[s].vpt; }
bool batch_shape_pair(int s) { return s >= 0 && s < kNumShapes && kShapes[s].kind == 1; }
bool batch_shape_line(int s) { return s >= 0 && s < kNumShapes && kShapes[s].kind == 2; }
int batch_shape_planes64(int s) { return kShapes[s].vpt; }

int batch_grid(int shape, int nc) {
    if (batch_shape_line(shape)) return batch_grid_line(0);
    return nc == 1 ? batch_grid_nc1(shape) : batch_grid_nc3(shape);
}

// types: members with FP32 arithmetic (1), FP64 (2), both (3).
// Steps pass0 .. pass1-1 of every item: step 0 is the backward pass, step 1 the forward pass.
void launch_sweep_batch(int shape, int nc, const BatchSolve* d_solves, const int2* d_items, int n_items,
                        int* d_ticket, int grid, cudaStream_t st, int pass0, int pass1, int types) {
    cudaMemsetAsync(d_ticket, 0, sizeof(int), st);
    if (batch_shape_line(shape)) {   // the FP32-arithmetic members, then the FP64 ones
        const int planes64 = batch_shape_planes64(shape);
        if (types & 1) batch_launch_line(d_solves, d_items, n_items, d_ticket, grid, st, pass0, pass1, 0);
        if (types & 2) {
            if (types & 1) cudaMemsetAsync(d_ticket, 0, sizeof(int), st);
            batch_launch_line(d_solves, d_items, n_items, d_ticket, batch_grid_line(planes64), st, pass0, pass1, planes64);
        }
        return;
    }
    if (nc == 1)
        batch_launch_nc1(shape, d_solves, d_items, n_items, d_ticket, grid, st, pass0, pass1);
    else
        batch_launch_nc3(shape, d_solves, d_items, n_items, d_ticket, grid, st, pass0, pass1);
}

}  // namespace gsis
