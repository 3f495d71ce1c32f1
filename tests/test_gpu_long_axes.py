"""Iterations on velocity grids with long x axes, where the moment pass's tables
take more of the shared memory: around the length that fits 256 threads' sums (168
FP64, 336 FP32 nodes), 128 threads' (776) and past it, against the FP64 oracle.
Tolerances: FP64 1e-10, FP32 2e-5, as in the other parity tests."""
import pytest

from workloads import shock_1d_case
from helpers import run_oracle, w_rel_err, rel_err, RTOL_W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,dtype", [(168, "f64"), (169, "f64"), (200, "f64"), (777, "f64"), (337, "f32"), (344, "f32")])
def test_long_axes(nx, dtype):
    from paper_2501_02245_gb300 import Solver
    case = shock_1d_case(Ma=1.6, n_cells=6, half_width=1.5, nv=(nx, 16, 16), vmax=8.0, macro_steps=5)
    s = Solver.from_case(case, vdf_dtype=dtype)
    s.iterate(2)
    W = s.W()
    s.close()
    _, ho = run_oracle(case, 2)
    if dtype == "f64":
        assert w_rel_err(W, ho[-1]) < RTOL_W
    else:
        assert max(rel_err(W[:, 0], ho[-1][:, 0]), rel_err(W[:, 4], ho[-1][:, 4])) < 2e-5
