"""States of long shocks, alone and in a batch, against recorded ones.  At cfl = 100
with four relaxation sweeps the pseudo-time iteration of a Mach 4 line amplifies a
difference in the last bit to 1e-8 of the state in five iterations and 1e-4 in
twenty, so these states hold the rounding of every FP64 operation of a line's
iteration (records, moments, high-order terms, synthetic solve, correction).  The
tolerances are those of the outputs' types, 2-norm of the difference over that of
the result: 1e-9 in FP64, 2e-5 in FP32."""
import os

import numpy as np
import pytest

from workloads import shock_1d_case

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "shock_lines.txt")
TOL = {"f64": 1e-9, "f32": 2e-5}


def _recorded(dtype):
    rows = [l.split() for l in open(GOLDEN) if l.startswith(dtype)]
    return np.array([int(r[1]) for r in rows]), np.array([[float(x) for x in r[2:]] for r in rows])


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("dtype,iterations", [("f64", 5), ("f32", 20)])
def test_long_shocks_end_in_the_recorded_states(dtype, iterations, batched):
    from paper_2501_02245_gb300 import Solver, iterate_batch
    case = shock_1d_case(Ma=4.0, n_cells=400, half_width=50.0, nv=(32, 20, 16), vmax=17.0, macro_steps=50)
    s = Solver.from_case(case, vdf_dtype=dtype, tol=0.0)
    if batched:
        other = Solver.from_case(shock_1d_case(n_cells=60, half_width=7.5, nv=(16, 8, 8), vmax=9.0), vdf_dtype="f32", tol=0.0)
        iterate_batch([other, s], iterations)
        other.close()
    else:
        s.iterate(iterations)
    W, hot = s.W(), s.hot()
    s.close()
    cells, ref = _recorded(dtype)
    got = np.stack([W[cells, 0], W[cells, 1], W[cells, 4], hot[cells, 0], hot[cells, 6]], axis=1)
    for q, name in enumerate(("rho", "ux", "T", "hot_sxx", "hot_qx")):
        e = np.linalg.norm(got[:, q] - ref[:, q]) / np.linalg.norm(ref[:, q])
        assert e < TOL[dtype], "%s %.2e" % (name, e)
