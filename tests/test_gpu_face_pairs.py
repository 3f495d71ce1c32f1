"""The two-lane face fluxes of the fused synthetic solve against the per-phase
kernels (one lane per face) at the sizes where they can go wrong: chunks of 16
faces that end before, at and after the last face, the largest solve that takes
them and the first that does not, and meshes with walls, periodic seams and
faces without area.  The tolerance is that of the other FP64 parity tests."""
import pytest

from workloads import cylinder_case, shock_1d_case, sphere_case
from helpers import w_rel_err, RTOL_W

pytestmark = pytest.mark.gpu


def _check(case):
    from paper_2501_02245_gb300 import Solver
    W = []
    for path in ("fused", "multi"):
        s = Solver.from_case(case)
        s.set_macro_path(path)
        s.iterate(2)
        W.append(s.W())
        s.close()
    assert w_rel_err(W[0], W[1]) < RTOL_W, "%.3e" % w_rel_err(W[0], W[1])


@pytest.mark.parametrize("cells", [5, 15, 16, 17, 33, 127, 128, 496, 497])
def test_lines(cells):
    _check(shock_1d_case(Ma=1.6, n_cells=cells, half_width=cells / 4.0, nv=(12, 10, 8), vmax=8.0, macro_steps=10))


def test_cylinder():
    case = cylinder_case(Ma=2.0, Kn=0.1, n_r=6, n_theta=8, nv=(14, 12, 6), adaptive=False, macro_steps=10,
                         cfl=5.0, k_sub=2, vbox=((-10, 10), (-9, 9), (-8, 8)))
    case.dt = 0.5
    _check(case)


def test_sphere():
    case = sphere_case(Ma=2.0, Kn=0.1, n_r=3, n_pol=4, n_az=4, nv=(10, 8, 8), adaptive=False, macro_steps=5,
                       vbox=((-10, 10), (-9, 9), (-9, 9)))
    case.dt = 0.5
    _check(case)
