"""The two-lane face fluxes round as the one-lane form: the fused synthetic
solve (two lanes per face while they fit) and the per-phase kernels (one) give
the same bits, at chunks of 16 faces that end before, at and after the last
face, with far-field and wall sides in one to three directions."""
import numpy as np
import pytest

from workloads import cylinder_case, shock_1d_case, sphere_case

pytestmark = pytest.mark.gpu


def _line(cells):
    return shock_1d_case(Ma=3.0, n_cells=cells, half_width=cells / 4.0, nv=(12, 10, 8), vmax=10.0, macro_steps=20)


def _body(case):
    case.dt = 0.5
    return case


CASES = {
    "line_5": lambda: _line(5), "line_16": lambda: _line(16), "line_33": lambda: _line(33), "line_496": lambda: _line(496),
    "line_497": lambda: _line(497),
    "cylinder": lambda: _body(cylinder_case(Ma=2.0, Kn=0.1, n_r=6, n_theta=8, nv=(14, 12, 6), adaptive=False, macro_steps=10,
                                            vbox=((-10, 10), (-9, 9), (-8, 8)))),
    "sphere": lambda: _body(sphere_case(Ma=2.0, Kn=0.1, n_r=3, n_pol=4, n_az=4, nv=(10, 8, 8), adaptive=False, macro_steps=5,
                                        vbox=((-10, 10), (-9, 9), (-9, 9)))),
}


@pytest.mark.parametrize("name", list(CASES))
def test_fused_and_per_phase_solves_give_the_same_bits(name):
    from paper_2501_02245_gb300 import Solver
    W = []
    for path in ("fused", "multi"):
        s = Solver.from_case(CASES[name]())
        s.set_macro_path(path)
        s.iterate(2)
        W.append(s.W())
        s.close()
    assert np.array_equal(W[0], W[1])
