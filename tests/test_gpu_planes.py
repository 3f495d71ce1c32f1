"""The velocity pairs on two planes (FP32 arithmetic) on 2D and 3D meshes against
the FP64 oracle at the sizes where they can go wrong: odd plane counts, partial
position tiles, hyperplanes with fewer cells than warps, walls, far field, the
periodic seams, polar faces without area, interfaces to NS cells and the reduced
grid.  Tolerances are the bounds of the precision tests."""
import numpy as np
import pytest

from workloads import cylinder_case, sphere_case
from helpers import run_oracle, rel_err

pytestmark = pytest.mark.gpu

BOUND = {"f32": 2e-5, "bf16": 3.9e-3, "f16": 9.8e-4}


def _check(case, dtype, flags=None):
    from paper_2501_02245_gb300 import Solver
    _, ho = run_oracle(case, 2, flags=flags)
    got = {}
    for name in ("p8_v1_c1", "planes", "planes_wide"):
        s = Solver.from_case(case, vdf_dtype=dtype, forced_flags=flags)
        s.set_sweep_tile(name)
        s.iterate(2)
        got[name] = s.W()
        s.close()
        e = max(rel_err(got[name][:, 0], ho[-1][:, 0]), rel_err(got[name][:, 4], ho[-1][:, 4]))
        assert e < BOUND[dtype], "%s: %.3e" % (name, e)
        # the operations and roundings of the other pair tiles (FP32 subnormals apart, far below W's last bit)
        assert np.array_equal(got[name], got["p8_v1_c1"]), name


def _cylinder(nv, adaptive=False, reduced=False):
    if reduced:
        c = cylinder_case(Ma=2.0, Kn=0.1, n_r=6, n_theta=8, nv=nv, vbox=((-10, 10), (-9, 9), (0, 1)), adaptive=False,
                          macro_steps=10, relax=1.0, reduced=True)
    else:
        c = cylinder_case(Ma=2.0, Kn=0.02 if adaptive else 0.1, n_r=8, n_theta=10, nv=nv, adaptive=adaptive,
                          Kn_ref=0.02, macro_steps=10, presolve_max_blocks=3, vbox=((-10, 10), (-9, 9), (-8, 8)))
        c.tol, c.adapt_every = 0.0, 1000
    c.dt = 0.5
    return c


@pytest.mark.parametrize("dtype", list(BOUND))
@pytest.mark.parametrize("nv", [(14, 12, 6), (14, 11, 7)])
def test_cylinder(dtype, nv):
    _check(_cylinder(nv), dtype)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_cylinder_at_ns_interfaces(dtype):
    case = _cylinder((14, 11, 7), adaptive=True)
    flags = run_oracle(case, 0)[0].dvm.copy()
    assert 0 < flags.sum() < flags.size
    _check(case, dtype, flags=flags)


def test_reduced_grid():
    _check(_cylinder((14, 11, 2), reduced=True), "f32")


@pytest.mark.parametrize("dtype", list(BOUND))
@pytest.mark.parametrize("nv", [(10, 8, 8), (10, 9, 7)])
def test_sphere(dtype, nv):
    case = sphere_case(Ma=2.0, Kn=0.1, n_r=3, n_pol=4, n_az=4, nv=nv, adaptive=False, macro_steps=5,
                       vbox=((-10, 10), (-9, 9), (-9, 9)))
    case.dt = 0.5
    _check(case, dtype)


def test_an_odd_row_is_refused():
    from paper_2501_02245_gb300 import Solver, GsisError
    s = Solver.from_case(_cylinder((13, 12, 6)), vdf_dtype="f32")
    with pytest.raises(GsisError):
        s.set_sweep_tile("planes")
    s.close()
