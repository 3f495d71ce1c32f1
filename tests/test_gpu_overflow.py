"""A value that overflows its storage in one pass (FP16: a cold wall that emits
for a dense hot cell beside it) and is formed again in the next one spoils what it
flows into and nothing else.  The pairs on two planes, which weigh the face value
of an outflow side with zero, end with the values of the pair tiles, which select:
a solve that comes through with those comes through with these."""
import numpy as np
import pytest

from workloads import cylinder_case, sphere_case

pytestmark = pytest.mark.gpu

BOX = ((-10, 10), (-10, 10), (-10, 10))
COMMON = dict(Ma=0.5, Kn=20.0, adaptive=False, macro_steps=1, k_sub=0, cfl=0.1, presolve_max_blocks=0, vbox=BOX, wall_T=0.6,
              first_cell_mfp=0.002)


def _cylinder():
    return cylinder_case(n_r=8, n_theta=10, nv=(14, 12, 5), **COMMON)


def _sphere():
    return sphere_case(n_r=5, n_pol=6, n_az=6, nv=(12, 10, 9), **COMMON)


# wall cell, its density at four times the gas's temperature, whether the pair tiles come through
@pytest.mark.parametrize("make,cell,rho,through", [(_cylinder, 40, 1000.0, True), (_cylinder, 40, 1500.0, False),
                                                   (_sphere, 100, 1000.0, True), (_sphere, 115, 1000.0, False)])
def test_an_overflow_stays_downstream(make, cell, rho, through):
    from paper_2501_02245_gb300 import Solver, GsisError
    case = make()
    case.W0 = np.array(case.W0)
    case.W0[cell] = [rho, 0.0, 0.0, 0.0, 4.0]
    out = []
    for tile in ("p8_v1_c1", "planes", "planes_wide"):
        s = Solver.from_case(case, vdf_dtype="f16")
        s.set_sweep_tile(tile)
        if through:
            s.iterate(1)
        else:
            with pytest.raises(GsisError):
                s.iterate(1)
        out.append(s.vdf(case.mesh.ncell)[1])
        s.close()
    assert np.isfinite(out[0]).all() == through
    for f in out[1:]:
        assert np.array_equal(f, out[0], equal_nan=True)
