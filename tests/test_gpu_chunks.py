"""The chunked reductions and corrections of FP32 arithmetic (x-rows of whole
16-byte chunks) at the sizes where they can go wrong: one chunk per row, odd chunk
counts, partial strips of iy and partial groups of planes, walls, the reduced grid.
The carried moments must equal a direct reduction of the stored VDF: the stored
values are rounded (one half unit each, 2^-24 for FP32; a whole unit, 2^-8 and
2^-11, for the stochastic rounding of BF16 and FP16) and the FP32 row sums of at
most 24 terms carry 24 * 2^-24; the bounds are twice the sum of the two."""
import numpy as np
import pytest

from workloads import cylinder_case, sphere_case, shock_1d_case
from helpers import run_gpu, run_oracle, rel_err, moment_scales

pytestmark = pytest.mark.gpu

UNIT = {"f32": 2.0 ** -24, "bf16": 2.0 ** -8, "f16": 2.0 ** -11}
BOUND = {"f32": 2e-5, "bf16": 3.9e-3, "f16": 9.8e-4}


def _cylinder(nv, reduced=False):
    vbox = ((-10, 10), (-9, 9), (0, 1) if reduced else (-8, 8))
    c = cylinder_case(Ma=2.0, Kn=0.1, n_r=6, n_theta=8, nv=nv, vbox=vbox, adaptive=False, macro_steps=10, relax=1.0,
                      reduced=reduced)
    c.dt = 0.5
    return c


@pytest.mark.parametrize("dtype", list(UNIT))
@pytest.mark.parametrize("nv", [(8, 11, 7), (16, 10, 8), (24, 13, 6), (24, 9, 9), (16, 10, 0)])
def test_carried_moments_equal_a_direct_reduction(dtype, nv):
    case = _cylinder(nv[:2] + (2,), reduced=True) if nv[2] == 0 else _cylinder(nv)
    _, ho = run_oracle(case, 2)
    s, hg, reps = run_gpu(case, 2, vdf_dtype=dtype)
    W = hg[-1]
    assert max(rel_err(W[:, 0], ho[-1][:, 0]), rel_err(W[:, 4], ho[-1][:, 4])) < BOUND[dtype]
    nd = reps[-1]["n_dvm"]
    carried = s.vdf_moments(nd, direct=False)
    direct = s.vdf_moments(nd, direct=True)
    err = (np.abs(carried - direct) / moment_scales(direct)).max()
    assert np.abs(direct[:, 13:]).max() > 0   # the case has diffuse-wall cells
    s.close()
    assert err < 2 * (UNIT[dtype] + 24 * 2.0 ** -24), "%.3e" % err
