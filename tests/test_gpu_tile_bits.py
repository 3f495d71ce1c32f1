"""Every tile of the FP64 sweep gives the bits of the general one: a solve must
not depend on which tile the autotuner's clock picked.  2D meshes with walls,
far field, the periodic seam, interfaces to NS cells and the reduced grid, with
odd axes and ragged plane groups."""
import numpy as np
import pytest

from workloads import cylinder_case
from helpers import run_oracle

pytestmark = pytest.mark.gpu

COLUMNS = ["col_z4_g4", "col_z4_g8", "col_z3_g4", "col_z2_g8", "col_z2_g12_p16"]


def _body(nv, adaptive=False):
    c = cylinder_case(Ma=2.0, Kn=0.02 if adaptive else 0.1, n_r=8, n_theta=10, nv=nv, adaptive=adaptive, Kn_ref=0.02,
                      macro_steps=10, presolve_max_blocks=3, vbox=((-10, 10), (-9, 9), (-8, 8)))
    c.tol, c.dt, c.adapt_every = 0.0, 0.5, 1000
    return c


def _reduced(nv):
    c = cylinder_case(Ma=2.0, Kn=0.1, n_r=6, n_theta=8, nv=nv, vbox=((-10, 10), (-9, 9), (0, 1)), adaptive=False,
                      macro_steps=10, relax=1.0, reduced=True)
    c.dt = 0.5
    return c


CASES = {"whole": lambda: _body((14, 12, 6)), "ragged": lambda: _body((13, 11, 7)),
         "interfaces": lambda: _body((13, 11, 7), adaptive=True), "reduced": lambda: _reduced((13, 11, 2))}


@pytest.mark.parametrize("name", list(CASES))
def test_fp64_columns_give_the_bits_of_the_general_sweep(name):
    from paper_2501_02245_gb300 import Solver
    case = CASES[name]()
    flags = run_oracle(case, 0)[0].dvm.copy() if case.adaptive else None
    n = case.mesh.ncell if flags is None else int(flags.sum())
    ref = None
    for tile in ["g4_v1_c1"] + COLUMNS:
        s = Solver.from_case(case, forced_flags=flags)
        s.set_sweep_tile(tile)
        s.iterate(3)
        out = (s.W(), s.vdf(n)[1])
        s.close()
        ref = ref or out
        assert np.array_equal(out[0], ref[0]) and np.array_equal(out[1], ref[1]), tile
