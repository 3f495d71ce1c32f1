"""Batches of one total size and different axes, one after the other in one
process: the autotuner's choice for an even nx must not serve an odd one (its
pair tiles need x-rows of whole pairs)."""
import pytest

from workloads import cylinder_case
from helpers import w_rel_err

pytestmark = pytest.mark.gpu

UNIT = {"f32": 2 ** -23, "bf16": 2 ** -8}


def _case(nv):
    c = cylinder_case(Ma=2.0, Kn=0.1, n_r=12, n_theta=16, nv=nv, adaptive=False, macro_steps=10,
                      vbox=((-10, 10), (-9, 9), (-8, 8)), presolve_max_blocks=2)
    c.dt = 0.5
    return c


def test_transposed_velocity_grids_are_tuned_apart():
    from paper_2501_02245_gb300 import Solver, iterate_batch, batch_info
    for nv in ((24, 21, 10), (21, 24, 10), (24, 21, 10)):
        batch = [Solver.from_case(_case(nv), vdf_dtype=d) for d in ("f32", "bf16")]
        iterate_batch(batch, 2)
        tile = batch_info(batch).split("tile=")[1].split()[0]
        assert nv[0] % 2 == 0 or not tile.startswith("pair"), tile
        for b, d in zip(batch, ("f32", "bf16")):
            s = Solver.from_case(_case(nv), vdf_dtype=d)
            s.iterate(2)
            assert w_rel_err(b.W(), s.W()) <= 4 * UNIT[d], (nv, d)
            s.close()
            b.close()
