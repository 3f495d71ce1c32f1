"""The line sweep gives the bits of the general one, and a batch of lines the
bits of its members iterated alone: far field, walls, closed ends, uneven cells,
odd velocity axes, every storage type, a member of another dimension."""
import numpy as np
import pytest

from workloads import cylinder_case, shock_1d_case
from workloads.meshes import _hexa_block, _tensor_vertices, BC_FARFIELD, BC_WALL, BC_NONE

pytestmark = pytest.mark.gpu


def _shock(cells=37, nv=(20, 9, 7)):
    return shock_1d_case(Ma=3.0, n_cells=cells, half_width=cells / 6.0, nv=nv, vmax=12.0, macro_steps=20)


def _gas(bc, cells=9, nv=(12, 11, 7)):
    """A moving gas between two ends of the given types, cells of uneven size."""
    case = shock_1d_case(Ma=1.6, n_cells=cells, half_width=cells / 4.0, nv=nv, vmax=7.0, macro_steps=10)
    xs = np.linspace(0.0, 3.0, cells + 1) ** 1.3
    P = _tensor_vertices(xs, np.array([0.0, 1.0]), np.array([0.0, 1.0]))
    states = [[1.0, 0, 0, 0, 1.2] if b != BC_NONE else [0.0] * 5 for b in bc]
    case.mesh = _hexa_block(P, 1, list(bc) + [BC_NONE] * 4, states + [[0.0] * 5] * 4, "line")
    case.W0 = np.tile(np.array([1.0, 0.1, 0.05, -0.02, 1.0]), (cells, 1))
    return case


CASES = {"shock": _shock, "walls": lambda: _gas((BC_WALL, BC_WALL)), "closed": lambda: _gas((BC_NONE, BC_FARFIELD)),
         "one cell": lambda: _gas((BC_FARFIELD, BC_WALL), cells=1)}


def _state(s, n):
    return [s.W(), s.hot(), s.vdf(n)[1]]


@pytest.mark.parametrize("name", list(CASES))
def test_fp64_lines_give_the_bits_of_the_general_sweep(name):
    from paper_2501_02245_gb300 import Solver
    case = CASES[name]()
    out = []
    for tile in (None, "g4_v1_c1"):
        s = Solver.from_case(case)
        if tile:
            s.set_sweep_tile(tile)
        s.iterate(4)
        out.append(_state(s, case.mesh.ncell))
        s.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("tile", ["line_w4", "line1_w4", "vpt1_cb1_w4"])
def test_batch_tiles_of_lines_give_the_same_bits(tile):
    from paper_2501_02245_gb300 import Solver, iterate_batch, batch_info
    from paper_2501_02245_gb300.gsis import set_batch_tile
    members = [(CASES[n](), d) for n in ("shock", "walls", "closed") for d in ("f64", "f32")]
    set_batch_tile(tile)
    try:
        batch = [Solver.from_case(c, vdf_dtype=d) for c, d in members]
        iterate_batch(batch, 3)
        assert "tile=" + tile + " " in batch_info(batch)
    finally:
        set_batch_tile(None)
    for b, (c, d) in zip(batch, members):
        s = Solver.from_case(c, vdf_dtype=d)
        s.iterate(3)
        assert np.array_equal(b.W(), s.W()), (c.name, d)
        s.close()
        b.close()


def test_few_fp64_tiles_take_one_plane_and_mixed_lines_are_searched():
    from paper_2501_02245_gb300 import Solver, iterate_batch, batch_info
    few, many = _shock(), _shock(12, (48, 40, 20))   # 42 and 1,200 one-plane tiles
    for members, tile in (([(few, "f64")] * 2, "line1_w4 (default)"), ([(many, "f64")], "line_w4 (default)"),
                          ([(few, "f32")] * 2, "line_w4 (default)"), ([(few, "f64"), (few, "f32")], "(autotuned)")):
        batch = [Solver.from_case(c, vdf_dtype=d) for c, d in members]
        iterate_batch(batch, 1)
        assert tile in batch_info(batch)
        for b in batch:
            b.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_batches_give_the_bits_of_their_members_alone(mixed):
    """mixed: with a 2D member every line runs in the 3-direction kernels."""
    from paper_2501_02245_gb300 import Solver, iterate_batch
    members = [(_shock(), d) for d in ("f64", "f32", "bf16", "f16")] + [(_shock(130, (16, 8, 8)), "f32")]
    members += [(CASES["walls"](), "f64"), (CASES["walls"](), "f32")]
    if mixed:
        c = cylinder_case(Ma=2.0, Kn=0.1, n_r=8, n_theta=12, nv=(12, 10, 6), adaptive=False, macro_steps=10,
                          vbox=((-10, 10), (-9, 9), (-8, 8)), presolve_max_blocks=2)
        c.dt = 0.5
        members.append((c, "f64"))
    batch = [Solver.from_case(c, vdf_dtype=d) for c, d in members]
    iterate_batch(batch, 4)
    for b, (c, d) in zip(batch, members):
        s = Solver.from_case(c, vdf_dtype=d)
        s.iterate(4)
        W, W1 = b.W(), s.W()
        assert np.array_equal(W, W1), (c.name, d, np.abs(W - W1).max())
        s.close()
        b.close()
