"""The window sweep of 1D lines against the FP64 oracle at the sizes where it
can go wrong: lines shorter than its ring, one cell, lengths around multiples
of the ring, odd velocity axes, fewer planes than a column, a velocity node at
rest, non-uniform cells, walls and closed ends, every storage type.
Tolerances are those of the other parity tests: FP64 1e-10 on the state and
the VDF; reduced storage the bounds of the precision tests."""
import numpy as np
import pytest

from workloads import shock_1d_case
from workloads.meshes import _hexa_block, _tensor_vertices, BC_FARFIELD, BC_WALL, BC_NONE
from helpers import run_oracle, w_rel_err, rel_err, vdf_by_cell, RTOL_W

pytestmark = pytest.mark.gpu

BOUND = {"f32": 2e-5, "bf16": 3.9e-3, "f16": 9.8e-4}


def _check(case, dtype="f64", n_iter=2, route="1D line"):
    from paper_2501_02245_gb300 import Solver, iterate_batch, batch_info
    o, ho = run_oracle(case, n_iter)
    single = Solver.from_case(case, vdf_dtype=dtype)
    single.iterate(n_iter)
    assert route in single.tuning_info()
    batch = [Solver.from_case(case, vdf_dtype=dtype), Solver.from_case(case, vdf_dtype=dtype)]
    iterate_batch(batch, n_iter)
    assert "tile=line" in batch_info(batch)
    for s in [single] + batch:
        W = s.W()
        if dtype == "f64":
            assert w_rel_err(W, ho[-1]) < RTOL_W, "%.3e" % w_rel_err(W, ho[-1])
            f = vdf_by_cell(s, o.N, o.N, o.vg.nv)
            assert rel_err(f, o.f) < 1e-10
        else:
            e = max(rel_err(W[:, 0], ho[-1][:, 0]), rel_err(W[:, 4], ho[-1][:, 4]))
            assert e < BOUND[dtype], "%.3e" % e
        s.close()


# cells, velocity grid
SIZES = [(5, (12, 10, 8)), (6, (13, 9, 7)), (7, (14, 8, 8)), (13, (17, 11, 9)), (30, (20, 10, 9))]


@pytest.mark.parametrize("cells,nv", SIZES)
def test_lines_fp64(cells, nv):
    _check(shock_1d_case(Ma=1.6, n_cells=cells, half_width=cells / 4.0, nv=nv, vmax=8.0, macro_steps=10))


# one plane per lane would give two warps a sub-partition, two planes not yet
# (the general sweep), and two planes two warps (the line again)
@pytest.mark.parametrize("nv,route", [((48, 47, 14), "1D or empty"), ((48, 47, 35), "1D line")])
def test_lines_fp64_by_the_number_of_tiles(nv, route):
    _check(shock_1d_case(Ma=1.6, n_cells=6, half_width=1.5, nv=nv, vmax=8.0, macro_steps=5), route=route)


@pytest.mark.parametrize("cells,nv", [(7, (13, 9, 7)), (30, (20, 10, 9))])
@pytest.mark.parametrize("dtype", list(BOUND))
def test_lines_reduced_storage(dtype, cells, nv):
    _check(shock_1d_case(Ma=1.6, n_cells=cells, half_width=cells / 4.0, nv=nv, vmax=8.0, macro_steps=10), dtype)


def _couette(bc, cells=9, nv=(13, 12, 10)):
    """A resting gas between two ends of the given types, cells of uneven size."""
    case = shock_1d_case(Ma=1.6, n_cells=cells, half_width=cells / 4.0, nv=nv, vmax=7.0, macro_steps=5)
    xs = np.linspace(0.0, 3.0, cells + 1) ** 1.3
    P = _tensor_vertices(xs, np.array([0.0, 1.0]), np.array([0.0, 1.0]))
    states = [[1.0, 0, 0, 0, 1.2] if b != BC_NONE else [0.0] * 5 for b in bc]
    case.mesh = _hexa_block(P, 1, list(bc) + [BC_NONE] * 4, states + [[0.0] * 5] * 4, "line")
    case.W0 = np.tile(np.array([1.0, 0.1, 0.05, -0.02, 1.0]), (cells, 1))
    return case


@pytest.mark.parametrize("bc", [(BC_WALL, BC_FARFIELD), (BC_FARFIELD, BC_WALL), (BC_WALL, BC_WALL),
                                (BC_NONE, BC_FARFIELD), (BC_FARFIELD, BC_NONE)])
def test_lines_with_walls_and_closed_ends(bc):
    _check(_couette(bc))


@pytest.mark.parametrize("dtype", list(BOUND))
@pytest.mark.parametrize("cells,nv", [(7, (16, 9, 7)), (30, (20, 10, 9)), (65, (24, 16, 13))])
def test_fp32_arithmetic_gives_the_bits_of_the_general_sweep(dtype, cells, nv):
    """(Compared where f >= 2^-100: the kernel halves the face speeds and doubles the
    sum, exact only while no product is an FP32 subnormal.)"""
    from paper_2501_02245_gb300 import Solver
    case = shock_1d_case(Ma=2.0, n_cells=cells, half_width=cells / 4.0, nv=nv, vmax=9.0, macro_steps=10)
    W = []
    for tile in (None, "g8_v1_c1"):
        s = Solver.from_case(case, vdf_dtype=dtype)
        if tile:
            s.set_sweep_tile(tile)
        s.iterate(3)
        W.append((s.W(), s.vdf(cells)[1]))
        s.close()
    assert np.array_equal(W[0][0], W[1][0])
    f, g = W[0][1], W[1][1]
    big = np.maximum(f, g) >= 2.0 ** -100
    assert big.any() and np.array_equal(f[big], g[big])
