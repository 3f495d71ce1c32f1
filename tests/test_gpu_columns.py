"""The velocity-column sweep of 2D meshes against the FP64 oracle at the sizes
where it can go wrong: odd axes (ragged position tiles and plane groups),
fewer planes than a column holds, walls, far field, the periodic seam,
interfaces to NS cells (Grad-13 records with stress terms), and the reduced
grid's two planes.  The tolerance is that of the other FP64 parity tests, 1e-10
on the macroscopic state and on the VDF."""
import pytest

from workloads import cylinder_case, shock_1d_case
from helpers import run_oracle, w_rel_err, rel_err, vdf_by_cell, RTOL_W

pytestmark = pytest.mark.gpu

SHAPES = ["col_z4_g4", "col_z4_g8", "col_z3_g4", "col_z2_g8", "col_z2_g12_p16"]
# (nx, ny, nz): whole and partial position tiles; odd axes with a ragged plane group
GRIDS = [(14, 12, 6), (13, 11, 7)]


def _case(nv, adaptive=False):
    c = cylinder_case(Ma=2.0, Kn=0.02 if adaptive else 0.1, n_r=8, n_theta=10, nv=nv, adaptive=adaptive, Kn_ref=0.02,
                      macro_steps=10, presolve_max_blocks=3, vbox=((-10, 10), (-9, 9), (-8, 8)))
    c.tol, c.dt, c.adapt_every = 0.0, 0.5, 1000
    return c


def _check(case, flags=None):
    from paper_2501_02245_gb300 import Solver
    o, ho = run_oracle(case, 2, flags=flags)
    for name in SHAPES:
        s = Solver.from_case(case, forced_flags=flags)
        s.set_sweep_tile(name)
        s.iterate(2)
        assert w_rel_err(s.W(), ho[-1]) < RTOL_W, "%s: %.3e" % (name, w_rel_err(s.W(), ho[-1]))
        f = vdf_by_cell(s, int(o.dvm.sum()), o.N, o.vg.nv)
        assert rel_err(f[o.dvm], o.f[o.dvm]) < 1e-10, name
        s.close()


@pytest.mark.parametrize("nv", GRIDS)
def test_columns_match_the_oracle(nv):
    _check(_case(nv))


def test_columns_at_ns_interfaces():
    case = _case(GRIDS[1], adaptive=True)
    flags = run_oracle(case, 0)[0].dvm.copy()
    assert 0 < flags.sum() < flags.size
    _check(case, flags=flags)


@pytest.mark.parametrize("nv", [(14, 12, 2), (13, 11, 2)])
def test_columns_on_the_reduced_grid(nv):
    """Two planes: columns of three and four are longer than the grid."""
    case = cylinder_case(Ma=2.0, Kn=0.1, n_r=6, n_theta=8, nv=nv, vbox=((-10, 10), (-9, 9), (0, 1)), adaptive=False,
                         macro_steps=10, relax=1.0, reduced=True)
    case.dt = 0.5
    _check(case)


def test_columns_need_fp64_and_a_2d_mesh():
    from paper_2501_02245_gb300 import Solver, GsisError
    for case, dtype in ((_case(GRIDS[0]), "f32"), (shock_1d_case(n_cells=8, half_width=4.0, nv=(8, 8, 8)), "f64")):
        s = Solver.from_case(case, vdf_dtype=dtype)
        with pytest.raises(GsisError):
            s.set_sweep_tile("col_z4_g4")
        s.close()
