"""Records of lines around the number from which four share a warp, whole and
ragged groups, against the FP64 oracle (1e-10 on the state and the VDF, as in the other
parity tests), and on the reduced grid."""
import pytest

from workloads import shock_1d_case
from workloads.cases import VGrid
from helpers import run_oracle, w_rel_err, rel_err, vdf_by_cell, RTOL_W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [152, 153, 304, 305, 307])
def test_line_records(cells):
    from paper_2501_02245_gb300 import Solver
    case = shock_1d_case(Ma=1.4, n_cells=cells, half_width=cells / 4.0, nv=(12, 10, 8), vmax=8.0, macro_steps=5)
    s = Solver.from_case(case)
    s.iterate(2)
    o, ho = run_oracle(case, 2)
    assert w_rel_err(s.W(), ho[-1]) < RTOL_W
    assert rel_err(vdf_by_cell(s, o.N, o.N, o.vg.nv), o.f) < 1e-10
    s.close()


@pytest.mark.parametrize("cells", [9, 307])
def test_line_records_on_the_reduced_grid(cells):
    from paper_2501_02245_gb300 import Solver
    case = shock_1d_case(Ma=1.4, n_cells=cells, half_width=cells / 4.0, nv=(12, 10, 2), vmax=8.0, macro_steps=5)
    case.vgrid = VGrid((12, 10, 2), (-8.0, -8.0, 0.0), (8.0, 8.0, 1.0), reduced=True)
    s = Solver.from_case(case)
    s.iterate(2)
    _, ho = run_oracle(case, 2)
    assert w_rel_err(s.W(), ho[-1]) < RTOL_W
    s.close()
