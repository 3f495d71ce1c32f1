"""The row-factored kernels of the single calls -- two-VDF reference pair and
moments, allocation-free Maxwellians -- against the oracle at the sizes where
their row blocks, thread groups and clusters can go wrong: odd axes, rows
longer than a block, rows longer than the tabulated length, one state and
more states than the SMs hold clusters of.  Tolerances are those of the other
parity tests of these calls (1e-11 and 1e-10 of the largest value)."""
import ctypes

import numpy as np
import pytest

from workloads import shock_1d_case
from oracle import model as M
from oracle.rykov import RykovGrid, NITROGEN

pytestmark = pytest.mark.gpu

# velocity grid, number of states
SIZES = [((17, 11, 9), 1), ((13, 7, 6), 700), ((300, 6, 5), 3), ((1100, 5, 4), 2)]


def _states(n):
    r = np.random.default_rng(5)
    return np.concatenate([r.uniform(0.5, 2.5, (n, 1)), r.uniform(-1, 1, (n, 3)), r.uniform(1.6, 2.4, (n, 2)),
                           r.uniform(-0.1, 0.1, (n, 6))], axis=1)


def _solver(nv):
    from paper_2501_02245_gb300 import Solver
    return Solver.from_case(shock_1d_case(n_cells=8, half_width=4.0, nv=nv, vmax=8.0))


def _grid(nv):
    return RykovGrid(M.VelocityGrid(nv, (-8.0,) * 3, (8.0,) * 3), NITROGEN["d_r"])


@pytest.mark.parametrize("nv,n", SIZES)
def test_two_vdf_reference_and_moments(nv, n):
    S, s, vg = _states(n), _solver(nv), _grid(nv)
    g = s.two_vdf_reference(S, NITROGEN["d_r"], NITROGEN["Z_r"], NITROGEN["A"])
    F = g.copy()   # moments of the pairs with a second, drifting population added
    F[:, 0] += 0.3 * np.roll(g[:, 0], 1, axis=1)
    m = s.two_vdf_moments(F, NITROGEN["d_r"])
    s.close()
    for k in sorted({0, n // 2, n - 1}):
        st = S[k]
        r0, r1 = vg.split(vg.reference(st[0], st[1:4], st[4], st[5], st[6:9], st[9:12], NITROGEN["Z_r"],
                                       NITROGEN["A"]))
        scale = max(np.max(np.abs(r0)), np.max(np.abs(r1)))
        assert np.max(np.abs(g[k, 0] - r0)) < 1e-11 * scale
        assert np.max(np.abs(g[k, 1] - r1)) < 1e-11 * scale
        rho, u, Tt, Tr, sig, qt, qr = vg.moments(vg.join(F[k, 0], F[k, 1]))
        ref = np.concatenate([[rho], u, [Tt, Tr], sig[[0, 1, 2, 0, 0, 1], [0, 1, 2, 1, 2, 2]], qt, qr])
        assert np.max(np.abs(m[k] - ref)) < 1e-11 * max(1.0, np.max(np.abs(ref)))


@pytest.mark.parametrize("nv,n", [((17, 11, 9), 1), ((13, 7, 6), 256), ((300, 20, 16), 2), ((260, 6, 5), 5)])
def test_noalloc_rows(nv, n):
    import torch
    from paper_2501_02245_gb300 import gsis
    S = _states(n)[:, :5]
    W = torch.from_numpy(np.ascontiguousarray(S)).cuda()
    out = torch.full((n, int(np.prod(nv))), float("nan"), dtype=torch.float64, device="cuda")
    vg = gsis.VGridDesc()
    for d in range(3):
        vg.n[d], vg.lo[d], vg.hi[d] = nv[d], -8.0, 8.0
    st = gsis.load().gsis_corrected_maxwellian_noalloc(
        ctypes.c_void_p(W.data_ptr()), n, ctypes.byref(vg), ctypes.c_void_p(out.data_ptr()),
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == gsis.GSIS_OK
    got = out.cpu().numpy()
    base = _grid(nv).base
    for k in range(n):
        ref = base.corrected_maxwellian(S[k, 0], S[k, 1:4], S[k, 4])
        assert np.max(np.abs(got[k] - ref)) < 1e-10 * np.max(np.abs(ref))
