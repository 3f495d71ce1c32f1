"""The work that users of this library have it do, as cases to be measured.

A case is a dict of plain values; `prepare` makes what a program holds before
the call, `run` is one pass through the public entry points, `work` the bytes
and flops that the pass cannot do without, and `exact` what `run` returns, in
64 bits and plain torch (None where that takes more than about 20 seconds).

Kinds of case ("op"):
  maxwellian         rows of conservation-corrected Maxwellians into the caller's
                     buffer (gsis_corrected_maxwellian_noalloc)
  two_vdf_reference  reference pairs (g0, g1) of the nitrogen model for given
                     states, on the device (gsis_two_vdf_reference)
  two_vdf_moments    moments of given pairs (gsis_two_vdf_moments)
  shock              GSIS iterations of one 1D normal shock, all cells kinetic
  batch              GSIS iterations of many uneven shocks together
  cylinder, sphere   GSIS iterations of an adaptive (or all-kinetic) blunt body
                     in mid-run: presolved, re-identified, tile shape chosen
An iteration case runs `steps` GSIS iterations and reads the fields that a
program watches: the macroscopic state, the high-order terms and, with walls,
the wall loads; a small shock reads its distribution as well.  Fields of a run
whose VDF is stored in 32 (16) bits come back in 32 (16) bits.

The seed moves the physical conditions by a percent or so (Mach number, wall
temperature, thickness of the initial profile, given states), as a sweep over
conditions does; sizes are the case's own.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2501_02245_gb300 import gsis, Solver
from workloads import (batch_vgrid_half_width, cylinder_case, shock_1d_case, shock_batch_cases, sphere_case)

GAMMA = 5.0 / 3.0
OMEGA = 0.81                 # viscosity index of the monatomic workloads
# nitrogen: internal degrees of freedom, collision number, relaxation rates A_tt, A_tr, A_rt, A_rr
D_R, Z_R, A_N2 = 2, 2.667, (0.786, -0.201, -0.059, 0.842)
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}
FIELD_TYPE = {"f64": np.float64, "f32": np.float32, "bf16": np.float16, "f16": np.float16}
W_FIELDS = ["rho", "ux", "uy", "uz", "T"]
HOT_FIELDS = ["hot_sxx", "hot_syy", "hot_szz", "hot_sxy", "hot_sxz", "hot_syz", "hot_qx", "hot_qy", "hot_qz"]
WALL_FIELDS = ["wall_q", "wall_p", "wall_tx", "wall_ty", "wall_tz"]
EXACT_POINTS = 4.0e7         # points x iterations that exact() gets through in about 20 s


# ---------------------------------------------------------------------------- the cases
def listed():
    return [
        # one state on the smallest velocity grid of the shock batch: a boundary condition or a probe
        # cell evaluated in a latency-critical loop; launches and their latency are all of it
        {"name": "maxwellian_one", "op": "maxwellian", "states": 1, "nx": 24, "ny": 24, "nz": 24},
        # the most states a call takes, on the cylinder's velocity grid: seeding a block of cells
        {"name": "maxwellian_rows", "op": "maxwellian", "states": 256, "nx": 48, "ny": 48, "nz": 24},
        # reference pairs of the nitrogen model for a block of cells
        {"name": "two_vdf_reference", "op": "two_vdf_reference", "states": 96, "nx": 48, "ny": 48, "nz": 24},
        # and the moments of as many pairs
        {"name": "two_vdf_moments", "op": "two_vdf_moments", "states": 96, "nx": 48, "ny": 48, "nz": 24},
        # the smallest solve: few cells, a ragged velocity grid, the distribution read back
        {"name": "shock_small", "op": "shock", "cells": 30, "nx": 20, "ny": 10, "nz": 9, "mach": 2.0,
         "half_width": 7.5, "vmax": 8.0, "macro_steps": 30, "dtype": "f64", "steps": 2, "vdf": True},
        # the 1D normal shock of the benchmark, the plain FP64 form
        {"name": "shock", "op": "shock", "cells": 200, "nx": 48, "ny": 24, "nz": 24, "mach": 2.0,
         "half_width": 25.0, "vmax": 6.0 * math.sqrt(2.0), "macro_steps": 50, "dtype": "f64", "steps": 2,
         "vdf": False},
        # the 64 uneven shocks (100 to 800 cells, 24^3 to 64^3 velocities, FP32 and BF16) as one batch
        {"name": "batch", "op": "batch", "solves": 64, "plan": 2501, "macro_steps": 50, "steps": 4},
        # the benchmark's cylinder in each storage type: the plain FP64 form, FP32, BF16
        {"name": "cylinder_f64", "op": "cylinder", "n_r": 128, "n_theta": 128, "nx": 48, "ny": 48, "nz": 24,
         "reduced": False, "adaptive": True, "share": 0.64, "mach": 5.0, "dtype": "f64", "presolve": 100, "steps": 2},
        {"name": "cylinder_f32", "op": "cylinder", "n_r": 128, "n_theta": 128, "nx": 48, "ny": 48, "nz": 24,
         "reduced": False, "adaptive": True, "share": 0.64, "mach": 5.0, "dtype": "f32", "presolve": 100, "steps": 4},
        {"name": "cylinder_bf16", "op": "cylinder", "n_r": 128, "n_theta": 128, "nx": 48, "ny": 48, "nz": 24,
         "reduced": False, "adaptive": True, "share": 0.64, "mach": 5.0, "dtype": "bf16", "presolve": 100, "steps": 4},
        # the same flow with the two reduced distributions of a 2D flow
        {"name": "cylinder_reduced", "op": "cylinder", "n_r": 128, "n_theta": 128, "nx": 48, "ny": 48, "nz": 2,
         "reduced": True, "adaptive": True, "share": 0.64, "mach": 5.0, "dtype": "f64", "presolve": 100, "steps": 4},
        # a 3D body: three flux directions, BF16, the sphere's velocity grid on a coarser mesh
        {"name": "sphere_bf16", "op": "sphere", "n_r": 32, "n_pol": 24, "n_az": 24, "nx": 48, "ny": 48, "nz": 48,
         "adaptive": True, "share": 0.64, "mach": 5.0, "dtype": "bf16", "presolve": 20, "steps": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["maxwellian", "two_vdf_reference", "two_vdf_moments", "shock", "shock", "batch",
                     "cylinder", "cylinder", "cylinder", "sphere"])
    dtype = rng.choice(["f64", "f32", "bf16", "f16"])
    if op == "maxwellian":
        return {"op": op, "states": _log(rng, 1, 256), "nx": rng.randint(17, 49), "ny": rng.randint(10, 48),
                "nz": rng.randint(9, 48)}
    if op in ("two_vdf_reference", "two_vdf_moments"):
        return {"op": op, "states": _log(rng, 2, 128), "nx": rng.randint(17, 48), "ny": rng.randint(12, 48),
                "nz": rng.randint(10, 32)}
    if op == "shock":
        mach = round(rng.uniform(1.5, 4.0), 2)
        cells = _log(rng, 30, 400)
        n = rng.randint(20, 48)
        return {"op": op, "cells": cells, "nx": n, "ny": rng.randint(10, n), "nz": rng.randint(9, n), "mach": mach,
                "half_width": cells / 8.0, "vmax": float(batch_vgrid_half_width(mach)),
                "macro_steps": rng.choice([30, 50]), "dtype": dtype, "steps": 2, "vdf": False}
    if op == "batch":
        return {"op": op, "solves": _log(rng, 3, 40), "plan": rng.randint(1, 9999), "macro_steps": 50, "steps": 2}
    if op == "cylinder":
        reduced = rng.random() < 0.25
        return {"op": op, "n_r": rng.randint(64, 128), "n_theta": rng.randint(64, 128), "nx": rng.randint(36, 48),
                "ny": rng.randint(36, 48), "nz": 2 if reduced else rng.randint(16, 24), "reduced": reduced,
                "adaptive": rng.random() < 0.75, "share": 0.64, "mach": round(rng.uniform(4.0, 5.0), 2),
                "dtype": dtype, "presolve": 100, "steps": 2}
    return {"op": op, "n_r": rng.randint(24, 40), "n_pol": rng.randint(16, 24), "n_az": rng.randint(16, 24),
            "nx": rng.randint(36, 48), "ny": rng.randint(36, 48), "nz": rng.randint(36, 48), "adaptive": True,
            "share": 0.64, "mach": round(rng.uniform(4.0, 5.0), 2), "dtype": rng.choice(["f32", "bf16", "f16"]),
            "presolve": 20, "steps": 2}


# ---------------------------------------------------------------------------- inputs
def _rng(seed):
    return np.random.default_rng(seed)


def _grid(case):
    """Velocity grid of the cases that take states: n nodes per axis on [-8, 8]."""
    vg = gsis.VGridDesc()
    for d, k in enumerate(("nx", "ny", "nz")):
        vg.n[d], vg.lo[d], vg.hi[d] = case[k], -8.0, 8.0
    return vg


def _states(case, seed):
    """(rho, u, T) of gas cells around a body: [states, 5]."""
    r, n = _rng(seed), case["states"]
    u = np.concatenate([r.uniform(0.0, 2.5, (n, 1)), r.uniform(-0.5, 0.5, (n, 2))], axis=1)
    return np.concatenate([r.uniform(0.5, 3.0, (n, 1)), u, r.uniform(0.8, 2.2, (n, 1))], axis=1)


def _two_vdf_states(case, seed):
    """rho, u, T_t, T_r, q_t, q_r out of equilibrium: [states, 12]."""
    r, n = _rng(seed), case["states"]
    return np.concatenate([r.uniform(0.5, 2.5, (n, 1)), r.uniform(-1.0, 1.0, (n, 3)), r.uniform(0.8, 2.0, (n, 2)),
                           r.uniform(-0.1, 0.1, (n, 6))], axis=1)


def _nodes(case, device="cpu"):
    """Node values of the three axes on [-8, 8], as broadcastable [nz, ny, nx] axes."""
    ax = [(-8.0 + (torch.arange(case[k], dtype=torch.float64, device=device) + 0.5) * (16.0 / case[k]))
          for k in ("nx", "ny", "nz")]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _pairs(case, seed, device):
    """Distribution pairs of states out of equilibrium: two drifting Maxwellians
    with a skewed internal-energy part, [states, 2, Nv]."""
    S = _two_vdf_states(case, seed)
    x, y, z = _nodes(case, device)
    F = torch.empty((S.shape[0], 2, case["nx"] * case["ny"] * case["nz"]), dtype=torch.float64, device=device)
    for k, s in enumerate(S.tolist()):
        rho, ux, uy, uz, Tt, Tr, qx, qy = s[:8]

        def maxwellian(n, a, b, c, T):
            return n * (2.0 * math.pi * T) ** -1.5 * (torch.exp((x - a) ** 2 * (-0.5 / T)) *
                                                      torch.exp((y - b) ** 2 * (-0.5 / T)) *
                                                      torch.exp((z - c) ** 2 * (-0.5 / T)))
        f0 = maxwellian(rho, ux, uy, uz, Tt) + maxwellian(0.2 * rho, ux + 1.0 + qx, uy + qy, uz, 0.7 * Tt)
        F[k, 0] = f0.reshape(-1)
        F[k, 1] = (0.5 * D_R * Tr * f0 * (1.0 + 0.1 * torch.sin(x - ux))).reshape(-1)
    return F


def _shock(case, seed):
    r = _rng(seed)
    return shock_1d_case(Ma=case["mach"] * (1.0 + 0.01 * r.uniform(-1.0, 1.0)), n_cells=case["cells"],
                         half_width=case["half_width"], nv=(case["nx"], case["ny"], case["nz"]), vmax=case["vmax"],
                         delta=r.uniform(1.5, 2.5), macro_steps=case["macro_steps"])


def _batch(case, seed):
    """The uneven shocks of a plan; the seed moves the thickness of their initial profiles."""
    r = _rng(seed)
    out = []
    for c in shock_batch_cases(n=case["solves"], seed=case["plan"], macro_steps=case["macro_steps"]):
        d = shock_1d_case(Ma=c.extra["Ma"], n_cells=c.mesh.ni, half_width=c.mesh.ni / 8.0, nv=c.vgrid.n,
                          vmax=c.vgrid.hi[0], delta=r.uniform(1.5, 2.5), macro_steps=case["macro_steps"])
        out.append((d, c.extra["vdf_dtype"]))
    return out


def _body(case, seed):
    """A blunt body at the seed's conditions.  The region is re-identified in
    the second iteration, so that a pass is one of the many that follow."""
    r = _rng(seed)
    mach, wall = case["mach"] * (1.0 + 0.01 * r.uniform(-1.0, 1.0)), 2.0 * (1.0 + 0.05 * r.uniform(-1.0, 1.0))
    nv = (case["nx"], case["ny"], case["nz"])
    if case["op"] == "cylinder":
        c = cylinder_case(Ma=mach, wall_T=wall, n_r=case["n_r"], n_theta=case["n_theta"], nv=nv,
                          adaptive=case["adaptive"], presolve_max_blocks=case["presolve"], reduced=case["reduced"])
    else:
        c = sphere_case(Ma=mach, wall_T=wall, n_r=case["n_r"], n_pol=case["n_pol"], n_az=case["n_az"], nv=nv,
                        adaptive=case["adaptive"], presolve_max_blocks=case["presolve"])
    c.adapt_every, c.tol = 1, 0.0
    return c


# ---------------------------------------------------------------------------- prepare, run
def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def prepare(case, seed):
    op = case["op"]
    if op == "maxwellian":
        n = case["states"]
        return {"op": op, "lib": gsis.load(), "grid": _grid(case), "n": n,
                "W": torch.from_numpy(_states(case, seed)).cuda(),
                "out": torch.empty((n, case["nx"] * case["ny"] * case["nz"]), dtype=torch.float64, device="cuda")}
    if op in ("two_vdf_reference", "two_vdf_moments"):
        # the context whose velocity grid the calls use
        c = shock_1d_case(n_cells=8, half_width=4.0, nv=(case["nx"], case["ny"], case["nz"]), vmax=8.0)
        s = {"op": op, "solver": Solver.from_case(c), "n": case["states"], "A": (ctypes.c_double * 4)(*A_N2)}
        if op == "two_vdf_reference":
            s["S"] = torch.from_numpy(_two_vdf_states(case, seed)).cuda()
            s["out"] = torch.empty((case["states"], 2, s["solver"].nv), dtype=torch.float64, device="cuda")
        else:
            s["F"] = _pairs(case, seed, "cuda")
            s["out"] = torch.empty((case["states"], 18), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()   # the library works on its own stream
        return s
    if op == "shock":
        c = _shock(case, seed)
        s = Solver.from_case(c, vdf_dtype=case["dtype"], tol=0.0)
        s.iterate(0)
        return {"op": op, "solver": s, "steps": case["steps"], "type": FIELD_TYPE[case["dtype"]],
                "vdf": case["cells"] if case["vdf"] else 0, "fields": W_FIELDS + HOT_FIELDS}
    if op == "batch":
        solvers = [Solver.from_case(c, vdf_dtype=t, tol=0.0) for c, t in _batch(case, seed)]
        gsis.iterate_batch(solvers, 1)   # starts the solves and records the graph
        return {"op": op, "solvers": solvers, "steps": case["steps"]}
    s = Solver.from_case(_body(case, seed), vdf_dtype=case["dtype"])
    s.iterate(2)
    return {"op": op, "solver": s, "steps": case["steps"], "type": FIELD_TYPE[case["dtype"]], "vdf": 0,
            "fields": W_FIELDS + HOT_FIELDS + WALL_FIELDS}


def _check(status, solver=None):
    if status != gsis.GSIS_OK:
        raise gsis.GsisError(status, "" if solver is None else solver.lib.gsis_last_error(solver.ctx).decode())


def _fields(solver, names, to):
    m = solver.moments(names)
    out = {"W": np.stack([m[k] for k in W_FIELDS], axis=1).astype(to),
           "hot": np.stack([m[k] for k in HOT_FIELDS], axis=1).astype(to)}
    if "wall_q" in m:
        out["wall"] = np.stack([m[k] for k in WALL_FIELDS], axis=1).astype(to)
    return out


def run(state):
    op = state["op"]
    if op == "maxwellian":
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        _check(state["lib"].gsis_corrected_maxwellian_noalloc(_ptr(state["W"]), state["n"],
                                                              ctypes.byref(state["grid"]), _ptr(state["out"]), stream))
        return state["out"]
    if op == "two_vdf_reference":
        s = state["solver"]
        _check(s.lib.gsis_two_vdf_reference(s.ctx, _ptr(state["S"]), state["n"], D_R, Z_R, state["A"],
                                            _ptr(state["out"])), s)
        return state["out"]
    if op == "two_vdf_moments":
        s = state["solver"]
        _check(s.lib.gsis_two_vdf_moments(s.ctx, _ptr(state["F"]), state["n"], D_R, _ptr(state["out"])), s)
        return state["out"]
    if op == "batch":
        gsis.iterate_batch(state["solvers"], state["steps"])
        f = [_fields(s, W_FIELDS + HOT_FIELDS, FIELD_TYPE[s.vdf_dtype]) for s in state["solvers"]]
        by = {}   # one array per storage type
        for s, m in zip(state["solvers"], f):
            for k, v in m.items():
                by.setdefault("%s_%s" % (k, s.vdf_dtype), []).append(v)
        return {k: np.concatenate(v) for k, v in by.items()}
    s = state["solver"]
    s.iterate(state["steps"])
    out = _fields(s, state["fields"], state["type"])
    if state["vdf"]:
        cells, f = s.vdf(state["vdf"])
        out["cells"], out["vdf"] = cells, f.astype(state["type"])
    return out


def work(case):
    op = case["op"]
    if op == "batch":
        points = [(c.mesh.ni * c.vgrid.nv, t) for c, t in _batch(case, 0)]
        # per point and iteration: VDF read and written once; 37 flops of the 1D update, 7 of the moments, 8 of Eq. updatef
        return {"bytes": case["steps"] * sum(2 * BYTES[t] * p for p, t in points),
                "flops": case["steps"] * 52.0 * sum(p for p, _ in points)}
    nv = case["nx"] * case["ny"] * case["nz"]
    if op == "maxwellian":   # a separable Gaussian times a polynomial of one value per axis
        return {"bytes": case["states"] * (8.0 * nv + 40.0), "flops": 6.0 * case["states"] * nv}
    if op == "two_vdf_reference":
        return {"bytes": case["states"] * (16.0 * nv + 96.0), "flops": 30.0 * case["states"] * nv}
    if op == "two_vdf_moments":
        return {"bytes": case["states"] * (16.0 * nv + 144.0), "flops": 14.0 * case["states"] * nv}
    cells = {"shock": lambda: case["cells"], "cylinder": lambda: case["n_r"] * case["n_theta"],
             "sphere": lambda: case["n_r"] * case["n_pol"] * case["n_az"]}[op]()
    if op != "shock" and case["adaptive"]:   # the criterion picks about this share of the cells
        cells *= case["share"]
    # 37 (1D), 67 (2D) or 97 (3D) flops of the update, 7 of the moments, 8 of Eq. updatef
    flops = {"shock": 52.0, "cylinder": 82.0, "sphere": 112.0}[op]
    return {"bytes": case["steps"] * 2.0 * BYTES[case["dtype"]] * cells * nv, "flops": case["steps"] * flops * cells * nv}


# ---------------------------------------------------------------------------- exact
class _Grid:
    """Midpoint grid on a box, flattened with x fastest; discrete sums over it."""

    def __init__(self, n, lo, hi):
        h = [(b - a) / k for k, a, b in zip(n, lo, hi)]
        ax = [a + (torch.arange(k, dtype=torch.float64) + 0.5) * d for k, a, d in zip(n, lo, h)]
        z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
        self.xi = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)])   # [3, Nv]
        self.w = h[0] * h[1] * h[2]
        self.psi = torch.cat([torch.ones_like(self.xi[:1]), self.xi, 0.5 * (self.xi ** 2).sum(0, keepdim=True)])

    def corrected(self, rho, u, T, q=None):
        """Shakhov form with heat flux q (a Maxwellian without) of one state,
        corrected with the Maxwellian-weighted multipliers to its discrete
        conserved moments."""
        c = self.xi - u[:, None]
        c2 = (c * c).sum(0)
        M = rho * (2.0 * math.pi * T) ** -1.5 * torch.exp(-c2 / (2.0 * T))
        D = M
        if q is not None:
            D = M * (1.0 + (q[:, None] * c).sum(0) * (c2 - 5.0 * T) / (15.0 * rho * T ** 3))
        U = torch.cat([torch.tensor([1.0], dtype=torch.float64), u, torch.stack([1.5 * T + 0.5 * (u * u).sum()])]) * rho
        # weighting polynomial (1, c, c^2) about u spans the same space as (1, xi, |xi|^2)
        phi = torch.cat([torch.ones_like(c2)[None], c, c2[None]])
        a = torch.linalg.solve(self.w * (self.psi * M) @ phi.T, U - self.w * self.psi @ D)
        return D + M * (a @ phi)


def _exact_two_vdf_reference(case, seed):
    g = _Grid((case["nx"], case["ny"], case["nz"]), (-8.0,) * 3, (8.0,) * 3)
    Att, Atr, Art, Arr = A_N2
    out = []
    for s in torch.from_numpy(_two_vdf_states(case, seed)):
        rho, u, Tt, Tr, qt, qr = s[0], s[1:4], s[4], s[5], s[6:9], s[9:12]
        T = (3.0 * Tt + D_R * Tr) / (3.0 + D_R)
        q0 = ((2.0 - 3.0 * Att) * Z_R + 1.0) * qt - 3.0 * Atr * Z_R * qr
        q1 = -Art * Z_R * qt + (1.0 - Arr * Z_R) * qr
        c = g.xi - u[:, None]
        g0t, g0r = g.corrected(rho, u, Tt, qt), g.corrected(rho, u, T, q0)
        Mt, Mr = g.corrected(rho, u, Tt), g.corrected(rho, u, T)
        g1t = 0.5 * D_R * Tr * g0t + Mt * (qr[:, None] * c).sum(0) / (rho * Tt)
        g1r = 0.5 * D_R * T * g0r + Mr * (q1[:, None] * c).sum(0) / (rho * T)
        b = 1.0 / Z_R
        out.append(torch.stack([(1.0 - b) * g0t + b * g0r, (1.0 - b) * g1t + b * g1r]))
    return torch.stack(out)


def _exact_two_vdf_moments(case, seed):
    g = _Grid((case["nx"], case["ny"], case["nz"]), (-8.0,) * 3, (8.0,) * 3)
    out = []
    for f0, f1 in _pairs(case, seed, "cpu"):
        rho = g.w * f0.sum()
        u = g.w * g.xi @ f0 / rho
        c = g.xi - u[:, None]
        c2 = (c * c).sum(0)
        P = g.w * (c * f0) @ c.T
        tr = P.trace()
        out.append(torch.cat([rho[None], u, (tr / (3.0 * rho))[None], (2.0 * g.w * f1.sum() / (D_R * rho))[None],
                              P.diagonal() - tr / 3.0, torch.stack([P[0, 1], P[0, 2], P[1, 2]]),
                              0.5 * g.w * c @ (c2 * f0), g.w * c @ f1]))
    return torch.stack(out)


def _half_minmod(a, b):
    return torch.where(a * b > 0.0, 0.5 * torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))


class _Shock:
    """One GSIS solve of a 1D shock, all cells kinetic, in plain torch.  Cells of
    size dx between two far-field states; unit cross-section."""

    def __init__(self, c):
        self.grid = _Grid(c.vgrid.n, c.vgrid.lo, c.vgrid.hi)
        self.W = torch.from_numpy(np.array(c.W0))
        self.n = self.W.shape[0]
        self.ends = [torch.from_numpy(np.array(c.mesh.bc_state[s])) for s in (0, 1)]
        x = c.mesh.centers[0, 0, :, 0]
        self.dx = float(x[1] - x[0])
        self.mu0 = c.Kn / math.sqrt(math.pi / 2.0)
        self.steps, self.cfl, self.k_sub, self.dt = c.macro_steps, c.cfl, c.k_sub, c.dt
        self.far = [self.maxwellian(w) for w in self.ends]
        self.f = torch.stack([self.maxwellian(w) for w in self.W])

    def maxwellian(self, w):
        return self.grid.corrected(w[0], w[1:4], w[4])

    def mu(self, T):
        return self.mu0 * T ** OMEGA

    # -- kinetic step
    def sweep(self):
        g, f, n = self.grid, self.f, self.n
        xn = g.xi[0] / self.dx
        src, it = [], []
        for k in range(n):
            w = self.W[k]
            c = g.xi - w[1:4, None]
            q = 0.5 * g.w * c @ ((c * c).sum(0) * f[k])
            it.append(w[0] * w[4] / self.mu(w[4]))
            src.append(g.corrected(w[0], w[1:4], w[4], q) * it[k])
        out_l, out_h = (-xn).clamp(min=0.0), xn.clamp(min=0.0)
        zero = torch.zeros_like(xn)
        for order in (range(n - 1, -1, -1), range(n)):
            for k in order:
                c0 = f[k]
                dl = c0 - f[k - 1] if k > 0 else zero
                dh = f[k + 1] - c0 if k < n - 1 else zero
                own = _half_minmod(dl, dh)
                f_l = f[k - 1] + (_half_minmod(f[k - 1] - f[k - 2], dl) if k > 1 else zero) if k > 0 else self.far[0]
                f_h = (f[k + 1] - (_half_minmod(dh, f[k + 2] - f[k + 1]) if k < n - 2 else zero) if k < n - 1
                       else self.far[1])
                num = src[k] + xn * torch.where(xn < 0.0, -own, f_l) - xn * torch.where(xn > 0.0, own, f_h)
                f[k] = num / (it[k] + out_l + out_h)

    # -- moments of f about the current velocity: state, stress and heat flux
    def half_state(self):
        g = self.grid
        W, sig, q = torch.empty_like(self.W), [], []
        for k in range(self.n):
            f = self.f[k]
            rho = g.w * f.sum()
            u = self.W[k, 1:4] + g.w * (g.xi - self.W[k, 1:4, None]) @ f / rho
            c = g.xi - u[:, None]
            P = g.w * (c * f) @ c.T
            p = P.trace() / 3.0
            W[k] = torch.cat([rho[None], u, (p / rho)[None]])
            sig.append(torch.cat([P.diagonal() - p, torch.stack([P[0, 1], P[0, 2], P[1, 2]])]))
            q.append(0.5 * g.w * c @ ((c * c).sum(0) * f))
        return W, torch.cat([torch.stack(sig), torch.stack(q)], dim=1)

    def nsf(self, W):
        """Navier-Stokes-Fourier stress and heat flux from least-squares gradients."""
        v = W[:, 1:5]
        d, num, den = self.dx, torch.zeros_like(v), torch.zeros(self.n, 1, dtype=torch.float64)
        num[1:] += d * (v[1:] - v[:-1])
        num[:-1] += d * (v[1:] - v[:-1])
        den[1:] += d * d
        den[:-1] += d * d
        num[0] += 0.5 * d * (v[0] - self.ends[0][1:5])
        num[-1] += 0.5 * d * (self.ends[1][1:5] - v[-1])
        den[0] += 0.25 * d * d
        den[-1] += 0.25 * d * d
        return self.stress(self.mu(W[:, 4]), num / den)

    @staticmethod
    def stress(mu, grad):
        """(sigma xx, yy, zz, xy, xz, yz; q) for gradients d(u, T)/dx."""
        o = torch.zeros(grad.shape[0], 9, dtype=torch.float64)
        o[:, 0], o[:, 1], o[:, 2] = -4.0 / 3.0 * mu * grad[:, 0], 2.0 / 3.0 * mu * grad[:, 0], 2.0 / 3.0 * mu * grad[:, 0]
        o[:, 3], o[:, 4], o[:, 6] = -mu * grad[:, 1], -mu * grad[:, 2], -3.75 * mu * grad[:, 3]
        return o

    # -- synthetic solve
    @staticmethod
    def cons(W):
        rho, u, T = W[:, :1], W[:, 1:4], W[:, 4:]
        return torch.cat([rho, rho * u, rho * (1.5 * T + 0.5 * (u * u).sum(1, keepdim=True))], dim=1)

    @staticmethod
    def prim(U):
        u = U[:, 1:4] / U[:, :1]
        return torch.cat([U[:, :1], u, (2.0 * U[:, 4:] / U[:, :1] - (u * u).sum(1, keepdim=True)) / 3.0], dim=1)

    @staticmethod
    def euler(U):
        u = U[:, 1] / U[:, 0]
        p = (GAMMA - 1.0) * (U[:, 4] - 0.5 * (U[:, 1:4] ** 2).sum(1) / U[:, 0])
        F = U * u[:, None]
        F[:, 1] += p
        F[:, 4] += p * u
        return F

    @staticmethod
    def half_range(q, sign):
        """Flux through x of the molecules of (rho, u, p) that move along sign."""
        rho, un, T = q[:, 0], q[:, 1], q[:, 4] / q[:, 0]
        s = un / T.sqrt()
        P = 0.5 * (1.0 + sign * torch.special.erf(s * math.sqrt(0.5)))
        D = sign * T.sqrt() * torch.exp(-0.5 * s * s) / math.sqrt(2.0 * math.pi)
        m0 = un * P + D
        m1 = (un * un + T) * P + un * D
        m2 = (un ** 3 + 3.0 * un * T) * P + (un * un + 2.0 * T) * D
        ut2 = q[:, 2] ** 2 + q[:, 3] ** 2
        return torch.stack([rho * m0, rho * m1, rho * m0 * q[:, 2], rho * m0 * q[:, 3],
                            0.5 * rho * (m2 + (ut2 + 2.0 * T) * m0)], dim=1)

    def fluxes(self, W, hot):
        """Fluxes through the n + 1 faces along +x and lambda of each."""
        q = torch.cat([W[:, :4], (W[:, 0] * W[:, 4])[:, None]], dim=1)
        slope = torch.zeros_like(q)
        slope[1:-1] = _half_minmod(q[1:-1] - q[:-2], q[2:] - q[1:-1])
        ends = [torch.cat([e[:4], (e[0] * e[4])[None]])[None] for e in self.ends]
        left = torch.cat([ends[0], (q + slope)[:-1], q[-1:]])
        right = torch.cat([q[:1], (q - slope)[1:], ends[1]])
        F = self.half_range(left, 1.0) + self.half_range(right, -1.0)
        S = torch.zeros(self.n + 1, 9, dtype=torch.float64)
        Tf = 0.5 * (W[1:, 4] + W[:-1, 4])
        S[1:-1] = self.stress(self.mu(Tf), (W[1:, 1:5] - W[:-1, 1:5]) / self.dx) + 0.5 * (hot[1:] + hot[:-1])
        S[0], S[-1] = hot[0], hot[-1]
        We = torch.cat([self.ends[0][None], W, self.ends[1][None]])
        uf = 0.5 * (We[1:, 1:4] + We[:-1, 1:4])
        t = S[:, [0, 3, 4]]
        F[:, 1:4] += t
        F[:, 4] += (t * uf).sum(1) + S[:, 6]
        a = (GAMMA * W[:, 4]).sqrt()
        lam = torch.empty(self.n + 1, dtype=torch.float64)
        lam[1:-1] = (uf[1:-1, 0].abs() + 0.5 * (a[1:] + a[:-1]) +
                     5.0 * self.mu(Tf) / (0.5 * (W[1:, 0] + W[:-1, 0]) * self.dx))
        for k in (0, -1):
            lam[k] = W[k, 1].abs() + a[k] + 5.0 * self.mu(W[k, 4]) / (W[k, 0] * self.dx)
        return F, lam

    def solve(self, Wh, hot):
        U, Un, W = self.cons(Wh), self.cons(self.W), Wh.clone()
        for _ in range(self.steps):
            F, lam = self.fluxes(W, hot)
            D = ((1.0 / self.cfl + 0.5) * (lam[1:] + lam[:-1]) + self.dx / self.dt)[:, None]
            R = F[:-1] - F[1:] - self.dx / self.dt * (U - Un)
            dU = R / D
            for _ in range(self.k_sub):
                dF, ld = self.euler(U + dU) - self.euler(U), lam[1:-1, None]
                acc = torch.zeros_like(U)
                acc[:-1] += dF[1:] - ld * dU[1:]
                acc[1:] -= dF[:-1] + ld * dU[:-1]
                dU = (R - 0.5 * acc) / D
            U = U + dU
            W = self.prim(U)
        return W

    def iterate(self):
        self.sweep()
        Wh, kinetic = self.half_state()
        self.hot = kinetic - self.nsf(Wh)
        self.W = self.solve(Wh, self.hot)
        for k in range(self.n):
            self.f[k] += self.maxwellian(self.W[k]) - self.maxwellian(Wh[k])


def exact(case, seed):
    op = case["op"]
    if op == "maxwellian":
        g = _Grid((case["nx"], case["ny"], case["nz"]), (-8.0,) * 3, (8.0,) * 3)
        return torch.stack([g.corrected(w[0], w[1:4], w[4]) for w in torch.from_numpy(_states(case, seed))])
    if op == "two_vdf_reference":
        return _exact_two_vdf_reference(case, seed)
    if op == "two_vdf_moments":
        return _exact_two_vdf_moments(case, seed)
    if op == "shock" and case["cells"] * case["nx"] * case["ny"] * case["nz"] * case["steps"] <= EXACT_POINTS:
        s = _Shock(_shock(case, seed))
        for _ in range(case["steps"]):
            s.iterate()
        out = {"W": s.W, "hot": s.hot}
        if case["vdf"]:
            out["cells"], out["vdf"] = None, s.f
        return out
    # the other flows (a batch, a body started from thousands of pseudo-steps of a presolve and an
    # adaptive region) take minutes in this form
    return None
