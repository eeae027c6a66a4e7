"""Boundary conditions beside interior nodes whose pressure is zero, negative or
not finite, or whose density is negative: their Mach number is not defined or
infinite, and the boundary node takes the branch that a comparison with it
selects (no comparison with a NaN holds, which leaves the free stream at the far
field and the extrapolation at the exit), as in the oracle.  Finite results
within the 1e-14 of the other boundary test, and the same nodes not finite."""
import numpy as np
import pytest

from gpu_helpers import device_ctx, oracle_params

pytestmark = pytest.mark.gpu

SHAPE = (48, 24, 32)


@pytest.fixture(scope="module")
def lj():
    from paper_2301_00817_gb300 import _build
    _build.build()
    import paper_2301_00817_gb300 as lj
    lj.load_library()
    return lj


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


def _limits(flat, rng):
    """Every node of flat ([5][n], a copy is returned) replaced by one of the
    states: p < 0, rho < 0 (p > 0), p = 0 exactly at rest and moving either
    way, p infinite and NaN."""
    q = flat.copy()
    for n in range(q.shape[1]):
        u = 0.4 * rng.standard_normal(3)
        kind = rng.integers(0, 6)
        if kind == 0:
            q[:, n] = (1.1, *(1.1 * u), 0.55 * (u @ u) - 0.3)
        elif kind == 1:
            q[:, n] = (-0.9, *(-0.9 * u), -0.45 * (u @ u) + 1.5)
        elif kind == 2:
            q[:, n] = (1.0, 0.0, 0.0, 0.0, 0.0)
        elif kind == 3:
            q[:, n] = (1.0, 0.0, 0.0, 0.0, 0.125)
            q[1 + rng.integers(0, 3), n] = rng.choice([-0.5, 0.5])
        else:
            q[:, n] = (1.0, *u, np.inf if kind == 4 else np.nan)
    return q


@pytest.mark.parametrize("where", ["far_field", "exit", "entrance"])
def test_undefined_mach_numbers(orc, lj, torch, where):
    kw = dict(periodic=(0, 0, 1), bc=lj.BC_JET_CHAR if where == "entrance" else lj.BC_JET)
    xyz = lj.synth.jet_grid(*SHAPE)
    ctx, _ = device_ctx(lj, torch, SHAPE, xyz, **kw)
    P = oracle_params(orc, **kw)
    M = orc.metrics(xyz, (0, 0, 1))
    rng = np.random.default_rng(7)
    prim = lj.synth.uniform_prim(SHAPE)
    prim[1:4] = 0.3 * rng.standard_normal((3,) + SHAPE)
    Q = orc.prim_to_cons(P, prim)
    face = {"far_field": np.s_[:, 1:-2, -2], "exit": np.s_[:, -2, 2:-2], "entrance": np.s_[:, 1, 2:-2]}[where]
    Q[face] = _limits(Q[face].reshape(5, -1), rng).reshape(Q[face].shape)
    Qd = torch.from_numpy(Q).cuda()
    ctx.les_apply_bc(Qd, 0.0)
    got, want = Qd.cpu().numpy(), orc.bc_jet(P, Q, M, xyz, 0.0)
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    ok = np.isfinite(want)
    assert np.abs(got[ok] - want[ok]).max() <= 1e-14 * np.abs(want[ok]).max()
