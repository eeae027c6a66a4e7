"""The fused stage kernel on rows that its 16-byte staging cannot take: row
lengths that are no multiple of four, shorter than a tile, one over a tile,
and eta extents around the tiles' 8 and 16 rows, on the jet grid and on boxes that
are periodic or open in every direction.  The residual against the oracle's,
within the 2e-5 of each component's flux scale of the other mixed-form
tests; then every variant of the stage on one such jet, five steps within
1e-5 (relative L2) of the oracle's."""
import numpy as np
import pytest

from gpu_helpers import device_ctx, oracle_params, rel_l2

pytestmark = pytest.mark.gpu


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


JETS = [(6, 15, 31), (7, 16, 33), (6, 17, 34), (5, 18, 35), (9, 33, 63), (6, 32, 65), (6, 19, 28)]
BOXES = [((6, 17, 33), (1, 1, 1)), ((7, 18, 31), (0, 0, 0)), ((6, 16, 66), (0, 1, 0)),
         ((6, 15, 36), (1, 0, 0))]


@pytest.mark.parametrize("shape,per", [(s, None) for s in JETS] + BOXES)
def test_residual_on_odd_rows(orc, lj, torch, shape, per):
    if per is None:
        kw, shift = dict(periodic=(0, 0, 1), bc=1), None
        xyz = lj.synth.jet_grid(*shape)
    else:
        kw = dict(periodic=per, bc=0)
        xyz, shift = lj.synth.box_grid(shape, (1.0, 1.3, 0.8), wave=0.25)
    P = oracle_params(orc, sgs_model=1, Re=2000.0, **kw)
    M = orc.metrics(xyz, kw["periodic"], shift)
    if per is None:
        Q = orc.init_jet(P, xyz, seed=5, noise=2e-2)
    else:
        Q = orc.prim_to_cons(P, lj.synth.smooth_periodic_prim(xyz, (1.0, 1.3, 0.8), amp=0.2, seed=2))
    ctx, _ = device_ctx(lj, torch, shape, xyz, shift, sgs_model=1, Re=2000.0,
                        precision=lj.PREC_MIXED, **kw)
    Qd = torch.from_numpy(Q).cuda()
    R = torch.empty_like(Qd)
    ctx.les_rhs(Qd, R)
    Rg, Ro = R.cpu().numpy(), orc.rhs(P, Q, M)
    fscale = (np.abs(M[9]) * np.sqrt(M[0] ** 2 + M[1] ** 2 + M[2] ** 2)).max()
    for c in range(5):
        qs = np.abs(Q[c]).max() + (np.abs(Q[4]).max() if c in (1, 2, 3, 4) else 0.0)
        assert np.abs(Rg[c] - Ro[c]).max() <= 2e-5 * fscale * qs, c


@pytest.mark.parametrize("option", ["plain", "local", "axis", "dynamic", "entrance"])
def test_steps_on_odd_rows(orc, lj, torch, option):
    shape = (21, 19, 37)
    kw = dict(sgs_model=3 if option == "dynamic" else 1, axis=int(option == "axis"),
              dt_mode=2 if option == "local" else 0, bc=2 if option == "entrance" else 1)
    xyz = lj.synth.jet_grid(*shape, r0=0.0 if option == "axis" else 0.02)
    P = oracle_params(orc, **kw)
    M = orc.metrics(xyz)
    Q0 = orc.init_jet(P, xyz, seed=3, noise=1e-2)
    Qo, _ = orc.run(P, Q0, M, xyz, 5)
    for pc in (lj.PREC_MIXED, lj.PREC_MIXED_COMPACT):
        ctx, _ = device_ctx(lj, torch, shape, xyz, precision=pc, **kw)
        Qd = torch.from_numpy(Q0).cuda()
        assert ctx.les_run_n_steps(5, Qd).status == 0
        assert rel_l2(Qd.cpu().numpy(), Qo) <= 1e-5
