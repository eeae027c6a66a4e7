"""The FP64 flux kernel's chunk lengths (1, 2, 4, 8 and 16 interfaces per thread,
chosen by the number of points) on extents that are no multiple of a chunk or
a block: jets and boxes, periodic and open along every direction, against the
oracle's residual within the 1e-13 of each component's flux scale of the
other FP64 residual tests."""
import numpy as np
import pytest

from gpu_helpers import device_ctx, oracle_params

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


@pytest.mark.parametrize("shape,per", [
    ((9, 7, 129), None), ((5, 5, 5), (1, 1, 1)), ((37, 31, 43), None), ((47, 41, 43), (0, 1, 0)),
    ((131, 75, 35), None), ((67, 71, 73), (1, 1, 1)),
    ((131, 75, 67), None), ((90, 87, 85), (0, 0, 0)), ((131, 75, 131), None),
    ((109, 111, 107), (1, 0, 0)), ((107, 109, 111), (0, 1, 0))])
def test_residual_for_every_chunk_length(orc, lj, torch, shape, per):
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
    ctx, _ = device_ctx(lj, torch, shape, xyz, shift, sgs_model=1, Re=2000.0, **kw)
    Qd = torch.from_numpy(Q).cuda()
    R = torch.empty_like(Qd)
    ctx.les_rhs(Qd, R)
    Rg, Ro = R.cpu().numpy(), orc.rhs(P, Q, M)
    fscale = (np.abs(M[9]) * np.sqrt(M[0] ** 2 + M[1] ** 2 + M[2] ** 2)).max()
    for c in range(5):
        qs = np.abs(Q[c]).max() + (np.abs(Q[4]).max() if c in (1, 2, 3, 4) else 0.0)
        assert np.abs(Rg[c] - Ro[c]).max() <= 1e-13 * fscale * qs, c
