"""The fused stage kernel's tile forms: two CTAs of 8 rows per SM (with the tiles
covering eta and zeta exactly, with eta or zeta cut, with rows in 8-byte pieces),
one of 16 rows (small grids with rows that take no 16-byte pieces, of even and of
odd length), one of 8 rows on grids of about a plane per SM, at eta extents
around a multiple of 8.  Every variant of the stage, three steps within 1e-5
(relative L2) of the FP64 oracle's."""
import pytest

from gpu_helpers import device_ctx, oracle_params, rel_l2

pytestmark = pytest.mark.gpu

PAIRS = [(64, 64, 64), (70, 60, 64), (21, 49, 64), (61, 17, 68), (61, 17, 66)]
TALL = [(70, 60, 63), (70, 60, 66)]
SHORT = [(31, 7, 32), (31, 8, 36), (31, 9, 35), (21, 17, 64)]


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


@pytest.mark.parametrize("shape", PAIRS + TALL + SHORT)
@pytest.mark.parametrize("option", ["plain", "local", "axis", "dynamic", "entrance"])
def test_stage_variants(orc, lj, torch, shape, option):
    kw = dict(sgs_model=3 if option == "dynamic" else 1, axis=int(option == "axis"),
              dt_mode=2 if option == "local" else 0, bc=2 if option == "entrance" else 1)
    xyz = lj.synth.jet_grid(*shape, r0=0.0 if option == "axis" else 0.02)
    P = oracle_params(orc, **kw)
    M = orc.metrics(xyz)
    Q0 = orc.init_jet(P, xyz, seed=3, noise=1e-2)
    Qo, _ = orc.run(P, Q0, M, xyz, 3)
    ctx, _ = device_ctx(lj, torch, shape, xyz, precision=lj.PREC_MIXED, **kw)
    Qd = torch.from_numpy(Q0).cuda()
    assert ctx.les_run_n_steps(3, Qd).status == 0
    assert rel_l2(Qd.cpu().numpy(), Qo) <= 1e-5
