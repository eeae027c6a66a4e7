"""The mixed forms' test filter (rows in fours, axial chunks of twelve planes or
more) on extents that are no multiple of its tiles, on boxes periodic and open
along every direction and on a jet: the dynamic procedure's six averaged terms
against the FP64 oracle's within 1e-4 of the larger of each pair (FP32 products
and filters; one wrong row, column or plane of these grids would show at 1e-3
and more)."""
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
    ((25, 21, 37), (1, 1, 1)), ((26, 9, 33), (0, 0, 0)), ((24, 18, 31), (1, 0, 1)), ((37, 23, 32), (0, 1, 0)),
    ((13, 7, 65), (0, 1, 1)), ((6, 6, 6), (1, 1, 1)), ((49, 23, 35), None)])
def test_mixed_averages(orc, lj, torch, shape, per):
    if per is None:
        kw, shift, xyz = dict(periodic=(0, 0, 1), bc=1), None, lj.synth.jet_grid(*shape)
    else:
        kw = dict(periodic=per, bc=0)
        xyz, shift = lj.synth.box_grid(shape, (1.0, 1.3, 0.8), wave=0.25)
    P = oracle_params(orc, sgs_model=3, **kw)
    M = orc.metrics(xyz, kw["periodic"], shift)
    L = (20.0, 20.0, 20.0) if per is None else (1.0, 1.3, 0.8)
    Q = orc.prim_to_cons(P, lj.synth.smooth_periodic_prim(xyz, L, amp=0.3, seed=4))
    want = orc.dynamic_coefficients(P, Q, M)
    for prec in (lj.PREC_MIXED, lj.PREC_MIXED_COMPACT):
        ctx, _ = device_ctx(lj, torch, shape, xyz, shift, sgs_model=lj.SGS_DYNAMIC, precision=prec, **kw)
        got = ctx.les_dynamic_coefficients(torch.from_numpy(Q).cuda())
        for num, den in (("numC", "denC"), ("numI", "denI"), ("numP", "denP")):
            scale = max(abs(want[num]), abs(want[den]))
            for k in (num, den):
                assert abs(got[k] - want[k]) <= 1e-4 * scale, (k, got[k], want[k])
