"""The float pair of the mixed forms' state: hi is the FP64 value rounded to
nearest, lo the rest rounded to nearest, and the join is their FP64 sum, bit
for bit, over the whole range (ties, carries into the next exponent, zeros of
both signs, values near and beyond the float range's ends, infinities) and
for counts that are no multiple of the kernels' four values per thread."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(5, 5, 5), (5, 6, 7), (9, 16, 32)])
def test_split_and_join_bits(shape):
    import torch
    from paper_2301_00817_gb300 import _build
    _build.build()
    import paper_2301_00817_gb300 as lj
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    ctx = lj.Context(lj.make_params(precision=lj.PREC_MIXED), shape)
    ctx.les_set_grid(torch.from_numpy(lj.synth.jet_grid(*shape)).cuda())
    rng = np.random.default_rng(3)
    n = 5 * int(np.prod(shape))
    bits = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    bits[::3] &= ~np.uint64((1 << 29) - 1)
    bits[::6] |= np.uint64(1 << 28)  # ties
    bits[1::7] |= np.uint64(((1 << 23) - 1) << 29)  # carries
    expo = rng.integers(1023 - 60, 1023 + 60, n).astype(np.uint64)
    expo[::11] = rng.integers(1023 - 71, 1023 + 126, len(expo[::11])).astype(np.uint64)
    v = (bits | (expo << np.uint64(52))).view(np.float64) * rng.choice([-1.0, 1.0], n)
    v[5:13] = [0.0, -0.0, np.inf, -np.inf, 2.0 ** -72, -(2.0 ** 126), 2.0 ** 127 * 1.5, 1e300]
    with np.errstate(over="ignore", invalid="ignore"):
        hi = v.astype(np.float32)
        lo = (v - hi.astype(np.float64)).astype(np.float32)
        joined = hi.astype(np.float64) + lo.astype(np.float64)
    Q = torch.from_numpy(v.reshape((5,) + shape)).cuda()
    ctx.les_state_load(Q)
    h, l = (t.cpu().numpy().reshape(-1) for t in ctx.state_views(0, Q))
    ok = ~np.isnan(joined)
    assert np.array_equal(h.view(np.uint32), hi.view(np.uint32))
    assert np.array_equal(l[ok].view(np.uint32), lo[ok].view(np.uint32))
    assert not np.isfinite(l[~ok]).any()
    out = torch.empty_like(Q)
    ctx.les_state_store(out)
    got = out.cpu().numpy().reshape(-1)
    assert np.array_equal(got[ok].view(np.uint64), joined[ok].view(np.uint64))
