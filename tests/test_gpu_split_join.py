"""The float pair of the mixed forms' state: hi is the FP64 value rounded to
nearest, lo the rest rounded to nearest (either a zero of its sign where that is
a subnormal float), and the join is their FP64 sum, bit for bit: ties, carries
into the next exponent, zeros of both signs, values near and beyond both ends of
the float range, infinities; counts that are no multiple of the kernels' four
values per thread; the join of any pair, subnormal parts among them, and the join
that also sums the totals."""
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


def _flush(x):
    """Subnormal floats to zeros of their sign."""
    return np.where(np.abs(x) < np.float32(2.0 ** -126), np.copysign(np.float32(0), x), x).astype(np.float32)


def _context(shape):
    import torch
    from paper_2301_00817_gb300 import _build
    _build.build()
    import paper_2301_00817_gb300 as lj
    ctx = lj.Context(lj.make_params(precision=lj.PREC_MIXED), shape)
    ctx.les_set_grid(torch.from_numpy(lj.synth.jet_grid(*shape)).cuda())
    return ctx


def test_low_end_of_the_range():
    """Below 2^-72, where the split converts, down to nothing: the three calls
    that join (the store, a run of no steps on a device state, and one on a
    pinned host state, whose join also sums the totals) give the same bits."""
    import torch
    shape = (5, 6, 7)
    ctx = _context(shape)
    rng = np.random.default_rng(4)
    n = 5 * int(np.prod(shape))
    v = np.ldexp((1.0 + rng.random(n)) * rng.choice([-1.0, 1.0], n), rng.integers(-160, -66, n))
    v[3:10] = [2.0 ** -149, 1e-300, -(2.0 ** -126), 1.3 * 2.0 ** -130, -5e-324, 2.0 ** -73 * (1 + 2.0 ** -30), -0.0]
    hi = _flush(v.astype(np.float32))
    lo = _flush((v - hi.astype(np.float64)).astype(np.float32))
    want = (hi.astype(np.float64) + lo.astype(np.float64)).view(np.uint64)
    Q = torch.from_numpy(v.reshape((5,) + shape)).cuda()
    ctx.les_state_load(Q)
    h, l = (t.cpu().numpy().reshape(-1) for t in ctx.state_views(0, Q))
    assert np.array_equal(h.view(np.uint32), hi.view(np.uint32))
    assert np.array_equal(l.view(np.uint32), lo.view(np.uint32))
    out = torch.empty_like(Q)
    ctx.les_state_store(out)
    run = Q.clone()
    host = Q.cpu().pin_memory()
    ctx.les_run_n_steps(0, run)
    ctx.les_run_host(0, host, torch.empty_like(Q))
    for got in (out, run, host):
        assert np.array_equal(got.cpu().numpy().reshape(-1).view(np.uint64), want)


def test_join_of_subnormal_parts():
    """The boundary kernels may leave a subnormal lo (or a subnormal pair) where
    the split leaves a zero."""
    import torch
    shape = (5, 6, 7)
    ctx = _context(shape)
    rng = np.random.default_rng(5)
    n = 5 * int(np.prod(shape))
    lo = (rng.integers(1, 1 << 23, n) | (rng.integers(0, 2, n) << 31)).astype(np.uint32).view(np.float32)
    hi = np.ldexp(rng.choice([-1.0, 0.0, 1.0], n), rng.integers(-149, -95, n)).astype(np.float32)
    Q = torch.empty((5,) + shape, dtype=torch.float64, device="cuda")
    for view, x in zip(ctx.state_views(0, Q), (hi, lo)):
        view.copy_(torch.from_numpy(x.reshape((5,) + shape)))
    ctx.les_state_store(Q)
    want = hi.astype(np.float64) + lo.astype(np.float64)
    assert np.array_equal(Q.cpu().numpy().reshape(-1).view(np.uint64), want.view(np.uint64))
