"""The exchanges and stop decisions of the whole-run kernel (needs a GPU): many
short runs in a row, whose results must not depend on how the blocks' warps
happen to be scheduled."""
import numpy as np
import pytest

import oracle
from parity import assert_within, eps32, precision_report

pytestmark = pytest.mark.gpu

EPS = 1e-5


@pytest.fixture(scope="module")
def fcm():
    from paper_1601_00072_gb300 import _build
    _build.build()
    from paper_1601_00072_gb300.fcm import FCM
    h = FCM(0)
    yield h
    h.close()


def _cuda(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _lone_pixels(n):
    """Almost every pixel sits near a center; a few lie between, mostly outside
    the sampled pairs, so that samples decide some iterations and not others."""
    rng = np.random.default_rng(n)
    x = np.where(rng.random(n) < 0.5, 20.0, 200.0) + np.rint(3.0 * rng.standard_normal(n))
    x[n // 3], x[n // 2 + 1] = 108.0, 113.0
    return x, np.array([60.3, 150.1])


@pytest.mark.parametrize("n", [600, 3001, 40000])
def test_decisions_repeat(fcm, n):
    """A block's warps agree on every decision: 200 runs give the same bits."""
    x, V0 = _lone_pixels(n)
    o = oracle.fcm(x, 2, 2.0, eps32(EPS), 300, V0=V0)
    dx, dv = _cuda(x), _cuda(V0)
    first = None
    for _ in range(200):
        g = fcm.run(dx, 2, 2.0, EPS, 300, V0=dv.clone())
        got = (g.status, g.iters, g.delta, g.J, g.V.cpu().numpy().tobytes())
        first = first or got
        assert got == first
    assert g.status == 0 and abs(g.iters - o["iters"]) <= 1
    if g.iters == o["iters"]:
        assert_within(precision_report(g.U.cpu().numpy(), g.V.cpu().numpy(), g.iters, o["U"], o["V"], o["iters"], g.J, o["J"][-1]))


@pytest.mark.parametrize("n", [520, 4000, 40001])
@pytest.mark.parametrize("max_iter", [1, 2, 3])
@pytest.mark.parametrize("kw", [{}, {"trace": True}], ids=["plain", "trace"])
def test_runs_that_end_at_max_iter(fcm, n, max_iter, kw):
    """The last iteration has no exchange of sums; its full pass follows an
    earlier slot exchange at once. Every run ends, alike, and as the oracle's."""
    x, V0 = _lone_pixels(n)
    o = oracle.fcm(x, 2, 2.0, 0.0, max_iter, V0=V0)
    dx, dv = _cuda(x), _cuda(V0)
    first = None
    for _ in range(100):
        g = fcm.run(dx, 2, 2.0, 0.0, max_iter, V0=dv.clone(), **kw)
        got = (g.status, g.iters, g.delta, g.J, g.V.cpu().numpy().tobytes())
        first = first or got
        assert got == first
    assert g.status == 1 and g.iters == max_iter
    assert_within(precision_report(g.U.cpu().numpy(), g.V.cpu().numpy(), g.iters, o["U"], o["V"], o["iters"], g.J, o["J"][-1]))


def test_undecided_iterations_before_max_iter(fcm):
    """Full passes of the last three iterations, one after the other."""
    x, V0 = _lone_pixels(3001)
    dx, dv = _cuda(x), _cuda(V0)
    end = fcm.run(dx, 2, 2.0, EPS, 300, V0=dv.clone()).iters
    for max_iter in range(2, end + 1):
        o = oracle.fcm(x, 2, 2.0, eps32(EPS), max_iter, V0=V0)
        for _ in range(20):
            g = fcm.run(dx, 2, 2.0, EPS, max_iter, V0=dv.clone())
            assert g.status in (0, 1) and abs(g.iters - o["iters"]) <= 1


def _tissues(n, seed):
    rng = np.random.default_rng(seed)
    x = np.where(rng.random(n) < 0.5, 30.0, 90.0) + 6.0 * rng.standard_normal(n)
    return x.astype(np.float32).astype(np.float64), rng


def _check_centers(fcm, x, C, m, V0, eps=EPS, max_iter=60):
    """Against the oracle at the same iteration count."""
    V0 = np.asarray(V0, np.float32).astype(np.float64)
    g = fcm.run(_cuda(x), C, m, eps, max_iter, V0=_cuda(V0))
    o = oracle.fcm(x, C, m, eps32(eps), max_iter, V0=V0)
    assert abs(g.iters - o["iters"]) <= 1
    k = min(g.iters, o["iters"])
    if g.iters != o["iters"]:
        g = fcm.run(_cuda(x), C, m, eps, k, V0=_cuda(V0))
        o = oracle.fcm(x, C, m, eps32(eps), k, V0=V0)
    assert_within(precision_report(g.U.cpu().numpy(), g.V.cpu().numpy(), g.iters, o["U"], o["V"], o["iters"]))
    return g


@pytest.mark.parametrize("m", [2.0, 1.5, 2.5])
@pytest.mark.parametrize("share", [0.0, 0.01, 0.3], ids=["one", "1pc", "30pc"])
@pytest.mark.parametrize("value", [1e6, -1e10, 1e12, 1e15, 1e18])
def test_tissues_beside_a_sentinel(fcm, value, share, m):
    """One far outlier, or a masked part at a sentinel value, with a cluster of
    its own: the other centers move as if it were not there."""
    n = 200004
    x, rng = _tissues(n, 3)
    if share:
        x[rng.random(n) < share] = np.float32(value)
    else:
        x[n // 3] = np.float32(value)
    _check_centers(fcm, x, 3, m, [20.0, 80.0, value])
    _check_centers(fcm, x, 3, m, [20.0, 80.0, value], eps=0.0, max_iter=9)


@pytest.mark.parametrize("m", [2.0, 1.5, 2.5])
def test_a_far_initial_center(fcm, m):
    """Differences from a center far outside the image have lost the bits of the
    pixels; the center that is formed from them has not."""
    x, _ = _tissues(200004, 4)
    for k in (1, 2, 12):
        _check_centers(fcm, x, 3, m, [20.0, 80.0, 1e6], eps=0.0, max_iter=k)
        if m == 2.0:
            _check_centers(fcm, x, 3, m, [20.0, 80.0, 1e10], eps=0.0, max_iter=k)


@pytest.mark.parametrize("n", [4001, 200004])
def test_a_center_that_leaves_a_sentinel(fcm, n):
    """A start that mixes tissue and a sentinel puts a center between them; it
    falls back to the tissue within two iterations, by 10^4 times its value."""
    x, rng = _tissues(n, 7)
    far = rng.random(n) < 0.3
    x[far] = 1e8
    u0 = np.where(far, np.array([[0.2], [0.8]]), np.array([[0.9], [0.1]])).astype(np.float32)
    for k in (1, 2, 3, 4, 8):
        g = fcm.run(_cuda(x), 2, 2.0, 0.0, k, U0=_cuda(u0))
        o = oracle.fcm(x, 2, 2.0, 0.0, k, U0=u0)
        assert_within(precision_report(g.U.cpu().numpy(), g.V.cpu().numpy(), g.iters, o["U"], o["V"], o["iters"]))


@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1e-12])
def test_tiny_intensities(fcm, scale):
    """All totals far below the largest unit."""
    x, _ = _tissues(40000, 5)
    x = (x * scale).astype(np.float32)
    V0 = np.array([20.0, 80.0]) * scale
    g = fcm.run(_cuda(x), 2, 2.0, 0.0, 8, V0=_cuda(V0))
    o = oracle.fcm(x.astype(np.float64), 2, 2.0, 0.0, 8, V0=V0.astype(np.float32).astype(np.float64))
    assert np.max(np.abs(g.V.cpu().numpy() - o["V"]) / o["V"]) <= 1e-5
    assert np.max(np.abs(g.U.cpu().numpy() - o["U"])) <= 1e-5


def test_overflowed_totals(fcm):
    """Totals that are infinite or NaN: squares beyond FP32 where no center sits
    on the pixel, an infinite center. The run ends as the one that launches a
    kernel per pass does, without waiting for sums that never arrive."""
    n = 40004
    x, rng = _tissues(n, 6)
    far = x.copy()
    far[rng.random(n) < 0.01] = 1e20
    u0 = oracle.memberships(x, np.array([20.0, 80.0]), 2.0)
    cases = [(far, {"V0": np.array([20.0, 80.0])}), (x, {"V0": np.array([20.0, 3e38])}), (1e9 * x, {"U0": 1e15 * u0}),
             (far, {"U0": u0})]
    for xs, start in cases:
        got = []
        for persistent in (True, False):
            g = fcm.run(_cuda(xs), 2, 2.0, 0.0, 5, persistent=persistent, **{k: _cuda(v) for k, v in start.items()})
            got.append(g)
        a, b = got
        assert (a.status, a.iters, a.flags) == (b.status, b.iters, b.flags)
        va, vb = a.V.cpu().numpy(), b.V.cpu().numpy()
        # (an overflowed quotient is NaN in compensated FP32 and infinite in FP64)
        ok = np.isfinite(va)
        assert np.array_equal(ok, np.isfinite(vb)) and np.allclose(va[ok], vb[ok], rtol=1e-5, atol=1e-5)
    # and the handle goes on as before
    _check_centers(fcm, x, 2, 2.0, [20.0, 80.0])


@pytest.mark.parametrize("n", [4000, 40001, 700000])
@pytest.mark.parametrize("m", [2.0, 1.2])
def test_masked_background(fcm, n, m):
    """An exact background whose center goes to 0, in blocks that hold nothing
    else, with and without a sentinel beside it; and a center that sits on 0."""
    x, _ = _tissues(n, 8)
    x[:n // 2] = 0.0
    _check_centers(fcm, x, 3, m, [3.0, 25.0, 80.0], max_iter=40)
    far = x.copy()
    far[:n // 8] = 1e9
    _check_centers(fcm, far, 4, m, [0.0, 25.0, 80.0, 1e9], eps=0.0, max_iter=24)
    levels = np.where(x > 60.0, 255.0, np.where(x > 0.0, 100.0, 0.0))
    _check_centers(fcm, levels, 3, m, [10.0, 90.0, 240.0], eps=0.0, max_iter=24)
