"""Starts whose centers lie far from the image, or between parts of it that are
far apart (needs a GPU): a center then moves by many times its new value in one
iteration. Against the FP64 oracle at the same iteration."""
import numpy as np
import pytest

import oracle
from parity import assert_within, center_err, precision_report

pytestmark = pytest.mark.gpu

STEPS = (1, 2, 12)


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


def tissues(n, seed, grey=False):
    rng = np.random.default_rng(seed)
    x = np.where(rng.random(n) < 0.5, 30.0, 90.0) + 6.0 * rng.standard_normal(n)
    x = np.clip(np.rint(x), 0, 255) if grey else x
    return x.astype(np.float32).astype(np.float64), rng


def mixed_start(n, seed):
    """Tissue beside a sentinel of 1e8, and memberships that mix them."""
    x, rng = tissues(n, seed)
    far = rng.random(n) < 0.3
    x[far] = 1e8
    return x, np.where(far, np.array([[0.2], [0.8]]), np.array([[0.9], [0.1]])).astype(np.float32)


def check(g, o):
    assert_within(precision_report(g.U.cpu().numpy(), g.V.cpu().numpy(), g.iters, o["U"], o["V"], o["iters"]))


@pytest.mark.parametrize("m", [2.0, 1.5, 2.5])
@pytest.mark.parametrize("far", [1e6, -300.0])
def test_histogram_run(fcm, far, m):
    x, _ = tissues(40001, 1, grey=True)
    V0 = np.array([20.0, 80.0, far])
    for k in STEPS:
        g = fcm.run_hist(_cuda(x), 3, m, 0.0, k, V0=_cuda(V0))
        check(g, oracle.fcm(x, 3, m, 0.0, k, V0=V0))


@pytest.mark.parametrize("far", [1e6, -300.0])
def test_batched_histogram_run(fcm, far):
    from paper_1601_00072_gb300.fcm import Slice
    V0 = [20.0, 80.0, far]
    for k in STEPS:
        xs = [tissues(n, n, grey=True)[0] for n in (4001, 40000)]
        sl = [Slice(x=_cuda(x), C=3, m=2.0, eps=0.0, max_iter=k, V0=V0) for x in xs]
        fcm.run_batched_hist(sl)
        for s, x in zip(sl, xs):
            check(s, oracle.fcm(x, 3, 2.0, 0.0, k, V0=np.array(V0)))


PLANS = {"queue": dict(block=256), "clusters": dict(block=512, cluster=4, big=2000),
         "teams": dict(schedule="teams", block=256, tile=10)}


@pytest.mark.parametrize("plan", PLANS.values(), ids=PLANS)
def test_batch(fcm, plan):
    """A far initial center, and a start that mixes tissue and a sentinel, in
    one CTA, in a cluster and in a team."""
    from paper_1601_00072_gb300.fcm import Slice
    fcm.set_batched_plan(**plan)
    try:
        for k in STEPS + (3, 4):
            sl, want = [], []
            for n in (37, 4001, 40000):
                x, _ = tissues(n, n)
                for m, far in ((2.0, 1e10), (2.0, -1e6), (1.5, 1e6), (2.5, 1e6)):
                    V0 = [20.0, 80.0, far]
                    sl.append(Slice(x=_cuda(x), C=3, m=m, eps=0.0, max_iter=k, V0=V0))
                    want.append(oracle.fcm(x, 3, m, 0.0, k, V0=np.array(V0)))
                x, u0 = mixed_start(n, n)
                sl.append(Slice(x=_cuda(x), C=2, m=2.0, eps=0.0, max_iter=k, U0=_cuda(u0)))
                want.append(oracle.fcm(x, 2, 2.0, 0.0, k, U0=u0))
            fcm.run_batched(sl)
            for s, o in zip(sl, want):
                check(s, o)
    finally:
        fcm.set_batched_plan()


@pytest.mark.parametrize("m", [2.0, 2.5])
@pytest.mark.parametrize("D", [1, 3])
@pytest.mark.parametrize("n", [37, 40001])
def test_multi_feature_run(fcm, n, D, m):
    """Far in one channel and in all, and a start that mixes tissue and a sentinel."""
    xs = np.stack([tissues(n, 10 + d)[0] for d in range(D)])
    for k in STEPS:
        for far in (np.full(D, 1e6), np.r_[1e6, np.full(D - 1, 50.0)]):
            V0 = np.stack([np.full(D, 20.0), np.full(D, 80.0), far])
            g = fcm.run_multi(_cuda(xs), 3, m, 0.0, k, V0=_cuda(V0))
            check(g, oracle.fcm_multi(xs, 3, m, 0.0, k, V0=V0))
    x, u0 = mixed_start(n, 5)
    xs[0] = x
    for k in (1, 2, 3, 4):
        g = fcm.run_multi(_cuda(xs), 2, m, 0.0, k, U0=_cuda(u0))
        o = oracle.fcm_multi(xs, 2, m, 0.0, k, U0=u0)
        assert center_err(g.V.cpu().numpy(), o["V"]) <= 1e-5
