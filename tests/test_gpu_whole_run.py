"""The whole-run kernel where its indexing and its stop test can go wrong
(needs a GPU): sizes around a quad, a 128-pixel tile and a block, unaligned x,
and images whose largest membership change lies outside the sampled pixels."""
import numpy as np
import pytest

import oracle
import phantom
from parity import assert_within, eps32, precision_report

pytestmark = pytest.mark.gpu

EPS, MAX_ITER = 1e-5, 300


@pytest.fixture(scope="module")
def fcm():
    from paper_1601_00072_gb300 import _build
    _build.build()
    from paper_1601_00072_gb300.fcm import FCM
    h = FCM(0)
    yield h
    h.close()


def _cuda(a, shift=0):
    """The array on the GPU, `shift` floats past a 16-byte boundary."""
    import torch
    a = np.ascontiguousarray(a, dtype=np.float32)
    buf = torch.zeros(a.size + 4, device="cuda")
    t = buf[shift:shift + a.size]
    t.copy_(torch.from_numpy(a.reshape(-1)))
    return t.view(a.shape)


def _check(fcm, x, C, m, shift=0, U0=None, V0=None, want=None):
    def run(max_iter):
        kw = {"U0": _cuda(U0, shift)} if U0 is not None else {"V0": _cuda(V0)}
        return fcm.run(_cuda(x, shift), C, m, EPS, max_iter, U=_cuda(np.zeros((C, x.size)), shift), **kw)

    g = run(MAX_ITER)
    assert g.launches == 1
    o = oracle.fcm(x.astype(np.float64), C, m, eps32(EPS), MAX_ITER, U0=U0, V0=V0)
    d = g.iters - o["iters"]
    k = min(g.iters, o["iters"])
    if g.iters > k:
        g = run(k)
    if o["iters"] > k:
        o = oracle.fcm(x.astype(np.float64), C, m, eps32(EPS), k, U0=U0, V0=V0)
    rep = precision_report(g.U.cpu().numpy(), g.V.cpu().numpy(), g.iters + d, o["U"], o["V"], o["iters"], g.J, o["J"][-1])
    assert_within(rep)
    assert rep["J_rel_err"] < 1e-5
    return g


SIZES = [(5, 0), (127, 0), (129, 1), (2048, 2), (2049, 0), (8192, 3)]


@pytest.mark.parametrize("n,shift,m", [(n, s, m) for n, s in SIZES for m in (2.0, 1.5, 3.0, 2.5)]
                         + [(311299, 0, 2.0), (311300, 1, 2.0)])
def test_sizes_and_alignments(fcm, n, shift, m):
    C = 3 if n > 100 else 1
    side = int(np.ceil(np.sqrt(n)))
    img, _ = phantom.phantom2d(4000 + n, side, side, 6.0, means=(10.0, 90.0, 200.0))
    x = img.reshape(-1)[:n]
    V0 = np.array([30.2, 110.7, 180.4])[:C]
    _check(fcm, x, C, m, shift, V0=V0)
    u0 = oracle.memberships(x.astype(np.float64), V0, m).astype(np.float32)
    _check(fcm, x, C, m, shift, U0=u0)


@pytest.mark.parametrize("at", [3, 350003, 699998])
@pytest.mark.parametrize("n", [700004, 700005])
def test_largest_change_outside_the_sample(fcm, n, at):
    """Almost every pixel sits near a center, where memberships hardly move;
    one lies between the centers. The run stops by that pixel's change."""
    rng = np.random.default_rng(n + at)
    x = np.where(rng.random(n) < 0.5, 20.0, 200.0)
    x[rng.integers(0, n, n // 50)] = 140.0
    x[x == 140.0] = 199.0
    x[at] = 108.0
    V0 = np.array([60.3, 150.1])
    g = _check(fcm, x, 2, 2.0, V0=V0)
    assert g.status == 0 and g.delta < EPS


def test_cluster_of_one_pixel(fcm):
    """A cluster whose share of the image is below what the fixed-point exchange
    words carry goes through the slots, in every iteration."""
    rng = np.random.default_rng(11)
    x = np.rint(rng.random(200004) * 100.0)
    x[77777] = 5000.0
    g = _check(fcm, x, 3, 2.0, V0=np.array([20.3, 80.1, 4900.5]))
    assert abs(float(g.V[2]) - 5000.0) < 50.0


@pytest.mark.parametrize("m", [2.0, 1.5, 2.5])
@pytest.mark.parametrize("C", [1, 2, 6, 8])
def test_cluster_counts(fcm, C, m):
    means = tuple(12.0 + 32.0 * j for j in range(C))
    img, _ = phantom.phantom2d(4500 + C, 90, 91, 4.0, means=means)
    x = img.reshape(-1)
    _check(fcm, x, C, m, V0=np.array(means) + 3.3)
