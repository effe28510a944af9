"""Which values of U^0 the batched histogram path refuses (needs a GPU)."""
import numpy as np
import pytest

import phantom

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


@pytest.mark.parametrize("value,refused", [(np.nan, True), (np.inf, True), (-np.inf, True), (-1e-6, True),
                                           (-0.0, False), (1e20, False), (1e-44, False)])
def test_which_memberships_are_bad_input(fcm, value, refused):
    """NaN, infinite and negative entries of U^0, and no others: one whose u^m
    overflows only empties its cluster, as in the other entry points. The
    slice beside it keeps its own status."""
    from paper_1601_00072_gb300.fcm import Slice
    img, _ = phantom.phantom2d(77, 64, 65, 6.0)
    x = img.reshape(-1).astype(np.float32)
    u0 = phantom.dirichlet_u0((77, 1), 3, x.size).astype(np.float32)
    bad = u0.copy()
    bad[1, 1234] = value
    sl = [Slice(x=_cuda(x), C=3, U0=_cuda(bad)), Slice(x=_cuda(x), C=3, U0=_cuda(u0))]
    fcm.run_batched_hist(sl)
    assert (sl[0].status == -4) == refused, sl[0].status
    assert sl[1].status == 0
    r = fcm.run(_cuda(x), 3, 2.0, EPS, 300, U0=_cuda(bad), raise_on_error=False)
    assert (r.status == -4) == refused, r.status
