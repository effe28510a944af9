"""The index guards of the whole-run kernel in the bounds-guarded build
(FCM_DEBUG_BOUNDS=1, needs a GPU): they are there, and they skip and report.

FCM_DEBUG_BOUNDS_SHORT makes the guards of that build take a few pixels off the
image, so that they reject accesses that are in bounds: nothing out of range is
ever asked for. The build is chosen when the library is loaded, so each run has
its own process.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUN = r"""
import sys
import numpy as np
import torch
sys.path.insert(0, ROOT)
from paper_1601_00072_gb300 import _build
_build.build()
from paper_1601_00072_gb300.fcm import FCM

out = {}
rng = np.random.default_rng(3)
h = FCM(0)
for n in (4096, 4101, 700000):
    x = torch.from_numpy((rng.random(n) * 200.0).astype(np.float32)).cuda()
    for start in ("U", "V"):
        V0 = torch.tensor([20.0, 90.0, 170.0], device="cuda")
        u0 = torch.full((3, n), 1.0 / 3.0, device="cuda") + 0.1 * torch.sin(torch.arange(3 * n, device="cuda").view(3, n).float())
        kw = {"U0": u0} if start == "U" else {"V0": V0}
        U = torch.full((3, n), -1.0, device="cuda")
        r = h.run(x, 3, 2.0, 0.0, 6, U=U, raise_on_error=False, **kw)
        out[f"{n}{start}_U"], out[f"{n}{start}_flags"] = U.cpu().numpy(), np.array(r.flags)
h.close()
np.savez(sys.argv[1], **out)
"""


def _run(tmp_path, name, **env):
    path = str(tmp_path / f"{name}.npz")
    e = {k: v for k, v in os.environ.items() if not k.startswith("FCM_DEBUG_BOUNDS")}
    subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + RUN, path], env={**e, **env}, check=True, timeout=600, cwd=ROOT)
    return dict(np.load(path))


def test_guards_skip_and_report(tmp_path):
    from paper_1601_00072_gb300 import _lib
    bit = _lib.FCM_FLAG_BOUNDS
    plain = _run(tmp_path, "plain", FCM_DEBUG_BOUNDS_SHORT="5")  # the normal build has no guards
    guarded = _run(tmp_path, "guarded", FCM_DEBUG_BOUNDS="1")
    short = _run(tmp_path, "short", FCM_DEBUG_BOUNDS="1", FCM_DEBUG_BOUNDS_SHORT="5")
    for k in plain:
        if k.endswith("_flags"):
            assert not plain[k] & bit and not guarded[k] & bit and short[k] & bit, k
            continue
        assert np.array_equal(plain[k], guarded[k]), k
        n = plain[k].shape[1]
        # the last five pixels are never written; all but their quads or tile are
        assert np.all(short[k][:, n - 5:] == -1.0), k
        assert np.all(short[k][:, :n - 133] >= 0.0), k
        assert np.all(plain[k] >= 0.0)
