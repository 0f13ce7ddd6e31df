"""Prefilter sample counts whose dynamic shared memory (26 bytes a sample) lies below 48 KB while the
kernel's whole shared memory does not: accepted in a process that has not prefiltered with more samples
before, for whole-column and fractional shifts.  Sums of at most 2048 FP32 terms in chunks of 64, an
error of a few 1e-7: the method's 1e-4 relative."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import sys
sys.path[:0] = [{root!r}, {root!r} + "/tests"]
import numpy as np, torch
import oracle, synth
import paper_2012_03325_gb300 as ep
from _common import REL_TOL_FP32
We, He, M = {We}, {He}, 4
env = synth.make_env(11, We, He)
t = torch.from_numpy(env).cuda()
for N in (1641, 1642, 1800, 1878, 1879, 1890, 1891, 2048):
    ibl = ep.Ibl(ep.ibl_params(M, N, 8, 8, 4, 2), We, He)
    ep.epbr_prefilter(t, N, ibl)
    for m in range(1, M):
        ref = oracle.prefilter_level(env, M, N, m)
        g = ibl.level(m).cpu().numpy()[..., :3]
        err = np.abs(g - ref) / np.maximum(np.abs(ref), 1e-3 * ref.mean())
        assert err.max() <= REL_TOL_FP32, (N, m, err.max())
"""


@pytest.mark.parametrize("We,He", [(64, 32), (50, 24)])
def test_counts_in_a_fresh_process(We, He):
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, We=We, He=He)], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
