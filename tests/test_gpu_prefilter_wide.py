"""Prefilter blocks of 512 threads (level 1 of 1024 to 2048 texels per row, 512 samples or more) at the edges of
that rule, and its narrower levels, where the threads left over share the samples.  Sums of at most 2048
FP32 terms in chunks of 64, an error of a few 1e-7: the method's 1e-4 relative."""
import numpy as np
import pytest

import oracle
import synth
from _common import REL_TOL_FP32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402


@pytest.mark.parametrize("We,He,M,N", [(2048, 4, 8, 512), (2048, 4, 3, 511), (2048, 2, 2, 2048), (2304, 4, 3, 600), (4096, 2, 4, 512),
                                       (4098, 2, 2, 512), (2046, 2, 2, 512), (8192, 2, 2, 512), (2560, 8, 6, 700)])
def test_wide_rows(We, He, M, N):
    env = synth.make_env(16, We, He)
    ibl = ep.Ibl(ep.ibl_params(M, N, 8, 8, 4, 2), We, He)
    ep.epbr_prefilter(torch.from_numpy(env).cuda(), N, ibl)
    for m in range(1, M):
        ref = oracle.prefilter_level(env, M, N, m)
        g = ibl.level(m).cpu().numpy()[..., :3]
        err = np.abs(g - ref) / np.maximum(np.abs(ref), 1e-3 * ref.mean())
        assert err.max() <= REL_TOL_FP32, (m, err.max())
