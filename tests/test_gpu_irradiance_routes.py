"""Irradiance of narrow environments, summed texel by texel below 192 columns unless these are whole segments
of 64, by intervals otherwise: widths around the line, one to a few columns, tall maps, and more outputs
than the 512 of a block's group.  Sums of non-negative FP32 terms in tiles of 256 texels, compensated
across, an error of a few 1e-7: the method's 1e-4 relative."""
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


@pytest.mark.parametrize("We,He,Wi,Hi", [(191, 20, 9, 5), (192, 20, 9, 5), (193, 20, 9, 5), (128, 20, 9, 5), (100, 50, 40, 30),
                                         (1, 1, 3, 2), (2, 700, 33, 16), (5, 1030, 7, 3), (190, 7, 1, 1), (65, 300, 32, 17)])
def test_narrow(We, He, Wi, Hi):
    env = synth.make_env(15, We, He)
    out = torch.zeros(Hi, Wi, 4, device="cuda")
    ep.epbr_irradiance(torch.from_numpy(env).cuda(), Wi, Hi, out)
    np.testing.assert_allclose(out.cpu().numpy()[..., :3], oracle.irradiance(env, Wi, Hi), rtol=REL_TOL_FP32)
