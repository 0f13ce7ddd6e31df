"""Rounding of the prefiltered levels' sums, over environments of one colour: every texel's weighted mean is
that colour, whatever the geometry, so what is left is the rounding of the sums.  With u = 2^-24: a plain
sum of 128 FMAs has a rounding error of about u sqrt(128 / 9) = 3.8 u of itself, independent between sums,
0.5 u of the whole for 64 of them; the compensated sums over them, the weights' sum, its reciprocal and
the product add at most 1.5 u.  Bound: 1.5 u + 6 x 0.5 u = 4.5 u.  (A plain sum over the 1052 samples
that fall between two rows of the first environment has about 11 u.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402

BOUND = 4.5 * 2.0 ** -24


@pytest.mark.parametrize("We,He,M", [(2048, 64, 8), (2048, 64, 16), (1024, 16, 3), (256, 1000, 4), (2048, 1024, 16)])
def test_one_colour(We, He, M):
    N, colour = 2048, np.array([0.7, 1.3, 3.1], np.float32)
    env = torch.ones(He, We, 4, device="cuda")
    env[..., :3] = torch.from_numpy(colour).cuda()
    ibl = ep.Ibl(ep.ibl_params(M, N, 8, 8, 4, 2), We, He)
    ep.epbr_prefilter(env, N, ibl)
    for m in (1, 2):
        if We >> m < 128:
            continue
        g = ibl.level(m).cpu().numpy()[..., :3].astype(np.float64)
        assert np.abs(g / colour - 1).max() <= BOUND, (m, np.abs(g / colour - 1).max() * 2.0 ** 24)
