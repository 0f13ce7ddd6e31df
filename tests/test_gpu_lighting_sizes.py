"""The lighting set at the sizes where its kernels change path, against the oracle.  Irradiance: rows
walked round (whole segments of 64 columns, at most 2048) and rows in pieces, intervals of a few
columns, outputs that do not divide the source, more outputs than a block has threads.  Prefilter:
rows staged in shared memory (texels 2 or 4 columns apart, shares of the samples) and read through L1,
sample counts below a warp, levels of one texel.  Both sum at most a few thousand non-negative FP32
terms per texel in chunks, an error of a few 1e-7: the method's 1e-4 relative."""
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


@pytest.mark.parametrize("We,He,Wi,Hi", [(64, 3, 32, 16), (128, 65, 5, 3), (2048, 17, 32, 16), (2112, 9, 32, 16),
                                         (4100, 5, 7, 4), (63, 31, 9, 5), (8, 8, 9, 7), (24, 30, 40, 20), (1, 9, 3, 2)])
def test_irradiance_sizes(We, He, Wi, Hi):
    env = synth.make_env(5, We, He)
    out = torch.zeros(Hi, Wi, 4, device="cuda")
    ep.epbr_irradiance(torch.from_numpy(env).cuda(), Wi, Hi, out)
    np.testing.assert_allclose(out.cpu().numpy()[..., :3], oracle.irradiance(env, Wi, Hi), rtol=REL_TOL_FP32)


@pytest.mark.parametrize("We,He,M,N", [(2048, 24, 3, 33), (2048, 8, 8, 200), (1536, 20, 3, 64), (1024, 40, 4, 100),
                                       (640, 20, 3, 64), (512, 64, 5, 128), (256, 33, 6, 7), (256, 2, 4, 1),
                                       (750, 31, 6, 50), (130, 4, 8, 40), (2176, 6, 3, 40)])
def test_prefilter_sizes(We, He, M, N):
    env = synth.make_env(6, We, He)
    ibl = ep.Ibl(ep.ibl_params(M, N, 8, 8, 4, 2), We, He)
    ep.epbr_prefilter(torch.from_numpy(env).cuda(), N, ibl)
    for m in range(1, M):
        ref = oracle.prefilter_level(env, M, N, m)
        g = ibl.level(m).cpu().numpy()[..., :3]
        err = np.abs(g - ref) / np.maximum(np.abs(ref), 1e-3 * ref.mean())
        assert err.max() <= REL_TOL_FP32, (m, err.max())
