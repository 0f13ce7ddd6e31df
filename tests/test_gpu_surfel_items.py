"""Surfel tiles at the limits of a batch's items: 32 surfels that cover a whole 8 x 4 tile (1024 items),
one more, and whole-tile surfels between surfels without a pixel in the tile.  Counts and depths equal
the oracle's bit for bit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402


@pytest.mark.parametrize("W,H,large,small", [(8, 4, 31, 0), (8, 4, 32, 0), (8, 4, 33, 0), (8, 4, 64, 0), (16, 4, 20, 44),
                                             (24, 12, 40, 200), (7, 3, 32, 5), (1, 4, 32, 0)])
def test_batches_of_items(W, H, large, small):
    g = np.random.default_rng(large + 7 * small + W)
    n = large + small
    rec = np.zeros((n, 16), np.float32)
    z = 4.0 * (1 + 0.004 * g.uniform(-1, 1, n))
    big = np.zeros(n, bool)
    big[g.permutation(n)[:large]] = True
    spread = np.where(big, 0.0, 0.7)
    rec[:, 0], rec[:, 1], rec[:, 2] = g.uniform(-1, 1, n) * spread * z, g.uniform(-1, 1, n) * spread * z, -z
    rec[:, 3] = np.where(big, 40.0, 0.02 * z)
    rec[:, 7] = rec[:, 3]
    rec[:, 6], rec[:, 8] = 1.0, 1.0
    rec[:, 2] -= np.where(big, 80.0, 0.0)  # in front of the near rule: nearer than a + b is dropped
    rec[:, 11:16] = g.uniform(0, 1, (n, 5))
    fov = 0.6
    col = np.eye(4, dtype=np.float32).reshape(-1)
    rt = [torch.full((H, W, 4), -1.0, device="cuda"), torch.full((H, W, 4), -1.0, device="cuda"),
          torch.full((H, W), -1.0, device="cuda")]
    wgt = torch.full((H, W), -1.0, device="cuda")
    ep.epbr_surfel_gbuffer(ep.Surfels(torch.from_numpy(rec).cuda()), ep.camera(col, fov, W, H), 0.05, 0.01,
                           ep.GBuffer.fp32(*rt), wgt)
    ogb, ow = oracle.surfels(rec, oracle.camera(col, float(np.float32(fov)), W, H), 0.05, float(np.float32(0.01)))
    assert ow.max() >= large or small
    np.testing.assert_array_equal(wgt.cpu().numpy(), ow)
    np.testing.assert_array_equal(rt[2].cpu().numpy(), ogb[..., 8].astype(np.float32))
    m = ow > 0
    got = torch.cat(rt[:2], 2).cpu().numpy()
    # means of at most a few hundred FP32 terms in [0, 1]
    np.testing.assert_allclose(got[m], ogb[m][:, :8], rtol=1e-4, atol=1e-5)
