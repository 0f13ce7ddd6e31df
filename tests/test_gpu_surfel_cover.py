"""Whole-tile surfels between surfels without a pixel in the tile, at the limits of a batch of 32, with a depth
window that leaves nothing out: the weight shows that every large surfel reached the tile's pixels.
Counts and depths equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402


@pytest.mark.parametrize("W,H,large,small", [(8, 4, 33, 0), (16, 4, 20, 44), (24, 12, 40, 200), (7, 3, 32, 5),
                                             (24, 12, 300, 40)])
def test_every_large_surfel_reaches_the_tile(W, H, large, small):
    g = np.random.default_rng(large + 7 * small + W)
    n, tol = large + small, 100.0
    rec = np.zeros((n, 16), np.float32)
    big = np.zeros(n, bool)
    big[g.permutation(n)[:large]] = True
    z = np.where(big, 84.0, 4.0) * (1 + 0.004 * g.uniform(-1, 1, n))
    rec[:, 0], rec[:, 1] = (g.uniform(-1, 1, n) * np.where(big, 0.0, 0.2) * z for _ in range(2))
    rec[:, 2] = -z
    rec[:, 3] = rec[:, 7] = np.where(big, 40.0, 0.01 * z)
    rec[:, 6], rec[:, 8] = 1.0, 1.0
    rec[:, 11:16] = g.uniform(0, 1, (n, 5))
    fov = 0.2
    col = np.eye(4, dtype=np.float32).reshape(-1)
    rt = [torch.full((H, W, 4), -1.0, device="cuda"), torch.full((H, W, 4), -1.0, device="cuda"),
          torch.full((H, W), -1.0, device="cuda")]
    wgt = torch.full((H, W), -1.0, device="cuda")
    ep.epbr_surfel_gbuffer(ep.Surfels(torch.from_numpy(rec).cuda()), ep.camera(col, fov, W, H), 0.05, tol,
                           ep.GBuffer.fp32(*rt), wgt)
    ogb, ow = oracle.surfels(rec, oracle.camera(col, float(np.float32(fov)), W, H), 0.05, tol)
    assert (ow >= large).all()
    np.testing.assert_array_equal(wgt.cpu().numpy(), ow)
    np.testing.assert_array_equal(rt[2].cpu().numpy(), ogb[..., 8].astype(np.float32))
