"""Surfel lists at the sizes where they change path: images smaller and larger than a tile by a
pixel, more surfels in a tile than one batch (32), boxes listed on coarser levels, and windows that a
nearer surfel moves past part of what was blended.  Counts and depths equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402


def disks(seed, n, lo, hi, depth, spread):
    """n disks of pixel-like sizes lo..hi (fractions of the view) facing roughly the camera at the origin."""
    g = np.random.default_rng(seed)
    r = np.zeros((n, 16), np.float32)
    z = depth * (1 + spread * g.uniform(-1, 1, n))
    r[:, 0], r[:, 1], r[:, 2] = g.uniform(-0.6, 0.6, n) * z, g.uniform(-0.6, 0.6, n) * z, -z
    r[:, 3] = np.exp(g.uniform(np.log(lo), np.log(hi), n)) * z
    r[:, 7] = r[:, 3] * g.uniform(0.4, 1.0, n)
    nrm = g.normal(size=(n, 3)) * 0.4 + (0, 0, 1)
    r[:, 4:7] = nrm / np.linalg.norm(nrm, axis=1, keepdims=True)
    r[:, 8:11] = g.normal(size=(n, 3))
    r[:, 11:16] = g.uniform(0, 1, (n, 5))
    return r


@pytest.mark.parametrize("W,H,n,lo,hi,depth,spread,tol", [
    (1, 1, 40, 0.01, 0.4, 3.0, 0.02, 0.01), (8, 4, 100, 0.01, 0.3, 3.0, 0.02, 0.01),
    (9, 5, 300, 0.01, 0.3, 3.0, 0.015, 0.01), (33, 17, 3000, 0.002, 0.05, 3.0, 0.012, 0.01),
    (200, 120, 4000, 0.003, 0.9, 5.0, 0.02, 0.02), (200, 120, 33, 0.2, 2.0, 5.0, 0.5, 0.05),
    (257, 259, 2000, 0.0005, 0.2, 4.0, 0.3, 0.0)])
def test_tiles_and_lists(W, H, n, lo, hi, depth, spread, tol):
    rec = disks(W + n, n, lo, hi, depth, spread)
    fov = 1.1
    col = np.eye(4, dtype=np.float32).reshape(-1)
    rt = [torch.full((H, W, 4), -1.0, device="cuda"), torch.full((H, W, 4), -1.0, device="cuda"),
          torch.full((H, W), -1.0, device="cuda")]
    wgt = torch.full((H, W), -1.0, device="cuda")
    ep.epbr_surfel_gbuffer(ep.Surfels(torch.from_numpy(rec).cuda()), ep.camera(col, fov, W, H), 0.05, tol,
                           ep.GBuffer.fp32(*rt), wgt)
    ogb, ow = oracle.surfels(rec, oracle.camera(col, float(np.float32(fov)), W, H), 0.05, float(np.float32(tol)))
    np.testing.assert_array_equal(wgt.cpu().numpy(), ow)
    np.testing.assert_array_equal(rt[2].cpu().numpy(), ogb[..., 8].astype(np.float32))
    m = ow > 0
    assert m.any()
    got = torch.cat(rt[:2], 2).cpu().numpy()
    # means of up to a few hundred FP32 terms in [0, 1]: well within the method's 1e-4
    np.testing.assert_allclose(got[m], ogb[m][:, :8], rtol=1e-4, atol=1e-5)
    assert (got[~m] == 0).all()
