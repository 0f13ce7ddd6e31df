"""Surfel clouds that fall on few tiles, where a tile's list is shared out to several warps: 256 surfels (not
shared out) and one more, lists of one part and remainders, surfels of a pixel and of whole tiles, lists
on several levels, more heavy tiles than the workspace has room for, and a dense spot in an ordinary
cloud.  Counts and depths equal the oracle's bit for bit; the means are sums of at most 20000 FP32 terms
in [0, 1] added in parts, an error of about u sqrt(20000 / 3) = 5e-6 against the method's 1e-4."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402

FOV = 0.8


def cloud(seed, W, H, n, px, spread, slant=0.3):
    """n disks of about px pixels, their centres in the middle `spread` of the view."""
    g = np.random.default_rng(seed)
    ky = 1 / np.tan(FOV / 2)
    r = np.zeros((n, 16), np.float32)
    z = 4.0 * (1 + 0.02 * g.uniform(-1, 1, n))
    r[:, 0] = (g.uniform(-1, 1, n) * spread + 0.01) * z * (W / H) / ky
    r[:, 1] = (g.uniform(-1, 1, n) * spread + 0.01) * z / ky
    r[:, 2] = -z
    r[:, 3] = np.minimum(px / (0.5 * H) * 4.0 / ky, 1.8) * g.uniform(0.7, 1.0, n)
    r[:, 7] = r[:, 3] * g.uniform(0.5, 1.0, n)
    nrm = g.normal(size=(n, 3)) * slant + (0, 0, 1)
    r[:, 4:7] = nrm / np.linalg.norm(nrm, axis=1, keepdims=True)
    r[:, 8:11] = g.normal(size=(n, 3))
    r[:, 11:16] = g.uniform(0, 1, (n, 5))
    r[::37, 3] = 0.0  # dropped
    return r


@pytest.mark.parametrize("W,H,n,px,spread,tol", [
    (8, 4, 256, 1.0, 0.6, 0.01), (8, 4, 257, 1.0, 0.6, 0.01), (8, 4, 5000, 0.6, 0.8, 0.0), (7, 3, 2000, 8.0, 0.5, 0.02),
    (24, 12, 900, 2.0, 0.1, 0.01), (64, 64, 300, 60.0, 0.1, 0.01), (64, 64, 20000, 2.5, 1.0, 0.01),
    (64, 64, 6000, 30.0, 1.0, 0.05), (64, 64, 6000, 200.0, 0.0, 0.01), (200, 120, 4000, 0.7, 0.0, 0.01), (200, 120, 3000, 9.0, 0.02, 0.0),
    (333, 77, 10000, 3.0, 0.05, 0.01), (1, 40, 1000, 1.5, 1.0, 0.01), (300, 1, 3000, 0.5, 1.0, 0.01)])
def test_few_tiles(W, H, n, px, spread, tol):
    check(W, H, cloud(W + n, W, H, n, px, spread), tol)


def test_dense_spot_in_a_cloud():
    check(320, 200, np.concatenate([cloud(1, 320, 200, 30000, 1.5, 1.0), cloud(2, 320, 200, 8000, 1.2, 0.01),
                                    cloud(3, 320, 200, 60, 90.0, 0.5)]), 0.01)


def check(W, H, rec, tol):
    col = np.eye(4, dtype=np.float32).reshape(-1)
    rt = [torch.full((H, W, 4), -1.0, device="cuda"), torch.full((H, W, 4), -1.0, device="cuda"),
          torch.full((H, W), -1.0, device="cuda")]
    wgt = torch.full((H, W), -1.0, device="cuda")
    ep.epbr_surfel_gbuffer(ep.Surfels(torch.from_numpy(rec).cuda()), ep.camera(col, FOV, W, H), 0.05, tol,
                           ep.GBuffer.fp32(*rt), wgt)
    ogb, ow = oracle.surfels(rec, oracle.camera(col, float(np.float32(FOV)), W, H), 0.05, float(np.float32(tol)))
    np.testing.assert_array_equal(wgt.cpu().numpy(), ow)
    np.testing.assert_array_equal(rt[2].cpu().numpy(), ogb[..., 8].astype(np.float32))
    m = ow > 0
    assert m.any()
    got = torch.cat(rt[:2], 2).cpu().numpy()
    np.testing.assert_allclose(got[m], ogb[m][:, :8], rtol=1e-4, atol=1e-5)
    assert (got[~m] == 0).all()


def test_one_tile_is_shared_out():
    """The pass over a cloud that falls on one point takes about twice as long as over the same number of
    surfels spread over the view (two passes over the entries); it was 200 times as long where one warp
    went over a tile's whole list.  Bound: 20 times."""
    W, H, n, col = 640, 480, 300000, np.eye(4, dtype=np.float32).reshape(-1)
    gb = ep.GBuffer.fp32(*(torch.zeros(H, W, c, device="cuda").squeeze(2) for c in (4, 4, 1)))
    ws = torch.empty(ep.epbr_surfel_workspace_size(n, W, H) + 256, dtype=torch.uint8, device="cuda")
    times = []
    for spread in (1.0, 0.0):
        s = ep.Surfels(torch.from_numpy(cloud(5, W, H, n, 0.6, spread)).cuda())
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = np.inf
        for _ in range(5):
            a.record()
            ep.epbr_surfel_gbuffer(s, ep.camera(col, FOV, W, H), 0.05, 0.01, gb, None, workspace=ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[1] <= 20 * times[0], times
