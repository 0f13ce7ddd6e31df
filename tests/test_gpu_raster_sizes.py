"""Mesh coverage at the sizes where it changes path: boxes a thread tests itself (32 pixels), boxes of
one and of several tasks (1024 pixels), edge functions of 32 and 64 bits (181 pixels of extent) and
areas above 2^32.  Ids and depths equal the oracle's bit for bit, as G-buffer and as shadow maps."""
import math

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402

NEAR = 0.05


def soup(seed, n, px, W, H, t):
    """n random triangles of about px pixels of extent before a camera at the origin (some off screen)."""
    g = np.random.default_rng(seed)
    z = g.uniform(1.0, 4.0, n)
    c = np.stack([g.uniform(-0.55, 0.55, n) * 2 * W / H * t, g.uniform(-0.55, 0.55, n) * 2 * t], 1)
    v = np.zeros((n, 3, 12), np.float32)
    off = g.uniform(-0.5, 0.5, (n, 3, 2)) * px * 2 * t / H
    v[:, :, 2] = -(z[:, None] * g.uniform(0.9, 1.1, (n, 3)))
    v[:, :, :2] = (c[:, None] + off) * -v[:, :, 2:3]
    v[:, :, 5] = 1.0
    v[:, :, 6:11] = g.uniform(0, 1, (n, 3, 5))
    return v.reshape(-1, 12), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


@pytest.mark.parametrize("px,n,W,H", [(3, 3000, 200, 150), (8, 2000, 200, 150), (33, 400, 200, 150), (70, 300, 333, 217),
                                      (185, 120, 640, 480), (400, 60, 640, 480), (9000, 40, 257, 193)])
def test_triangle_sizes(px, n, W, H):
    fov = math.radians(60.0)
    verts, tris = soup(px, n, px, W, H, math.tan(0.5 * fov))
    col = np.eye(4, dtype=np.float32).reshape(-1)
    mesh = ep.Mesh(torch.from_numpy(verts).cuda(), torch.from_numpy(tris).cuda())
    rt = [torch.zeros(H, W, 4, device="cuda"), torch.zeros(H, W, 4, device="cuda"), torch.zeros(H, W, device="cuda")]
    ids = torch.zeros(H, W, dtype=torch.int32, device="cuda")
    ep.epbr_raster_gbuffer(mesh, ep.camera(col, fov, W, H), NEAR, ep.GBuffer.fp32(*rt), ids)
    ogb, oids = oracle.raster(verts, tris, oracle.camera(col, float(np.float32(fov)), W, H), NEAR)
    np.testing.assert_array_equal(ids.cpu().numpy(), oids)
    np.testing.assert_array_equal(rt[2].cpu().numpy(), ogb[..., 8].astype(np.float32))
    assert (oids >= 0).any()


@pytest.mark.parametrize("S,lights,tris_per", [(16, 70, 5), (300, 3, 200)])
def test_map_groups(S, lights, tris_per):
    """More maps than a launch takes, and maps whose boxes are queued as one and as several tasks."""
    fov = math.radians(90.0)
    parts = [soup(k, tris_per, px, S, S, 1.0) for k, px in enumerate((4, 40, 150))]
    verts = np.concatenate([p[0] for p in parts])
    tris = np.arange(len(verts), dtype=np.int32).reshape(-1, 3)
    mesh = ep.Mesh(torch.from_numpy(verts).cuda(), torch.from_numpy(tris).cuda())
    cols = []
    for i in range(lights):
        m = synth.camera_matrix((0.3 * math.sin(i), 0.2 * math.cos(i), 0.5), (0.0, 0.0, -2.0))
        cols.append(m.astype(np.float32).T.reshape(-1).copy())
    maps = torch.zeros(lights, S, S, device="cuda")
    ep.epbr_shadow_maps(mesh, [ep.camera(c, fov, S, S) for c in cols], NEAR, maps)
    got = maps.cpu().numpy()
    for i, c in enumerate(cols):
        ogb, _ = oracle.raster(verts, tris, oracle.camera(c, float(np.float32(fov)), S, S), NEAR)
        np.testing.assert_array_equal(got[i], ogb[..., 8].astype(np.float32))
    assert np.isfinite(got).any()
