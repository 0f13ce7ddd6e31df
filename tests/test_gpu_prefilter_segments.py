"""The lighting set where its launches change form: rows of a level split into segments of 512 down to
128 texels (the fewer the rows, the shorter), remainders of a few texels, whole-column and fractional
shifts, and the whole set (its kernels overlapped) against the parts called one by one."""
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


@pytest.mark.parametrize("We,He,M", [(2080, 6, 3), (1032, 12, 4), (258, 6, 3), (254, 6, 3), (1024, 4, 5), (3000, 2, 2),
                                     (2304, 40, 3), (1100, 640, 2)])
def test_row_segments(We, He, M):
    env, N = synth.make_env(8, We, He), 9
    ibl = ep.Ibl(ep.ibl_params(M, N, 8, 8, 4, 2), We, He)
    ep.epbr_prefilter(torch.from_numpy(env).cuda(), N, ibl)
    np.testing.assert_array_equal(ibl.level(0).cpu().numpy()[..., :3], env[..., :3])
    for m in range(1, M):
        ref = oracle.prefilter_level(env, M, N, m)
        g = ibl.level(m).cpu().numpy()[..., :3]
        err = np.abs(g - ref) / np.maximum(np.abs(ref), 1e-3 * ref.mean())
        assert err.max() <= REL_TOL_FP32, (m, err.max())


@pytest.mark.parametrize("We,He,M", [(64, 32, 1), (64, 32, 4), (512, 256, 2), (512, 256, 6), (750, 31, 5)])
def test_set_equals_parts(We, He, M):
    env = torch.from_numpy(synth.make_env(9, We, He)).cuda()
    p = ep.ibl_params(M, 64, 16, 64, 8, 4)
    a, b = ep.Ibl(p, We, He), ep.Ibl(p, We, He)
    irr, lut = torch.zeros(4, 8, 4, device="cuda"), torch.zeros(16, 16, 2, device="cuda")
    ep.epbr_precompute_ibl(env, a)
    ep.epbr_prefilter(env, 64, b)
    ep.epbr_irradiance(env, 8, 4, irr)
    ep.epbr_brdf_lut(16, 64, lut)
    for m in range(M):
        assert torch.equal(a.level(m), b.level(m)), m
    assert torch.equal(a.irradiance().view(4, 8, 4), irr) and torch.equal(a.lut().view(16, 16, 2), lut)


@pytest.mark.parametrize("We,He,M", [(64, 32, 1), (512, 256, 6), (750, 31, 5)])
def test_set_under_capture(We, He, M):
    env = torch.from_numpy(synth.make_env(10, We, He)).cuda()
    p = ep.ibl_params(M, 64, 16, 64, 8, 4)
    a, b = ep.Ibl(p, We, He), ep.Ibl(p, We, He)
    ep.epbr_precompute_ibl(env, a)
    ws = torch.empty(ep.epbr_precompute_ibl_workspace_size(p, We, He) + 512, dtype=torch.uint8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ep.epbr_precompute_ibl(env, b, workspace=ws)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    for m in range(M):
        assert torch.equal(a.level(m), b.level(m)), m
    assert torch.equal(a.irradiance(), b.irradiance()) and torch.equal(a.lut(), b.lut())
