"""The shadowed compose one light and two lights at a time: a list too short for pairs equals the same list
padded with lights of intensity 0 to a length that takes pairs (their terms are exact zeros), bit for
bit, white and coloured, also where a chunk holds both, and the diffuse-only mode, which has no pairs."""
import numpy as np
import pytest

import synth
from _common import gpu_ibl, gpu_inputs, make_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402


@pytest.mark.parametrize("flags", [ep.EPBR_SHADE_ALL, ep.EPBR_SHADE_ALL | ep.EPBR_SHADE_DIFFUSE_ONLY])
@pytest.mark.parametrize("coloured", [0, 1, 100])
@pytest.mark.parametrize("n,size", [(1, 64), (6, 2), (14, 64), (15, 64)])
def test_short_list_equals_padded(n, size, coloured, flags):
    total = 40
    inp = make_inputs("small", W=45, H=29, lights=total)
    d = gpu_inputs(inp)
    ibl = gpu_ibl(inp, d["env"])
    lights = d["lights"].clone()
    k = min(coloured, n)
    lights[:k, 4:7] = torch.rand(k, 3, generator=torch.Generator().manual_seed(n)).cuda() + 0.1
    if coloured > 1:  # the padding coloured as well
        lights[n:, 4:7] = 0.5 + 0.5 * torch.rand(total - n, 3, generator=torch.Generator().manual_seed(1)).cuda()
    padded = lights.clone()
    padded[n:, 3] = 0.0
    maps = torch.from_numpy(np.random.default_rng(3).uniform(2, 12, (total, size, size)).astype(np.float32)).cuda()
    _, cams = synth.shadow_cameras(inp.scene)
    cams = torch.from_numpy(cams).cuda()
    out = []
    for li in (lights[:n].contiguous(), padded):
        hdr = torch.zeros(inp.H, inp.W, 4, device="cuda")
        ldr = torch.zeros(inp.H, inp.W, 4, dtype=torch.uint8, device="cuda")
        sh = ep.Shadows(maps[:len(li)].contiguous(), cams[:len(li)].contiguous())
        ep.epbr_shade_shadows(d["gb"], d["cam"], li, ibl, ep.shade_params(flags), sh, hdr, 0, ep.tonemap_params(), ldr)
        out.append((hdr.cpu(), ldr.cpu()))
    assert out[0][0].abs().max() > 0
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
