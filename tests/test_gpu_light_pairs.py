"""Light loops that take two pixels or two lights at a time: light counts around their pairs and chunks
(128 with shadows, 256 without), coloured and monochrome lists, a pixel whose pair partner is background
or outside the image, maps too small for a whole 3x3 block.  A list of n lights equals the list of its
first n padded with lights of intensity 0, bit for bit (their terms are exact zeros), and the padded
list takes the loops through another split into pairs and chunks."""
import numpy as np
import pytest

import synth
from _common import gpu_ibl, gpu_inputs, make_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402


@pytest.mark.parametrize("shadow", [0, 1, 2, 5, 64])
@pytest.mark.parametrize("colour", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 127, 128, 129])
def test_padding_a_light_list_changes_nothing(n, colour, shadow):
    inp = make_inputs("small", W=37, H=23, lights=n + 3)
    d = gpu_inputs(inp)
    ibl = gpu_ibl(inp, d["env"])
    lights = d["lights"].clone()
    if colour:
        lights[:, 4:7] = torch.rand(n + 3, 3, generator=torch.Generator().manual_seed(n)).cuda() + 0.1
    padded = lights.clone()
    padded[n:, 3] = 0.0
    out = []
    for li in (lights[:n].contiguous(), padded):
        hdr = torch.zeros(inp.H, inp.W, 4, device="cuda")
        ldr = torch.zeros(inp.H, inp.W, 4, dtype=torch.uint8, device="cuda")
        if shadow:
            maps = torch.from_numpy(np.random.default_rng(3).uniform(2, 12, (n + 3, shadow, shadow)).astype(np.float32))
            _, cams = synth.shadow_cameras(inp.scene)
            sh = ep.Shadows(maps[:len(li)].cuda().contiguous(), torch.from_numpy(cams[:len(li)]).cuda().contiguous())
            ep.epbr_shade_shadows(d["gb"], d["cam"], li, ibl, ep.shade_params(), sh, hdr, 0, ep.tonemap_params(), ldr)
        else:
            ep.epbr_shade_tonemap(d["gb"], d["cam"], li, ibl, ep.shade_params(), hdr, 0, ep.tonemap_params(), ldr)
        out.append((hdr.cpu(), ldr.cpu()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
