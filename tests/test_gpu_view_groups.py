"""How a view's samples are grouped (batches, bundles of rays, staged boxes or none, which CTA takes
which group) must not matter: each sample's value is the same bits."""
import numpy as np
import pytest

from gpu_util import ensure_built

pytestmark = pytest.mark.gpu
CAM = {"eye": [1.9, 1.1, 2.0], "forward": [-0.64, -0.37, -0.673], "right": [0.724, 0.0, -0.69],
       "up": [-0.255, 0.929, -0.268], "scale": 0.45, "ortho": 0}


def _model(shape, grid, precision, max_points):
    from paper_2308_02494_gb300 import synth
    from paper_2308_02494_gb300.model import SRN

    nb = grid[0] * grid[1] * grid[2]
    ms = synth.ModelShape(*shape, 64)
    net = SRN(ms, n_bricks=nb, precision=precision, max_points=max_points)
    net.set_params([synth.parity_model(ms, 3 + b, shrink=0.3) for b in range(nb)])
    boxes = []
    for k in range(grid[2]):
        for j in range(grid[1]):
            for i in range(grid[0]):
                lo = [64 // g * a for a, g in zip((i, j, k), grid)]
                boxes.append(lo + [63 if a == g - 1 else v + 64 // g for a, g, v in zip((i, j, k), grid, lo)])
    return net, np.array(boxes)


@pytest.mark.parametrize("shape", [(16, 9, 1), (32, 20, 2), (64, 32, 2)])
@pytest.mark.parametrize("precision", ["bf16", "fp32"])
# few samples per node (no boxes), many (boxes), and a view that most rays miss
@pytest.mark.parametrize("width,height,samples,scale", [(61, 47, 24, 0.45), (200, 150, 300, 0.45), (129, 97, 98, 1.6)])
@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 1, 2)])
def test_batches_and_replays_give_the_same_image(shape, precision, width, height, samples, scale, grid):
    import torch

    ensure_built()
    cam = {**CAM, "scale": scale, "ortho": scale > 1}
    lut = torch.linspace(0, 1, 256, device="cuda")[:, None].repeat(1, 4).contiguous()
    lut[:, 3] *= 0.01
    images = []
    for most in (1 << 24, 40_000):
        net, boxes = _model(shape, grid, precision, most)

        def go(rgba):
            return net.render(cam, lut, 0.0, 1.0, width, height, samples, grid, boxes, 64, rgba=rgba)

        images.append(go(torch.full((height, width, 4), -1.0, device="cuda")).clone())
    assert torch.equal(images[0], images[1])
    out = torch.zeros_like(images[0])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        go(out)
    for _ in range(3):   # each batch leaves the counter of its groups at zero
        out.fill_(-1.0)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, images[0])
