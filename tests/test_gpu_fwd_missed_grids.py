"""Float32 queries of a model with 64 nodes per axis, some of whose grids a group of points
misses on one axis alone."""
import numpy as np
import pytest

from gpu_util import ensure_built, morton_order

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 64, 2), (128, 59, 1)])
@pytest.mark.parametrize("order", ["bins", "shuffled"])
def test_missed_grids_do_not_change_the_query(shape, order):
    """One large batch (staged boxes) is bit-equal to the same points in small ones (no boxes)."""
    import torch

    from paper_2308_02494_gb300 import synth
    from paper_2308_02494_gb300.model import SRN

    ensure_built()
    n = 20_000
    ms = synth.ModelShape(*shape, 64)
    p = synth.parity_model(ms, 5, shrink=0.0)
    g = np.zeros((shape[0], 3, 4), dtype=np.float32)
    for d in range(3):
        g[:, d, d] = 1
    g[::2, 2, 2], g[::2, 2, 3] = 2, 1.6      # beyond z = -0.3
    g[1::4, 0, 0], g[1::4, 0, 3] = 2, -1.6   # beyond x = 0.3
    p["G"] = g
    net = SRN(ms, n_bricks=1, precision="fp32", max_points=n)
    net.set_params([p])
    r = np.random.default_rng(1)
    x = r.uniform(-1, 1, (n, 3)).astype(np.float32)
    if order == "bins":
        x = x[morton_order(x)]
    xt = torch.as_tensor(x, device="cuda")
    whole = net.forward(xt, [0, n])
    parts = torch.cat([net.forward(xt[a:a + 1000].contiguous(), [0, 1000]) for a in range(0, n, 1000)])
    assert torch.equal(whole, parts)
