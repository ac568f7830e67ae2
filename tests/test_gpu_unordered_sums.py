"""Gradients of a batch in no order: the sums over points keep what float32 sums keep, also small
contributions beside large ones, infinities and NaN, however the batch is run."""
import numpy as np
import pytest

from gpu_util import ensure_built, rel_l2

pytestmark = pytest.mark.gpu
SHAPES = [(16, 9, 1), (32, 20, 2), (64, 32, 2)]


def _model(shape, n_bricks, n):
    from paper_2308_02494_gb300 import synth
    from paper_2308_02494_gb300.model import SRN

    ms = synth.ModelShape(*shape, 64)
    net = SRN(ms, n_bricks=n_bricks, precision="bf16", max_points=n)
    net.set_params([synth.parity_model(ms, 3 + b, shrink=0.3) for b in range(n_bricks)])
    return net


def _grad(net, x, up, off):
    net.backward(x, up, off, upstream=True)
    return net.grads[net.lay.off_F:net.lay.off_W1].clone()


# with a sorted copy, and too few points for one
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [60_001, 3_001])
def test_small_contributions_beside_large_ones(shape, n):
    """An upstream of 2^-30 on a slab thinner than a tile, and of 1 elsewhere: dL/dy of a point is its
    upstream times the same number, exactly, so the gradient is the sum of both parts', and what only
    the slab's points reach is theirs, scaled."""
    import torch

    ensure_built()
    r = np.random.default_rng(n)
    x = torch.as_tensor(r.uniform(-1, 1, (n, 3)).astype(np.float32), device="cuda")
    slab = (x[:, 0] > 0.02) & (x[:, 0] < 0.3)
    net = _model(shape, 1, n)
    sign = torch.as_tensor(r.choice([-1.0, 1.0], n).astype(np.float32), device="cuda")
    zero = torch.zeros(n, device="cuda")
    ours = _grad(net, x, torch.where(slab, sign, zero), [0, n])
    theirs = _grad(net, x, torch.where(slab, zero, sign), [0, n])
    both = _grad(net, x, torch.where(slab, sign * 2.0 ** -30, sign), [0, n])
    only = (theirs == 0) & (ours != 0)
    assert int(only.sum()) > 0
    # float32 sums of up to a few hundred terms: 2^-24 each of a partial sum, in the norm
    assert rel_l2((both[only] * 2.0 ** 30).double().cpu(), ours[only].double().cpu()) < 1e-5
    assert rel_l2(both[~only].double().cpu(), theirs[~only].double().cpu()) < 1e-5


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [60_001, 3_001])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_an_infinite_upstream_shows_in_its_nodes(shape, n, bad):
    import torch

    ensure_built()
    r = np.random.default_rng(n)
    x = torch.as_tensor(r.uniform(-1, 1, (n, 3)).astype(np.float32), device="cuda")
    net = _model(shape, 1, n)
    up = torch.as_tensor(r.standard_normal(n).astype(np.float32), device="cuda")
    one = torch.zeros(n, device="cuda")
    one[n // 2] = 1.0
    nodes = _grad(net, x, one, [0, n]) != 0
    assert 8 <= int(nodes.sum())
    up[n // 2] = bad
    g = _grad(net, x, up, [0, n])
    assert not bool(torch.isfinite(g[nodes]).any())
    assert int((~torch.isfinite(g)).sum()) <= 8 * shape[0] * shape[2]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [1_000, 12_007, 160_001])
@pytest.mark.parametrize("density", [False, True])
def test_gradients_do_not_depend_on_the_run(shape, n, density):
    """Three bricks' batch in no order against the same points in smaller calls of one brick each."""
    import torch

    ensure_built()
    r = np.random.default_rng(n)
    off = [0, n // 4, n // 4, n]
    off[2] = n // 4 + 200
    x = torch.as_tensor(r.uniform(-1, 1, (n, 3)).astype(np.float32), device="cuda")
    t = torch.as_tensor(r.uniform(0, 1, n).astype(np.float32), device="cuda")
    net = _model(shape, 3, n)
    losses = net.backward(x, t, off, density=density).cpu().numpy().copy()
    got = net.get("grads")
    from paper_2308_02494_gb300 import synth

    for b in range(3):
        a, e = off[b], off[b + 1]
        m = _model(shape, 1, n)
        m.set_params([synth.parity_model(synth.ModelShape(*shape, 64), 3 + b, shrink=0.3)])
        p = torch.randperm(e - a, device="cuda")
        want_l = m.backward(x[a:e][p].contiguous(), t[a:e][p].contiguous(), [0, e - a], density=density).cpu().numpy()
        want = m.get("grads")[0]
        np.testing.assert_allclose(losses[b], want_l[0], rtol=1e-5)
        for k in ("F", "W1", "W2", "w3") + (("G",) if density else ()):
            assert rel_l2(got[b][k], want[k]) < 1e-4, (b, k)


@pytest.mark.parametrize("shape", [(16, 9, 1), (16, 16, 1), (32, 20, 1), (32, 21, 2), (64, 32, 2)])
def test_features_do_not_depend_on_the_run(shape):
    """A batch large enough for a sorted copy against its two halves, which are not: the same features,
    so the gradients differ by the roundings of float32 sums only (a feature's other rounding to
    bfloat16 flips ReLU masks: 1e-4 and more)."""
    import torch

    ensure_built()
    n = 90_000
    r = np.random.default_rng(n)
    x = torch.as_tensor(r.uniform(-1, 1, (n, 3)).astype(np.float32), device="cuda")
    up = torch.as_tensor(r.standard_normal(n).astype(np.float32), device="cuda")
    net = _model(shape, 1, n)
    whole = _grad(net, x, up, [0, n])
    h = n // 2
    parts = _grad(net, x[:h].contiguous(), up[:h].contiguous(), [0, h]) + _grad(net, x[h:].contiguous(), up[h:].contiguous(), [0, h])
    assert rel_l2(whole.double().cpu(), parts.double().cpu()) < 1e-5
