"""Large queries of points in no order go through a sorted copy; small ones, and those on another
stream meanwhile, do without.  The results are the same bits."""
import numpy as np
import pytest

from gpu_util import ensure_built

pytestmark = pytest.mark.gpu


def _model(shape, n_bricks, max_points, precision):
    from paper_2308_02494_gb300 import synth
    from paper_2308_02494_gb300.model import SRN

    ms = synth.ModelShape(*shape, 64)
    net = SRN(ms, n_bricks=n_bricks, precision=precision, max_points=max_points)
    net.set_params([synth.parity_model(ms, 3 + b, shrink=0.3) for b in range(n_bricks)])
    return net


def _in_parts(net, x, n_bricks, off, most=10_000):
    """The same points in queries too small for a copy."""
    import torch

    out = torch.empty(len(x), device="cuda")
    for b in range(n_bricks):
        for a in range(off[b], off[b + 1], most):
            e = min(off[b + 1], a + most)
            o = [0] * (b + 1) + [e - a] * (n_bricks - b)
            out[a:e] = net.forward(x[a:e].contiguous(), o)
    return out


# shapes beyond the size below which no batch is sorted: odd resolutions and one channel too
@pytest.mark.parametrize("shape", [(64, 32, 2), (128, 13, 1), (32, 21, 2), (16, 26, 1)])
@pytest.mark.parametrize("precision", ["bf16", "fp32"])
@pytest.mark.parametrize("n_bricks", [1, 3])
def test_sorted_copy_gives_the_same_bits(shape, precision, n_bricks):
    import torch

    ensure_built()
    n = 200_003
    r = np.random.default_rng(n)
    x = r.uniform(-1.02, 1.02, (n, 3)).astype(np.float32)
    x[7], x[8], x[11] = [-1, -1, -1], [1, 1, 1], [3e38, -3e38, 3e38]
    x[9, 1], x[10, 0] = np.nan, np.inf
    x = torch.as_tensor(x, device="cuda")
    off = [0] + [n * (b + 1) // n_bricks for b in range(n_bricks)]
    net = _model(shape, n_bricks, n, precision)
    want = _in_parts(net, x, n_bricks, off)
    for _ in range(2):   # each call's order count is cleared by the one before
        assert torch.equal(net.forward(x, off), want)
    s = torch.argsort(x[:, 0].nan_to_num(0), stable=True)   # a batch in order of x only
    one = [0] + [n] * n_bricks
    assert torch.equal(net.forward(x[s].contiguous(), one), _in_parts(net, x[s].contiguous(), n_bricks, one))
    out = torch.zeros(n, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):   # a captured call does without the copy
        net.forward(x, off, out=out)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


@pytest.mark.parametrize("precision", ["bf16", "fp32"])
def test_a_query_does_not_wait_for_another_streams(precision):
    """Work that one stream has queued before its query holds that query, not another stream's."""
    import torch

    ensure_built()
    n = 200_003
    net = _model((32, 20, 2), 1, n, precision)
    x = [torch.rand((n, 3), device="cuda") * 2 - 1 for _ in range(2)]
    want = [net.forward(v, [0, n]).clone() for v in x]
    out = [torch.zeros(n, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(a):
        torch.cuda._sleep(400_000_000)   # about 0.2 s
    net.forward(x[0], [0, n], out=out[0], stream=a)
    done = torch.cuda.Event()
    done.record(a)
    net.forward(x[1], [0, n], out=out[1], stream=b)
    b.synchronize()
    assert not done.query()
    torch.cuda.synchronize()
    assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])


@pytest.mark.parametrize("n_bricks", [1, 3])
def test_points_written_during_a_query_cost_only_their_values(n_bricks):
    """Points that another stream overwrites while they are being sorted may come out as anything,
    but nothing beyond the batch's outputs is written."""
    import torch

    ensure_built()
    n, most = 200_003, 400_000
    net = _model((32, 20, 2), n_bricks, most, "bf16")
    big = torch.rand((most, 3), device="cuda") * 2 - 1
    net.forward(big, [0] + [most * (b + 1) // n_bricks for b in range(n_bricks)])   # places beyond n, from before
    x = big[:n].clone()
    other = torch.rand((n, 3), device="cuda") * 2 - 1
    out = torch.full((n + 2 * 65536,), 7.5, device="cuda")
    off = [0] + [n * (b + 1) // n_bricks for b in range(n_bricks)]
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for k in range(40):
        with torch.cuda.stream(b):
            x.copy_(other if k % 2 else big[:n])
        net.forward(x, off, out=out[65536:65536 + n], stream=a)
    torch.cuda.synchronize()
    assert bool((out[:65536] == 7.5).all()) and bool((out[65536 + n:] == 7.5).all())
