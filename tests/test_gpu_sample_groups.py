"""The grouped BF16 queries and the sorted copies of batches: where a point lies in its
batch, and which way its corners are read (staged boxes or the grid), must not matter."""
import numpy as np
import pytest

from gpu_util import ensure_built, morton_order, rel_l2

pytestmark = pytest.mark.gpu
SHAPES = [(8, 16, 2), (16, 9, 1), (64, 13, 1), (32, 20, 2), (64, 32, 2)]


def _model(shape, n_bricks, max_points, seed=3, precision="bf16"):
    from paper_2308_02494_gb300 import synth
    from paper_2308_02494_gb300.model import SRN

    ms = synth.ModelShape(*shape, 64)
    net = SRN(ms, n_bricks=n_bricks, precision=precision, max_points=max_points)
    net.set_params([synth.parity_model(ms, seed + b, shrink=0.3) for b in range(n_bricks)])
    return net


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [1, 127, 129, 3000, 40_001, 180_001])
def test_forward_bits_do_not_depend_on_the_order(shape, n):
    """Bin-sorted points read staged boxes, shuffled ones the grid (small batches) or a
    sorted copy (large ones): the same bits per point, also inside a captured graph."""
    import torch

    ensure_built()
    r = np.random.default_rng(n)
    x = r.uniform(-1.02, 1.02, (n, 3)).astype(np.float32)
    x = x[morton_order(x)]
    if n > 200:
        x[7] = [-1, -1, -1]
        x[8] = [1, 1, 1]
        x[9, 1] = np.nan
        x[10, 0] = np.inf
        x[11] = [3e38, -3e38, 3e38]
    perm = r.permutation(n)
    net = _model(shape, 2, 2 * n)
    xs = torch.as_tensor(np.concatenate([x, x[perm]]), device="cuda")
    a = net.forward(xs[:n].contiguous(), [0, n // 3, n])
    # the shuffle keeps each brick's points
    cut = n // 3
    p = np.concatenate([r.permutation(cut), cut + r.permutation(n - cut)])
    y = xs[:n][torch.as_tensor(p, device="cuda")].contiguous()
    b = net.forward(y, [0, cut, n])
    np.testing.assert_array_equal(a.cpu().numpy()[p], b.cpu().numpy())
    if n in (3000, 40_001):
        out = torch.zeros(n, device="cuda")
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            net.forward(y, [0, cut, n], out=out)
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(a.cpu().numpy()[p], out.cpu().numpy())


def test_sorted_queries_on_two_streams():
    """Both streams' queries go through the handle's one sorted copy, in turn."""
    import torch

    ensure_built()
    n = 200_003
    net = _model((32, 20, 2), 1, n)
    x = [torch.rand((n, 3), device="cuda") * 2 - 1 for _ in range(2)]
    want = [net.forward(v, [0, n]).clone() for v in x]
    torch.cuda.synchronize()
    s = [torch.cuda.Stream() for _ in range(2)]
    got = [[torch.empty(n, device="cuda") for _ in range(6)] for _ in range(2)]
    for k in range(6):
        for i in range(2):
            net.forward(x[i], [0, n], out=got[i][k], stream=s[i])
    torch.cuda.synchronize()
    for i in range(2):
        for k in range(6):
            assert torch.equal(got[i][k], want[i])


@pytest.mark.parametrize("shape", [(16, 9, 1), (32, 20, 2), (64, 32, 2)])
# (33, 2) and (129, 2): the shorter brick's last blocks are empty
@pytest.mark.parametrize("vox,grid", [(33, (2, 1, 1)), (50, (1, 1, 1)), (9, (2, 2, 2)), (129, (1, 1, 2))])
def test_decode_is_the_query_at_the_voxels(shape, vox, grid):
    import torch

    ensure_built()
    nb = grid[0] * grid[1] * grid[2]
    net = _model(shape, nb, vox ** 3)
    boxes, own, loc = [], [], []
    for k in range(grid[2]):
        for j in range(grid[1]):
            for i in range(grid[0]):
                w = [vox // g for g in grid]
                lo = [max(0, a * v - 1) for a, v in zip((i, j, k), w)]
                hi = [vox - 1 if a == g - 1 else min(vox - 1, a * v + v) for a, v, g in zip((i, j, k), w, grid)]
                boxes.append(lo + hi)
    got = net.decode(grid, np.array(boxes), vox).cpu().numpy()
    v = np.stack(np.meshgrid(*[np.arange(vox)] * 3, indexing="ij")[::-1], -1).reshape(-1, 3)   # x, y, z; x fastest
    own = np.zeros(len(v), dtype=np.int64)
    for a, m in ((0, 1), (1, grid[0]), (2, grid[0] * grid[1])):
        own += m * np.minimum(grid[a] * v[:, a] // (vox - 1), grid[a] - 1)
    order = np.argsort(own, kind="stable")
    off = [0] + list(np.cumsum(np.bincount(own, minlength=nb)))
    bx = np.array(boxes)[own]
    f32 = np.float32
    x = ((v.astype(f32) - bx[:, :3].astype(f32)) / (bx[:, 3:] - bx[:, :3]).astype(f32) * f32(2) - f32(1)).astype(f32)
    f = net.forward(torch.as_tensor(x[order], device="cuda"), [int(o) for o in off]).cpu().numpy()
    # (the device may fuse the last product and subtraction: a coordinate differs by an ulp)
    assert rel_l2(got.reshape(-1)[order], f) < 1e-3


@pytest.mark.parametrize("shape", [(16, 9, 1), (32, 20, 2), (64, 32, 2)])
@pytest.mark.parametrize("n", [32_768, 100_003])
@pytest.mark.parametrize("density", [False, True])
def test_training_batch_in_no_order(shape, n, density):
    """The gradients of a shuffled batch (through its sorted copy) and of the same points in
    bin order.  The two read Eq. 2 in two roundings, so a feature in 2^16 / 2 rounds to
    the neighbouring bfloat16 and flips its share of ReLU masks: the BF16 path's own
    tolerance bounds the gradients, and the losses agree to the features' rounding."""
    import torch

    ensure_built()
    r = np.random.default_rng(n)
    x = r.uniform(-1, 1, (n, 3)).astype(np.float32)
    t = r.uniform(0, 1, n).astype(np.float32)
    o = morton_order(x)
    net = _model(shape, 1, n)
    res = []
    for idx in (o, np.arange(n)):
        xs, ts = torch.as_tensor(x[idx], device="cuda"), torch.as_tensor(t[idx], device="cuda")
        losses = net.backward(xs, ts, [0, n], density=density).cpu().numpy().copy()
        res.append((losses, net.get("grads")[0]))
    net.status()
    (la, ga), (lb, gb) = res
    np.testing.assert_allclose(la, lb, rtol=1e-4)
    for k in ("F", "W1", "W2", "w3"):
        assert rel_l2(gb[k], ga[k]) < 2e-3, k
    if density:
        assert rel_l2(gb["G"], ga["G"]) < 2e-3


@pytest.mark.parametrize("ordered", [True, False])
def test_captured_backward_follows_its_batch(ordered):
    """A captured backward pass decides on the device, at each replay, whether the points
    then in its buffer need the sorted copy."""
    import torch

    ensure_built()
    n = 40_000
    r = np.random.default_rng(5)
    x = r.uniform(-1, 1, (n, 3)).astype(np.float32)
    t = r.uniform(0, 1, n).astype(np.float32)
    o = morton_order(x)
    first, then = (np.arange(n), o) if ordered else (o, np.arange(n))
    net = _model((32, 20, 2), 1, n)
    xs, ts = torch.as_tensor(x[first], device="cuda"), torch.as_tensor(t[first], device="cuda")
    net.backward(xs, ts, [0, n], density=True)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        net.backward(xs, ts, [0, n], density=True)
    xs.copy_(torch.as_tensor(x[then], device="cuda"))
    ts.copy_(torch.as_tensor(t[then], device="cuda"))
    g.replay()
    torch.cuda.synchronize()
    got, losses = net.get("grads")[0], net.losses.cpu().numpy().copy()
    want_l = net.backward(xs, ts, [0, n], density=True).cpu().numpy()
    want = net.get("grads")[0]
    np.testing.assert_allclose(losses, want_l, rtol=1e-6)
    for k in ("F", "W1", "W2", "w3", "G"):
        assert rel_l2(got[k], want[k]) < 1e-5, k
