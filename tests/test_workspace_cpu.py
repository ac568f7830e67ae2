"""What a handle's workspace holds per point."""
import pytest

from gpu_util import ensure_built


@pytest.mark.parametrize("bf16,most", [(False, 36), (True, 36 + 4 * 128 + 20 + 4)])
def test_bytes_per_point(bf16, most):
    """Float32: rho, the squared error, the sampler's rank, a render's value (4 bytes each) and a query's
    sorted copy (20); BF16 also Y and dL/dy (2 bytes each of K), a training batch's copy (20) and, per
    kMinTilePoints points, tiles and maxima (under 4)."""
    ensure_built()
    from paper_2308_02494_gb300 import srn

    cfg = srn.Config(1, 64, 2, 32, 64, srn.SRN_BF16 if bf16 else srn.SRN_FP32, 10, 1e-8, 1e-2, 1e-3, 0.9, 0.99, 1e-8)
    n = (1 << 24, 1 << 26)
    a, b = (srn.srn_workspace_size(cfg, k) for k in n)
    assert (b - a) / (n[1] - n[0]) <= most
