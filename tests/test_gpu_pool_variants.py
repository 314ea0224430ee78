"""The stem's fused BatchNorm + ReLU + max pool on large tensors, where a thread walks a run of output rows,
against the two-step path, bit for bit."""
import pytest
import torch

from gpu_common import check_status, load_dbl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    return load_dbl()


@pytest.mark.parametrize("n,h,w,c", [
    (41, 141, 139, 64),   # odd sides: windows clipped on both, a last run of rows with fewer
    (300, 145, 150, 8),   # one channel group
    (11, 142, 141, 256),  # eight pixel pairs per CTA
    (3, 513, 515, 64),    # few, large images
])
def test_large_pool_equals_bn_then_maxpool(D, n, h, w, c):
    g = torch.Generator(device="cuda").manual_seed(n)
    y = torch.empty((n, h, w, c), device="cuda").normal_(0.3, 1.0, generator=g)
    y = (y * 2).round().div(2).to(torch.bfloat16)  # ties, and many zeros after the ReLU
    assert y.numel() * 2 >= 96 << 20
    gamma = torch.empty(c, device="cuda").uniform_(-1.5, 1.5, generator=g)
    beta = torch.empty(c, device="cuda").normal_(0.0, 0.3, generator=g)
    shape = D.bn_shape(n * h * w, c, 1e-5, True)
    s1, s2 = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
    D.dbl_bn_stats(shape, y, s1, s2)
    out, stats = torch.empty_like(y), [torch.empty(c, device="cuda") for _ in range(4)]
    p, q = (h - 1) // 2 + 1, (w - 1) // 2 + 1
    got = []
    for fused in (False, True):
        a = torch.full((n, p, q, c), float("nan"), dtype=torch.bfloat16, device="cuda")
        arg = torch.full((n, p, q, c), 255, dtype=torch.uint8, device="cuda")
        if fused:
            D.dbl_bn_relu_maxpool_fwd(shape, n, h, w, y, s1, s2, gamma, beta, stats[2], stats[3], a, arg)
        else:
            D.dbl_bn_relu_fused(shape, y, s1, s2, gamma, beta, None, out, stats[0], stats[1])
            D.dbl_maxpool_fwd(n, h, w, c, out, a, arg)
        got.append((a, arg))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    check_status(D)
