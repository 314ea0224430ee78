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
    (161, 141, 142, 32),  # 64 pixel pairs per CTA
    (2700, 27, 27, 64),   # the fewest output rows
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


@pytest.mark.parametrize("n,h,w,c,two", [
    (1, 1, 1, 64, False),     # one pixel: the two passes
    (5, 51, 51, 64, True),    # the smallest general size: odd sides, partials with one block or none
    (3, 140, 71, 64, True),   # even and odd sides
    (2, 97, 200, 256, False),  # eight blocks per step
    (2, 41, 80, 1024, False),  # the most channels
    (1, 85, 80, 2048, False),  # the two passes
    (40, 60, 62, 8, True),    # one channel group
    (33, 112, 112, 64, True),  # several steps per thread
])
def test_pool_bn_backward_equals_two_steps(D, n, h, w, c, two):
    """da bit for bit; dx, dgamma and dbeta up to the order of the channel sums."""
    g = torch.Generator(device="cuda").manual_seed(n + h)
    normal = lambda *s: torch.empty(s, device="cuda").normal_(0.1, 1.0, generator=g)
    p, q = (h - 1) // 2 + 1, (w - 1) // 2 + 1
    x = normal(n, h, w, c).to(torch.bfloat16)
    dp, dp2 = normal(n, p, q, c).to(torch.bfloat16), normal(n, p, q, c).to(torch.bfloat16) if two else None
    gamma, beta = normal(c) + 1.0, normal(c)
    shape = D.bn_shape(n * h * w, c, 1e-5, True)
    s1, s2, mean, istd = (torch.empty(c, device="cuda") for _ in range(4))
    D.dbl_bn_stats(shape, x, s1, s2)
    pooled = torch.empty((n, p, q, c), dtype=torch.bfloat16, device="cuda")
    arg = torch.empty((n, p, q, c), dtype=torch.uint8, device="cuda")
    D.dbl_bn_relu_maxpool_fwd(shape, n, h, w, x, s1, s2, gamma, beta, mean, istd, pooled, arg)
    wsb = D.dbl_bn_workspace_bytes(shape)
    got = []
    for fused in (False, True):
        work = torch.full((wsb // 4,), float("nan"), device="cuda")
        da, dx = (torch.full((n, h, w, c), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        dg, db = (torch.full((c,), float("nan"), device="cuda") for _ in range(2))
        if fused:
            D.dbl_maxpool_bn_relu_bwd(shape, n, h, w, dp, dp2, arg, x, gamma, beta, mean, istd, da, dx, dg, db, work, wsb)
        else:
            D.dbl_maxpool_bwd(n, h, w, c, dp, dp2, arg, da)
            D.dbl_bn_relu_fused_bwd(shape, da, None, x, None, gamma, mean, istd, dx, None, dg, db, work, wsb, beta=beta)
        got.append((da, dx, dg, db))
    (da0, dx0, dg0, db0), (da1, dx1, dg1, db1) = got
    assert torch.equal(da0, da1)
    # fp32 sums of the same terms in two orders: chains of at most 2 * 33 * 112 * 112 / (256 * 32) additions per
    # thread and 32 more per partial lose at most 2 * (101 + 32) * 2^-24 of the sum of the terms' sizes
    m = da0.float().abs() * (x.float() - mean).mul(istd).abs().clamp(min=1.0)
    bound = 2 * 133 * 2.0 ** -24 * m.sum((0, 1, 2)) + 1e-30
    assert torch.all((dg0 - dg1).abs() <= bound) and torch.all((db0 - db1).abs() <= bound)
    # their share in dx is far below its rounding: half a unit of bf16 is at most 2^-8 of the value
    assert torch.all((dx0.float() - dx1.float()).abs() <= 2.0 ** -7 * dx0.float().abs() + 1e-5 * dx0.float().abs().max())
    check_status(D)


def test_pool_bn_backward_loses_no_more_than_two_steps(D):
    """dgamma and dbeta against 64 bits, over eight draws of 64 channels: the root mean square of the errors. (Of the
    same distribution in both forms, two such figures differ by less than 10% in 99 of 100 pairs.)"""
    n, h, w, c = 64, 64, 64, 64
    p, shape = h // 2, D.bn_shape(n * h * w, c, 1e-5, True)
    wsb = D.dbl_bn_workspace_bytes(shape)
    err = {False: 0.0, True: 0.0}
    for seed in range(8):
        g = torch.Generator(device="cuda").manual_seed(seed)
        normal = lambda *s: torch.empty(s, device="cuda").normal_(0.0, 1.0, generator=g)
        x, dp, dp2 = (normal(*s).to(torch.bfloat16) for s in ((n, h, w, c), (n, p, p, c), (n, p, p, c)))
        gamma, beta, mean, istd = normal(c).abs() + 0.5, 0.5 * normal(c), 0.1 * normal(c), normal(c).abs() + 0.5
        arg = torch.randint(0, 9, (n, p, p, c), device="cuda", dtype=torch.uint8, generator=g)
        for fused in (False, True):
            work, da, dx = torch.empty(wsb, dtype=torch.uint8, device="cuda"), torch.empty_like(x), torch.empty_like(x)
            dg, db = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
            if fused:
                D.dbl_maxpool_bn_relu_bwd(shape, n, h, w, dp, dp2, arg, x, gamma, beta, mean, istd, da, dx, dg, db, work,
                                          wsb)
            else:
                D.dbl_maxpool_bwd(n, h, w, c, dp, dp2, arg, da)
                D.dbl_bn_relu_fused_bwd(shape, da, None, x, None, gamma, mean, istd, dx, None, dg, db, work, wsb,
                                        beta=beta)
            sc = gamma * istd
            shift = (beta - mean * sc).double()  # the mask as the kernels decide it: one rounding of y * scale + shift
            gg = torch.where((x.double() * sc.double() + shift).float() > 0, da.double(), 0.0)
            xhat = (x.double() - mean.double()) * istd.double()
            scale = (gg * xhat).square().sum((0, 1, 2)).sqrt()
            err[fused] += float(((dg.double() - (gg * xhat).sum((0, 1, 2))) / scale).square().sum())
            err[fused] += float(((db.double() - gg.sum((0, 1, 2))) / scale).square().sum())
    assert err[True] <= 1.1 ** 2 * err[False]
    check_status(D)
