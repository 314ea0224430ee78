"""The kernels chosen by shape in the binary16 build, whose packed conversions, comparisons and maxima are other
instructions than bfloat16's: each once at an awkward size, against 64 bits or the path it replaces."""
import pytest
import torch

from gpu_common import check_status, load_dbl, ws

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    dbl = load_dbl()
    with dbl.precision("f16"):
        yield dbl


def gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def normal(g, *s):
    return torch.randn(s, device="cuda", generator=g)


def max_rel(a, b):
    return float((a.double() - b).abs().max() / b.abs().max())


def conv64(x, w, stride, pad_h, pad_w):
    x = torch.nn.functional.pad(x.double(), (0, 0, pad_w, pad_w, pad_h, pad_h))
    k, r, s, c = w.shape
    p, q = (x.shape[1] - r) // stride + 1, (x.shape[2] - s) // stride + 1
    y = torch.zeros((x.shape[0], p, q, k), dtype=torch.float64, device="cuda")
    for a in range(r):
        for b in range(s):
            y += x[:, a:a + stride * p:stride, b:b + stride * q:stride] @ w[:, a, b].double().T
    return y


def dgrad64(dy, w, x_shape, stride, pad):
    n, h, wd, c = x_shape
    k, r, s, _ = w.shape
    dx = torch.zeros((n, h + 2 * pad, wd + 2 * pad, c), dtype=torch.float64, device="cuda")
    p, q = dy.shape[1:3]
    for a in range(r):
        for b in range(s):
            dx[:, a:a + stride * p:stride, b:b + stride * q:stride] += dy.double() @ w[:, a, b].double()
    return dx[:, pad:pad + h, pad:pad + wd]


def wgrad64(x, dy, r, s, stride, pad_h, pad_w):
    x = torch.nn.functional.pad(x.double(), (0, 0, pad_w, pad_w, pad_h, pad_h))
    p, q, k = dy.shape[1:]
    d2 = dy.double().reshape(-1, k)
    return torch.stack([torch.stack([d2.T @ x[:, a:a + stride * p:stride, b:b + stride * q:stride].reshape(-1, x.shape[3])
                                     for b in range(s)], 1) for a in range(r)], 1)


OUT_TOL = 2.0 ** -10  # one rounding to 11 bits is 2^-12 to 2^-11 of the value; and the fp32 sums
WGRAD_TOL = 1e-5  # fp32 sums of exact products


@pytest.mark.parametrize("n,h,w,c,k,stride", [
    (3, 5, 10, 64, 64, 1),    # pixel pairs
    (2, 7, 9, 64, 64, 1),     # odd width: the window kernel
    (29, 3, 3, 512, 512, 1),  # tiles split over pairs
    (9, 8, 8, 256, 512, 2),
    (5, 10, 10, 128, 128, 1),  # window pairs of 128 columns
])
def test_conv_forward_and_data_gradient(D, n, h, w, c, k, stride):
    g = gen(n + h)
    x, wt = normal(g, n, h, w, c).half(), (normal(g, k, 3, 3, c) * (2.0 / (9 * c)) ** 0.5).half()
    shape = D.conv_shape(n, h, w, c, k, 3, stride, 1)
    y = torch.full((n, (h - 1) // stride + 1, (w - 1) // stride + 1, k), float("nan"), dtype=torch.float16, device="cuda")
    s1, s2 = torch.empty(k, device="cuda"), torch.empty(k, device="cuda")
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_FWD)
    D.dbl_conv_fwd(shape, x, wt, y, s1, s2, ws(wsb), wsb)
    assert max_rel(y, conv64(x, wt, stride, 1, 1)) <= OUT_TOL
    rows = y.double().reshape(-1, k)
    assert float((s1.double() - rows.sum(0)).abs().max() / rows.abs().sum(0).max()) <= 1e-5
    assert max_rel(s2, rows.square().sum(0)) <= 1e-5
    dy = normal(g, *y.shape).half()
    dx = torch.full_like(x, float("nan"))
    D.dbl_conv_dgrad(shape, dy, wt, dx)
    assert max_rel(dx, dgrad64(dy, wt, x.shape, stride, 1)) <= OUT_TOL
    check_status(D)


@pytest.mark.parametrize("n,h,w,c,k,r,s,stride,pad_h,pad_w", [
    (3, 13, 21, 64, 64, 3, 3, 1, 1, 1),      # rows
    (2, 9, 70, 64, 64, 4, 1, 1, 0, 0),       # bands
    (3, 14, 37, 64, 64, 3, 1, 1, 1, 0),      # bands, three taps
    (2, 9, 20, 64, 64, 5, 2, 1, 0, 0),       # window
    (220, 23, 26, 128, 128, 3, 3, 1, 1, 1),  # filter rows
    (33, 5, 5, 256, 128, 3, 3, 1, 1, 1),     # split tiles of 128 columns
    (17, 14, 14, 128, 256, 3, 3, 2, 1, 1),   # and of 256
])
def test_weight_gradient(D, n, h, w, c, k, r, s, stride, pad_h, pad_w):
    g = gen(n + w)
    p, q = (h + 2 * pad_h - r) // stride + 1, (w + 2 * pad_w - s) // stride + 1
    x, dy = normal(g, n, h, w, c).half(), normal(g, n, p, q, k).half()
    shape = D.conv_shape(n, h, w, c, k, r, stride, pad_h, s=s, stride_w=stride, pad_w=pad_w)
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_WGRAD)
    dw = torch.full((k, r, s, c), float("nan"), device="cuda")
    D.dbl_conv_wgrad(shape, x, dy, dw, False, ws(wsb), wsb)
    # sums over up to 130,000 positions in chains of up to 3,000: 190 steps that each cut 2^-24 of their partial sum
    assert max_rel(dw, wgrad64(x, dy, r, s, stride, pad_h, pad_w)) <= WGRAD_TOL
    check_status(D)


def test_batchnorm_in_one_launch(D):
    """Forward as in two launches, bit for bit; backward against 64 bits."""
    count, C = 577, 256
    g = gen(1)
    y, res = (normal(g, count, C) * 2.0 + 0.5).half(), normal(g, count, C).half()
    gamma, beta = 1.0 + 0.2 * normal(g, C), 0.1 * normal(g, C)
    parts = torch.zeros((160, 2, C), device="cuda")
    parts[:, 0], parts[:, 1] = y.float().sum(0) / 16, y.float().square().sum(0) / 16
    parts[16:] = 0.0
    shape, got = D.bn_shape(count, C, 1e-5, True), []
    for n in (16, 160):
        out, st = torch.full_like(y, float("nan")), torch.full((2, C), float("nan"), device="cuda")
        D.dbl_bn_relu_fused_parts(shape, y, parts, n, gamma, beta, res, out, st[0], st[1])
        got.append((out, st))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    out, (mean, istd) = got[0][0], got[0][1].double()
    xhat = (y.double() - mean) * istd
    assert max_rel(out, torch.relu(xhat * gamma.double() + beta.double() + res.double())) <= OUT_TOL
    dout = normal(g, count, C).half()
    dy, dres = torch.full_like(y, float("nan")), torch.full_like(y, float("nan"))
    dg, db = torch.empty(C, device="cuda"), torch.empty(C, device="cuda")
    wsb = D.dbl_bn_workspace_bytes(shape)
    D.dbl_bn_relu_fused_bwd(shape, dout, None, y, out, gamma, got[0][1][0], got[0][1][1], dy, dres, dg, db, ws(wsb), wsb)
    gg = torch.where(out > 0, dout.double(), 0.0)
    assert torch.equal(dres.double(), gg)
    assert max_rel(dg, (gg * xhat).sum(0)) <= 1e-5 and max_rel(db, gg.sum(0)) <= 1e-5
    want = gamma.double() * istd * (gg - gg.mean(0) - xhat * (gg * xhat).mean(0))
    assert max_rel(dy, want) <= OUT_TOL
    check_status(D)


def test_stem_pool(D):
    """Forward by rows as the two steps, bit for bit; backward's pooled gradient too, its sums against theirs."""
    n, h, w, c = 41, 141, 139, 64
    g = gen(2)
    x = (normal(g, n, h, w, c) * 2 + 0.6).round().div(2).half()
    gamma, beta = normal(g, c), 0.3 * normal(g, c)
    shape = D.bn_shape(n * h * w, c, 1e-5, True)
    s1, s2 = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
    D.dbl_bn_stats(shape, x, s1, s2)
    p, q = (h + 1) // 2, (w + 1) // 2
    st = torch.empty((4, c), device="cuda")
    a, b = (torch.full((n, p, q, c), float("nan"), dtype=torch.float16, device="cuda") for _ in range(2))
    ia, ib = (torch.full((n, p, q, c), 255, dtype=torch.uint8, device="cuda") for _ in range(2))
    out = torch.empty_like(x)
    D.dbl_bn_relu_fused(shape, x, s1, s2, gamma, beta, None, out, st[0], st[1])
    D.dbl_maxpool_fwd(n, h, w, c, out, a, ia)
    D.dbl_bn_relu_maxpool_fwd(shape, n, h, w, x, s1, s2, gamma, beta, st[2], st[3], b, ib)
    assert torch.equal(a, b) and torch.equal(ia, ib)
    dp, dp2 = normal(g, n, p, q, c).half(), normal(g, n, p, q, c).half()
    wsb, got = D.dbl_bn_workspace_bytes(shape), []
    for fused in (False, True):
        da, dx = torch.full_like(x, float("nan")), torch.full_like(x, float("nan"))
        dg, db = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
        if fused:
            D.dbl_maxpool_bn_relu_bwd(shape, n, h, w, dp, dp2, ia, x, gamma, beta, st[0], st[1], da, dx, dg, db, ws(wsb),
                                      wsb)
        else:
            D.dbl_maxpool_bwd(n, h, w, c, dp, dp2, ia, da)
            D.dbl_bn_relu_fused_bwd(shape, da, None, x, None, gamma, st[0], st[1], dx, None, dg, db, ws(wsb), wsb,
                                    beta=beta)
        got.append((da, dx, dg, db))
    (da0, dx0, dg0, db0), (da1, dx1, dg1, db1) = got
    assert torch.equal(da0, da1)
    size = (da0.float().abs() * ((x.float() - st[0]) * st[1]).abs().clamp(min=1.0)).sum((0, 1, 2))
    bound = 200 * 2.0 ** -24 * size  # chains of at most 90 additions and 32 more, in both orders
    assert torch.all((dg0 - dg1).abs() <= bound) and torch.all((db0 - db1).abs() <= bound)
    assert float((dx0.float() - dx1.float()).abs().max() / dx0.float().abs().max()) <= OUT_TOL
    check_status(D)
