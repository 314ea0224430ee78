"""The head at the sizes where its products are cut differently: odd class counts (no 16-byte rows), fewer rows
than a tile, several clusters per tile, and gradients in launches of their own; against 64 bits."""
import pytest
import torch

from gpu_common import check_status, load_dbl

pytestmark = pytest.mark.gpu

DTYPE = {"bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def D():
    return load_dbl()


def rel(a, b):
    return float((a.double() - b).norm() / b.norm())


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("n,hw,c,classes", [
    (3, 4, 64, 7),       # one tile, odd rows of classes
    (70, 1, 8, 3),       # a second row tile with six rows, eight features
    (1, 1, 512, 1001),   # one image, odd classes
    (5, 1, 2048, 1000),  # clusters that share the logits' reduction; the gradients apart
    (2, 1, 512, 9999),   # long sums over classes for two images
    (2100, 1, 64, 10),   # long sums over images for ten classes
    (8192, 1, 512, 10),  # the longest
])
def test_head_matches_64_bits(D, prec, n, hw, c, classes):
    gen = torch.Generator(device="cuda").manual_seed(n + classes)
    normal = lambda *s: torch.randn(s, device="cuda", generator=gen)
    x = normal(n, hw, c).abs().to(DTYPE[prec])
    w, b = 0.05 * normal(classes, c), 0.1 * normal(classes)
    lab = torch.randint(0, classes, (n,), device="cuda", dtype=torch.int32, generator=gen)
    loss, dw, db = (torch.full(s, float("nan"), device="cuda") for s in ((1,), (classes, c), (classes,)))
    dx = torch.full_like(x, float("nan"))
    scale = torch.tensor([1024.0], device="cuda")  # so that binary16 holds the gradients
    with D.precision(prec):
        wsb = D.dbl_head_workspace_bytes(n, c, classes)
        work = torch.full((wsb,), 255, dtype=torch.uint8, device="cuda")
        D.dbl_head_fwd_bwd_ex(n, hw, c, classes, x, w, b, lab, D.head_opts(loss_scale=scale), loss, dw, db, dx, work,
                              wsb)
        check_status(D)
    feat = x.double().mean(1)
    logits = feat @ w.double().T + b.double()
    lse = torch.logsumexp(logits, 1)
    row = torch.arange(n, device="cuda")
    dl = torch.softmax(logits, 1)
    dl[row, lab.long()] -= 1.0
    dl *= 1024.0 / n
    assert abs(float(loss) - float((lse - logits[row, lab.long()]).mean())) <= 1e-6 * float(lse.abs().max())
    # a sum in chunks of L terms loses about 2^-24 sqrt(L / 6) of its norm: 2.8e-7 at the longest chunks here,
    # 1e-6 and more in chunks of thousands; the logits' own error adds up to 2e-7
    assert rel(dw, dl.T @ feat) <= 5e-7 and rel(db, dl.sum(0)) <= 5e-7
    # one rounding to 16 bits (2^-9 of bf16 values, 2^-12 of f16 ones, whose small ones are subnormal)
    want = (dl @ w.double() / hw)[:, None].expand(n, hw, c)
    assert rel(dx, want) <= 2.0 ** -8
