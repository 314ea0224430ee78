"""Edges of the one-launch BatchNorm passes of small tensors: the backward (a cluster of CTAs per 32
channels) against the fp64 oracle, the forward against the two launches of larger ones."""
from decimal import Context, Decimal

import numpy as np
import pytest
import torch

import oracle as orc
from conftest import max_norm_rel
from gpu_common import bf16_values, check_status, host, load_dbl, rng, to_bf16_dev, to_f32_dev, ws

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    return load_dbl()


@pytest.mark.parametrize("count,C", [
    (1, 512),      # one row: seven CTAs of a cluster have none
    (9, 64),       # fewer rows than CTAs
    (577, 256),    # a last CTA with fewer rows
    (4096, 512),   # the largest with g stored
    (6400, 512),   # the largest without
    (6401, 512),   # the general path
])
@pytest.mark.parametrize("mask", ["out", "y", "none"])
def test_small_bn_backward_matches_oracle(D, count, C, mask):
    """mask "out": with a second gradient and the masked gradient stored over it; "y": the mask from y."""
    g = rng(count + C)
    y = bf16_values(g.standard_normal((count, C)) * 2.0 + 0.5)
    gamma = (1.0 + 0.2 * g.standard_normal(C)).astype(np.float32)
    beta = (0.1 * g.standard_normal(C)).astype(np.float32)
    mean, istd = y.mean(0).astype(np.float32), (1.0 / np.sqrt(y.var(0) + 1e-5)).astype(np.float32)
    dout, dout2 = (bf16_values(g.standard_normal((count, C))) for _ in range(2))
    sc = gamma * istd  # the forward pass's fp32 operations
    pre = y.astype(np.float32) * sc + (beta - mean * sc)
    out = bf16_values(np.maximum(pre, 0.0)) if mask != "none" else bf16_values(pre)
    sure = np.abs(pre) > 1e-5  # elements whose mask a fused multiply-add cannot decide otherwise
    dout, dout2 = dout * sure, dout2 * sure
    two = mask == "out"
    shape = D.bn_shape(count, C, 1e-5, mask != "none")
    dy = torch.full((count, C), float("nan"), dtype=torch.bfloat16, device="cuda")
    dg, db = torch.full((C,), float("nan"), device="cuda"), torch.full((C,), float("nan"), device="cuda")
    d2 = to_bf16_dev(dout2) if two else None
    wsb = D.dbl_bn_workspace_bytes(shape)
    D.dbl_bn_relu_fused_bwd(shape, to_bf16_dev(dout), d2, to_bf16_dev(y), to_bf16_dev(out) if two else None,
                            to_f32_dev(gamma), to_f32_dev(mean), to_f32_dev(istd), dy, d2, dg, db, ws(wsb), wsb,
                            beta=to_f32_dev(beta))
    rdy, rdg, rdb, rres = orc.bn_bwd(dout, out, y, gamma, mean.astype(np.float64), istd.astype(np.float64),
                                     relu=mask != "none", dout2=dout2 if two else None, want_dres=True)
    # dy = A*(g - ...), A = gamma/std: g rounded to bf16 where it is stored (bf16 has 8 significant bits:
    # half a unit is at most 2^-8 of the value) and dy once more, 2^-7 together; of a single row the exact
    # dy is 0 and A is 316
    scale = max(np.abs(rdy).max(), np.abs(gamma * istd).max() * np.abs(rres).max())
    assert np.abs(host(dy) - rdy).max() <= 2.0 ** -7 * scale
    for got, ref in ((dg, rdg), (db, rdb)):
        assert np.abs(host(got) - ref).max() <= 1e-5 * (np.abs(rres).sum(0).max() * 4)
    if two:
        assert max_norm_rel(host(d2), rres) <= 4e-3
    check_status(D)


@pytest.mark.parametrize("count,C,nparts", [
    (1, 32, 1),        # one row, one partial
    (63, 512, 33),     # fewer rows than a CTA covers; a second round of a stream
    (4099, 256, 104),  # the most partials; a ragged last run of rows
    (8192, 512, 7),    # the largest tensor
])
@pytest.mark.parametrize("residual", [False, True])
def test_one_launch_bn_forward_gives_the_same_bits(D, count, C, nparts, residual):
    """Partial rows of zeros leave the sums as they are and take the call to the two-launch path."""
    g = rng(count)
    y = to_bf16_dev(g.standard_normal((count, C)) + 0.5)
    res = to_bf16_dev(g.standard_normal((count, C))) if residual else None
    gamma, beta = to_f32_dev(1.0 + 0.2 * g.standard_normal(C)), to_f32_dev(0.1 * g.standard_normal(C))
    parts = np.zeros((160, 2, C), dtype=np.float32)
    w = g.random((nparts, 1, C)).astype(np.float32)
    parts[:nparts, :1] = 0.5 * count * w / w.sum(0)
    parts[:nparts, 1:] = 1.25 * count * w / w.sum(0)
    pd = to_f32_dev(parts)
    got = []
    for n in (nparts, 160):
        out = torch.full((count, C), float("nan"), dtype=torch.bfloat16, device="cuda")
        mean, istd = torch.full((C,), float("nan"), device="cuda"), torch.full((C,), float("nan"), device="cuda")
        D.dbl_bn_relu_fused_parts(D.bn_shape(count, C, 1e-5, True), y, pd, n, gamma, beta, res, out, mean, istd)
        got.append((out, mean, istd))
    assert all(torch.isfinite(t.float()).all() for t in got[0])
    assert all(torch.equal(a, b) for a, b in zip(*got))
    check_status(D)


@pytest.mark.parametrize("nparts", [8, 160])  # one launch, and two
def test_channel_sums_keep_what_fp64_keeps(D, nparts):
    """Partial rows whose tree needs all 53 bits of fp64: 1, 2^-25, 2^-52, 0, -1, -2^-25 leave 2^-52 (and the
    sums of the backward's clusters, added in rank order, the same)."""
    C, count = 32, 4
    parts = torch.zeros((nparts, 2, C), device="cuda")
    parts[:6, 0] = torch.tensor([1.0, 2.0 ** -25, 2.0 ** -52, 0.0, -1.0, -2.0 ** -25], device="cuda")[:, None]
    parts[0, 1] = count
    y = torch.zeros((count, C), dtype=torch.bfloat16, device="cuda")
    out, (mean, istd) = torch.empty_like(y), torch.full((2, C), float("nan"), device="cuda")
    gamma, beta = torch.ones(C, device="cuda"), torch.zeros(C, device="cuda")
    D.dbl_bn_relu_fused_parts(D.bn_shape(count, C, 1e-5, True), y, parts, nparts, gamma, beta, None, out, mean, istd)
    assert torch.equal(mean, torch.full_like(mean, 2.0 ** -54))
    rows = torch.zeros((16, C), dtype=torch.bfloat16, device="cuda")  # one per CTA of a cluster
    rows[:5] = torch.tensor([1.0, 2.0 ** -25, 2.0 ** -52, -1.0, -2.0 ** -25], device="cuda")[:, None]
    shape = D.bn_shape(16, C, 1e-5, False)
    wsb = D.dbl_bn_workspace_bytes(shape)
    dg, db = torch.full((2, C), float("nan"), device="cuda")
    D.dbl_bn_relu_fused_bwd(shape, rows, None, torch.zeros_like(rows), None, gamma, beta, gamma,
                            torch.empty_like(rows), None, dg, db, ws(wsb), wsb)
    assert torch.equal(db, torch.full_like(db, 2.0 ** -52))
    check_status(D)


@pytest.mark.parametrize("nparts", [8, 160])
def test_channel_sums_beyond_fp32_are_infinite(D, nparts):
    """Finite partials whose sum fp32 cannot hold: the variance is infinite, 1/std zero and the output beta."""
    C, count = 32, 4
    parts = torch.zeros((nparts, 2, C), device="cuda")
    parts[:3, 1] = 3e38
    y = torch.ones((count, C), dtype=torch.bfloat16, device="cuda")
    out, (mean, istd) = torch.empty_like(y), torch.full((2, C), float("nan"), device="cuda")
    gamma, beta = torch.ones(C, device="cuda"), torch.full((C,), 0.5, device="cuda")
    D.dbl_bn_relu_fused_parts(D.bn_shape(count, C, 1e-5, True), y, parts, nparts, gamma, beta, None, out, mean, istd)
    assert torch.equal(istd, torch.zeros_like(istd)) and torch.equal(mean, torch.zeros_like(mean))
    assert torch.equal(out, torch.full_like(out, 0.5))
    check_status(D)


@pytest.mark.parametrize("C", [16, 32])  # two launches, and one
def test_inverse_std_rounds_like_fp64(D, C):
    """Sums of squares over three rows (fp32 bit patterns) whose 1/std lies above the middle of two fp32 values
    by 2^-50 to 2^-47 of it: fp64's 1/sqrt (wrong by at most 2^-52) decides the rounding, less does not."""
    bits = [1072431535, 1085111321, 1111793036, 1124728303, 1134414601, 1154234959, 1168073971, 1170294655,
            1174906697, 1180708072]
    sq = np.resize(np.array(bits, dtype=np.uint32), C).view(np.float32)
    exact = [Decimal(float(q) * (1.0 / 3) + float(np.float32(1e-5))).sqrt(Context(prec=50)) for q in sq]
    want = []
    for e in exact:
        f = np.float32(1 / float(e))
        near = [np.nextafter(f, np.float32(0)), f, np.nextafter(f, np.float32(9))]
        want.append(min(near, key=lambda t: abs(Decimal(float(t)) * e - 1)))
    parts = torch.zeros((1, 2, C), device="cuda")
    parts[0, 1] = to_f32_dev(sq)
    y = torch.zeros((3, C), dtype=torch.bfloat16, device="cuda")
    mean, istd = torch.full((2, C), float("nan"), device="cuda")
    D.dbl_bn_relu_fused_parts(D.bn_shape(3, C, 1e-5, True), y, parts, 1, torch.ones(C, device="cuda"),
                              torch.zeros(C, device="cuda"), None, torch.empty_like(y), mean, istd)
    assert np.array_equal(istd.cpu().numpy(), np.array(want))
    check_status(D)
