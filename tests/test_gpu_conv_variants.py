"""Edges of the convolution kernels chosen by shape: row-block weight gradients (3x3 stride 1, 64
channels) and tiles split over clusters of CTA pairs, against the fp64 oracle."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle as orc
from conftest import max_norm_rel
from gpu_common import bf16_values, check_status, host, load_dbl, rng, to_bf16_dev, ws

pytestmark = pytest.mark.gpu

# products of two bf16 values are exact in fp32, so the error is that of fp32 sums: n terms of equal
# size in a row lose about sqrt(n) * 2^-24 of their norm, 4e-6 at the 4,500 positions used here
WGRAD_TOL = 1e-5


@pytest.fixture(scope="module")
def D():
    return load_dbl()


@pytest.mark.parametrize("n,h,w,pad", [
    (1, 1, 30, 1),     # one K-block: a single slice, written straight into dw
    (1, 8, 8, 1),      # the narrowest rows, padded to a pitch of 16
    (3, 13, 21, 1),    # rows padded to the pitch, a last K-block past the image
    (2, 17, 12, 0),    # no padding
    (2, 9, 20, 2),     # padding of two
    (64, 8, 14, 1),    # several rows per K-block
    (1, 3, 206, 1),    # the widest rows
])
def test_row_block_wgrad_matches_oracle(D, n, h, w, pad):
    g = rng(1000 * n + w)
    x = bf16_values(g.standard_normal((n, h, w, 64)))
    dy = bf16_values(g.standard_normal((n, h + 2 * pad - 2, w + 2 * pad - 2, 64)))
    ref = orc.conv2d_wgrad(x, dy, (64, 3, 3, 64), 1, pad)
    shape = D.conv_shape(n, h, w, 64, 64, 3, 1, pad)
    assert D.dbl_conv_plan(shape, D.DBL_PASS_WGRAD).kernel == D.DBL_KERNEL_WINDOW_WGRAD
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_WGRAD)

    dw = torch.full((64, 3, 3, 64), float("nan"), device="cuda")
    work, xd, dyd = ws(wsb), to_bf16_dev(x), to_bf16_dev(dy)
    D.dbl_conv_wgrad(shape, xd, dyd, dw, False, work, wsb)
    assert np.all(np.isfinite(host(dw)))
    assert max_norm_rel(host(dw), ref) <= WGRAD_TOL
    D.dbl_conv_wgrad(shape, xd, dyd, dw, True, work, wsb)
    assert max_norm_rel(host(dw), 2 * ref) <= WGRAD_TOL
    check_status(D)


@pytest.mark.parametrize("n,h,w,r,ph", [
    (1, 4, 16, 4, 0),    # one output row, one K-block's width
    (1, 5, 1, 4, 0),     # the narrowest rows
    (2, 9, 70, 4, 0),    # a last band past the image
    (3, 14, 37, 3, 1),   # odd widths, padded rows, the unused half of three taps
    (1, 40, 23, 3, 0),   # a last block of rows past the image
    (2, 7, 256, 4, 2),   # the widest rows that one band could hold
    (1, 4, 300, 3, 1),   # wider than any band
    (64, 35, 32, 4, 0),  # several K-blocks per CTA
])
def test_band_wgrad_matches_oracle(D, n, h, w, r, ph):
    g = rng(1000 * n + w)
    x = bf16_values(g.standard_normal((n, h, w, 64)))
    p = h + 2 * ph - r + 1
    dy = bf16_values(g.standard_normal((n, p, w, 64)))
    xp = np.pad(x.astype(np.float64), ((0, 0), (ph, ph), (0, 0), (0, 0)))
    d2 = dy.astype(np.float64).reshape(-1, 64)
    ref = np.stack([d2.T @ xp[:, t:t + p].reshape(-1, 64) for t in range(r)], axis=1)[:, :, None]
    shape = D.conv_shape(n, h, w, 64, 64, r, 1, ph, s=1, stride_w=1, pad_w=0)
    assert D.dbl_conv_plan(shape, D.DBL_PASS_WGRAD).kernel == D.DBL_KERNEL_WINDOW_WGRAD
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_WGRAD)
    dw = torch.full((64, r, 1, 64), float("nan"), device="cuda")
    work, xd, dyd = ws(wsb), to_bf16_dev(x), to_bf16_dev(dy)
    D.dbl_conv_wgrad(shape, xd, dyd, dw, False, work, wsb)
    assert np.all(np.isfinite(host(dw)))
    assert max_norm_rel(host(dw), ref) <= WGRAD_TOL
    D.dbl_conv_wgrad(shape, xd, dyd, dw, True, work, wsb)
    assert max_norm_rel(host(dw), 2 * ref) <= WGRAD_TOL
    check_status(D)


@pytest.mark.parametrize("n,h,w,r,k", [
    (3, 14, 37, 2, 5),   # ten taps
    (2, 9, 20, 5, 2),
    (40, 24, 24, 5, 2),  # several K-blocks per CTA
    (1, 4, 13, 1, 3),    # three taps: the unused half of the last pair
    (2, 5, 10, 2, 2),    # the narrowest rows
])
def test_window_wgrad_of_other_filters_matches_oracle(D, n, h, w, r, k):
    g = rng(10 * n + w)
    x = bf16_values(g.standard_normal((n, h, w, 64)))
    p, q = h - r + 1, w - k + 1
    dy = bf16_values(g.standard_normal((n, p, q, 64)))
    d2 = dy.reshape(-1, 64)
    ref = np.stack([np.stack([d2.T @ x[:, a:a + p, b:b + q].reshape(-1, 64) for b in range(k)], axis=1)
                    for a in range(r)], axis=1)
    shape = D.conv_shape(n, h, w, 64, 64, r, 1, 0, s=k)
    assert D.dbl_conv_plan(shape, D.DBL_PASS_WGRAD).kernel == D.DBL_KERNEL_WINDOW_WGRAD
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_WGRAD)
    dw = torch.full((64, r, k, 64), float("nan"), device="cuda")
    D.dbl_conv_wgrad(shape, to_bf16_dev(x), to_bf16_dev(dy), dw, False, ws(wsb), wsb)
    assert np.all(np.isfinite(host(dw)))
    assert max_norm_rel(host(dw), ref) <= WGRAD_TOL
    check_status(D)


# 16-bit outputs: one rounding of the result, at most 2^-8 of its size (bf16), and the fp32 sums' error
CONV_TOL = 4e-3


def _conv_case(D, n, h, c, k, r, stride, pad, seed):
    g = rng(seed)
    x = bf16_values(g.standard_normal((n, h, h, c)))
    wt = bf16_values(g.standard_normal((k, r, r, c)) * np.sqrt(2.0 / (r * r * c)))
    p = (h + 2 * pad - r) // stride + 1
    return D.conv_shape(n, h, h, c, k, r, stride, pad), x, wt, p


@pytest.mark.parametrize("n,h,c,k,r,stride,pad,pairs,dgrad_pairs", [
    (1, 3, 512, 512, 3, 1, 1, 8, 8),     # 9 rows in a 256-row tile: eight pairs per tile
    (29, 3, 512, 512, 3, 1, 1, 8, 8),    # 261 rows: a second tile with five rows, all of rank 1's beyond the batch
    (100, 3, 512, 512, 3, 1, 1, 4, 4),   # 8 tiles: four pairs per tile
    (65, 8, 256, 512, 3, 2, 1, 4, 2),    # ragged batch, two column tiles
    (500, 3, 512, 512, 3, 1, 1, 2, 2),   # 36 tiles: two pairs per tile
    (32, 6, 256, 256, 1, 2, 0, 2, 2),    # a short reduction: two K-blocks a pair
    (32, 6, 128, 256, 1, 2, 0, 1, None),  # two K-blocks: not split
])
def test_split_conv_matches_oracle(D, n, h, c, k, r, stride, pad, pairs, dgrad_pairs):
    """Forward (with its channel sums) and data gradient of layers with few 256-column tiles."""
    shape, x, wt, p = _conv_case(D, n, h, c, k, r, stride, pad, n + h)
    for pss, want in ((D.DBL_PASS_FWD, pairs), (D.DBL_PASS_DGRAD, dgrad_pairs)):
        info = D.dbl_conv_plan(shape, pss)
        assert want is None or (info.kernel == D.DBL_KERNEL_IGEMM and info.grid == 2 * want * info.tiles)
    xd, wd = to_bf16_dev(x), to_bf16_dev(wt)
    y = torch.full((n, p, p, k), float("nan"), dtype=torch.bfloat16, device="cuda")
    s1, s2 = torch.empty(k, device="cuda"), torch.empty(k, device="cuda")
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_FWD)
    D.dbl_conv_fwd(shape, xd, wd, y, s1, s2, ws(wsb), wsb)
    ref = orc.conv2d_fwd(x, wt, stride, pad)
    assert np.all(np.isfinite(host(y)))
    assert max_norm_rel(host(y), ref) <= CONV_TOL
    rows = host(y).reshape(-1, k)  # the statistics are those of the stored values, summed in fp32
    assert max_norm_rel(host(s1), rows.sum(0)) <= 1e-4
    assert max_norm_rel(host(s2), (rows * rows).sum(0)) <= 1e-5
    if r == 3:
        dy = bf16_values(rng(n).standard_normal((n, p, p, k)))
        dx = torch.full((n, h, h, c), float("nan"), dtype=torch.bfloat16, device="cuda")
        D.dbl_conv_dgrad(shape, to_bf16_dev(dy), wd, dx)
        assert np.all(np.isfinite(host(dx)))
        assert max_norm_rel(host(dx), orc.conv2d_dgrad(dy, wt, x.shape, stride, pad)) <= CONV_TOL
    check_status(D)


@pytest.mark.parametrize("n,h,w,c,k,pad", [
    (220, 23, 26, 128, 128, 1),  # a ragged last block of every image
    (700, 12, 12, 128, 128, 1),  # the twelve rows of one image per block
    (1500, 8, 14, 128, 128, 0),  # whole small images per block, no padding, the last block past the batch
    (40, 30, 62, 128, 128, 2),   # padding of two
    (160, 14, 30, 256, 128, 1),  # two input-channel blocks
    (160, 14, 30, 128, 256, 1),  # two output-channel blocks
    (64, 20, 102, 128, 128, 1),  # one wide row per block
])
def test_filter_row_wgrad_matches_oracle(D, n, h, w, c, k, pad):
    g = rng(1000 * n + w)
    p, q = h + 2 * pad - 2, w + 2 * pad - 2
    # the oracle's loops are too slow for these sizes: gradients at 24 outputs, the tensor's corners among
    # them, of which x and dy are nonzero everywhere
    x = bf16_values(g.standard_normal((n, h, w, c), dtype=np.float32))
    dy = bf16_values(g.standard_normal((n, p, q, k), dtype=np.float32))
    at = [(0, 0, 0, 0), (k - 1, 2, 2, c - 1), (0, 2, 0, c - 1), (k - 1, 0, 2, 0)]
    at += [tuple(int(g.integers(0, m)) for m in (k, 3, 3, c)) for _ in range(20)]
    ref = np.array([orc.conv2d_wgrad_at(x, dy, (k, 3, 3, c), 1, pad, *i) for i in at])
    shape = D.conv_shape(n, h, w, c, k, 3, 1, pad)
    info = D.dbl_conv_plan(shape, D.DBL_PASS_WGRAD)
    assert info.kernel == D.DBL_KERNEL_WINDOW_WGRAD and info.tile_cols == 128
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_WGRAD)
    dw = torch.full((k, 3, 3, c), float("nan"), device="cuda")
    work, xd, dyd = ws(wsb), to_bf16_dev(x), to_bf16_dev(dy)
    D.dbl_conv_wgrad(shape, xd, dyd, dw, False, work, wsb)
    got = host(dw)
    assert np.all(np.isfinite(got))
    # each of a CTA's accumulation steps (16 positions; at most ~250 here) may lose 2^-24 of its partial sum
    # by rounding towards zero, all of them the same way
    assert np.abs(np.array([got[i] for i in at]) - ref).max() <= 250 * 2.0 ** -24 * np.abs(ref).max()
    D.dbl_conv_wgrad(shape, xd, dyd, dw, True, work, wsb)
    assert np.abs(host(dw) - 2 * got).max() <= 2.0 ** -22 * np.abs(got).max()
    check_status(D)


@pytest.mark.parametrize("n,h,w", [
    (1, 1, 8),       # the narrowest rows
    (3, 5, 10),      # tiles spanning small images
    (2, 9, 98),      # the widest rows
    (2, 7, 100),     # wider: the window kernel without pixel pairs
    (5, 13, 22),     # a ragged last tile
])
def test_pixel_pair_conv_matches_oracle(D, n, h, w):
    """64 to 64 channels, 3x3 stride 1: forward with its channel sums, and the data gradient."""
    g = rng(n * h + w)
    x = bf16_values(g.standard_normal((n, h, w, 64)))
    wt = bf16_values(g.standard_normal((64, 3, 3, 64)) * np.sqrt(2.0 / 576))
    shape = D.conv_shape(n, h, w, 64, 64, 3, 1, 1)
    xd, wd = to_bf16_dev(x), to_bf16_dev(wt)
    y = torch.full((n, h, w, 64), float("nan"), dtype=torch.bfloat16, device="cuda")
    s1, s2 = torch.empty(64, device="cuda"), torch.empty(64, device="cuda")
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_FWD)
    D.dbl_conv_fwd(shape, xd, wd, y, s1, s2, ws(wsb), wsb)
    assert np.all(np.isfinite(host(y)))
    assert max_norm_rel(host(y), orc.conv2d_fwd(x, wt, 1, 1)) <= CONV_TOL
    rows = host(y).reshape(-1, 64)
    assert np.abs(host(s1) - rows.sum(0)).max() <= 1e-5 * np.abs(rows).sum(0).max()
    assert max_norm_rel(host(s2), (rows * rows).sum(0)) <= 1e-5
    dy = bf16_values(rng(n).standard_normal((n, h, w, 64)))
    dx = torch.full((n, h, w, 64), float("nan"), dtype=torch.bfloat16, device="cuda")
    D.dbl_conv_dgrad(shape, to_bf16_dev(dy), wd, dx)
    assert np.all(np.isfinite(host(dx)))
    assert max_norm_rel(host(dx), orc.conv2d_dgrad(dy, wt, x.shape, 1, 1)) <= CONV_TOL
    check_status(D)


@pytest.mark.parametrize("n,h,c,k,r,stride,pairs,slices", [
    (33, 14, 64, 128, 3, 2, 2, 7),   # 128 columns, two pairs per tile, seven slices; a last row tile of 64
    (33, 5, 256, 128, 3, 1, 4, 1),   # 128 columns, four pairs, no slices: written straight into dw
    (65, 3, 512, 512, 3, 1, 2, 1),   # 256 columns, two pairs of three and two K-blocks
    (65, 14, 256, 512, 1, 2, 4, 7),  # four pairs, seven slices, pairs without a K-block
    (17, 14, 128, 256, 3, 2, 8, 1),  # eight pairs
])
def test_split_wgrad_matches_oracle(D, n, h, c, k, r, stride, pairs, slices):
    """Weight gradients whose tiles are shared by clusters of CTA pairs."""
    pad = 1 if r == 3 else 0
    shape, x, wt, p = _conv_case(D, n, h, c, k, r, stride, pad, n + c)
    info = D.dbl_conv_plan(shape, D.DBL_PASS_WGRAD)
    assert info.kernel == D.DBL_KERNEL_IGEMM and info.zdim == slices and info.grid == 2 * pairs * info.tiles
    dy = bf16_values(rng(n).standard_normal((n, p, p, k)))
    ref = orc.conv2d_wgrad(x, dy, wt.shape, stride, pad)
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_WGRAD)
    dw = torch.full((k, r, r, c), float("nan"), device="cuda")
    work, xd, dyd = ws(wsb), to_bf16_dev(x), to_bf16_dev(dy)
    D.dbl_conv_wgrad(shape, xd, dyd, dw, False, work, wsb)
    assert np.all(np.isfinite(host(dw)))
    assert max_norm_rel(host(dw), ref) <= WGRAD_TOL
    D.dbl_conv_wgrad(shape, xd, dyd, dw, True, work, wsb)
    assert max_norm_rel(host(dw), 2 * ref) <= WGRAD_TOL
    check_status(D)


_SMALL_CLUSTERS = r"""
import sys, torch
sys.path.insert(0, sys.argv[1])
from paper_2509_26092_gb300 import dbl as D
gen = torch.Generator(device="cuda").manual_seed(5)
normal = lambda *s: torch.randn(s, device="cuda", generator=gen)
shape = D.conv_shape(1, 3, 3, 512, 512, 3, 1, 1)
assert D.dbl_conv_plan(shape, 0).grid <= int(sys.argv[3]) * 2
x, w = normal(1, 3, 3, 512).to(torch.bfloat16), (0.02 * normal(512, 3, 3, 512)).to(torch.bfloat16)
y, dw = torch.empty_like(x), torch.empty((512, 3, 3, 512), device="cuda")
D.dbl_conv_fwd(shape, x, w, y)
work = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
D.dbl_conv_wgrad(shape, x, y, dw, False, work, work.numel())
bn = D.bn_shape(577, 64, 1e-5, False)
u, v = normal(577, 64).to(torch.bfloat16), normal(577, 64).to(torch.bfloat16)
one, dg, db, dx = torch.ones(64, device="cuda"), torch.empty(64, device="cuda"), torch.empty(64, device="cuda"), torch.empty_like(u)
before = D.dbl_kernel_launches()
D.dbl_bn_relu_fused_bwd(bn, u, None, v, None, one, 0 * one, one, dx, None, dg, db, work, work.numel())
torch.cuda.synchronize()
assert D.dbl_device_status() == D.DBL_OK
torch.save([t.float().cpu() for t in (y, dw, dx, dg, db)] + [D.dbl_kernel_launches() - before], sys.argv[2])
"""


def test_devices_that_place_smaller_clusters_run_the_same_calls(tmp_path):
    """DBL_MAX_CLUSTER (read once per process) as the answer of such a device: sixteen CTAs, eight, none."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    got = {}
    for n in (16, 8, 1):
        path = str(tmp_path / f"{n}.pt")
        r = subprocess.run([sys.executable, "-c", _SMALL_CLUSTERS, root, path, str(max(n, 2))], capture_output=True,
                           text=True, timeout=600, env=dict(os.environ, DBL_MAX_CLUSTER=str(n)))
        assert r.returncode == 0, r.stderr[-2000:]
        got[n] = torch.load(path)
    assert [got[n][-1] for n in (16, 8, 1)] == [1, 3, 3]  # the BatchNorm backward's launches
    for n in (8, 1):
        for a, b, tol in zip(got[16], got[n], (2.0 ** -7, 2.0 ** -6, 2.0 ** -7, 1e-5, 1e-5)):
            # 16-bit outputs: a rounding decided otherwise by the order of fp32 sums (y is also dw's operand)
            assert (a - b).abs().max() <= tol * a.abs().max()


@pytest.mark.parametrize("n,h,c,k,stride,steps", [
    (256, 4, 256, 256, 1, 32),   # four pairs per tile, eight K-blocks each
    (64, 8, 256, 256, 1, 32),
    (37, 32, 128, 256, 2, 40),   # eight pairs
    (128, 7, 256, 128, 1, 56),   # 128 columns
])
def test_split_wgrad_sums_no_longer_chains_than_slices(D, n, h, c, k, stride, steps):
    """The tensor core rounds its sums towards zero: a chain of K-steps of 16 positions loses with its length.
    Random terms leave partial sums of sqrt(i / L) of the result after step i of L, each cut by half a unit of 2^-23
    on average: L / 3 * 2^-24 for all, a quarter more for the fp32 additions.  steps: L of the slices that run
    without clusters."""
    shape = D.conv_shape(n, h, h, c, k, 3, stride, 1)
    info = D.dbl_conv_plan(shape, D.DBL_PASS_WGRAD)
    assert info.kernel == D.DBL_KERNEL_IGEMM and info.grid > 2 * info.tiles  # tiles split over pairs
    gen = torch.Generator(device="cuda").manual_seed(n)
    p = (h - 1) // stride + 1
    x = torch.randn((n, h, h, c), device="cuda", generator=gen).to(torch.bfloat16)
    dy = torch.randn((n, p, p, k), device="cuda", generator=gen).to(torch.bfloat16)
    wsb = D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_WGRAD)
    dw = torch.full((k, 3, 3, c), float("nan"), device="cuda")
    D.dbl_conv_wgrad(shape, x, dy, dw, False, ws(wsb), wsb)
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    d2 = dy.double().reshape(-1, k)
    ref = torch.stack([torch.stack([d2.T @ xp[:, a:a + stride * p:stride, b:b + stride * p:stride].reshape(-1, c)
                                    for b in range(3)], 1) for a in range(3)], 1)
    err = float((dw.double() - ref).norm() / ref.norm())
    assert err <= 1.25 * steps / 3 * 2.0 ** -24
    check_status(D)
