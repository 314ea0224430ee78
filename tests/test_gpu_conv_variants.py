"""Edges of the convolution kernels chosen by shape: row-block weight gradients (3x3 stride 1, 64
channels), against the fp64 oracle."""
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
