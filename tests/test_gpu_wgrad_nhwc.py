"""Weight and bias gradients straight from the NHWC arrays (uot_conv_tc_wgrad_nhwc) against the
FP64 network oracle on BF16-rounded operands, at the edges of its row chains: dilations that
leave one or two rows per chain, image heights that are no multiple of the dilation, dilations
past the image, splits that cut chains, and 2- and 4-channel layers.

BF16 products are exact in FP32, so only the accumulation rounds: a chain of P/16 additions of
16-product sums per output at most (P pixels), then the splits; each addition rounds or truncates
to 2^-23 of a partial sum that is at most sum |g||x|."""
import numpy as np
import pytest
import torch

import oracle.net_oracle as NO
from paper_1607_05816_gb300 import uot as U

pytestmark = pytest.mark.gpu


def bf(a):
    return torch.as_tensor(np.asarray(a, np.float32)).to(torch.bfloat16).float().double().numpy()


def nhwc(a, ld):
    N, C, H, W = a.shape
    out = np.zeros((N, H, W, ld), np.float32)
    out[..., :C] = np.transpose(a, (0, 2, 3, 1))
    return torch.as_tensor(out.reshape(N * H * W, ld)).to(torch.bfloat16).cuda()


@pytest.mark.parametrize("N,H,Cin,ldx,Cout,ldg,dil,splits", [
    (1, 1, 128, 128, 128, 128, 1, 1),     # one row, no neighbours
    (2, 8, 128, 128, 128, 128, 2, 5),     # splits cut the chains
    (1, 7, 128, 128, 128, 128, 3, 2),     # ragged chains
    (2, 6, 128, 128, 128, 128, 4, 3),     # chains of one and two rows
    (2, 5, 128, 128, 128, 128, 32, 4),    # dilation past the image
    (3, 16, 64, 64, 64, 64, 1, 7),        # 64-channel tiles
    (3, 4, 4, 64, 128, 128, 1, 12),       # first layer
    (2, 8, 128, 128, 2, 16, 3, 50),       # last layer, more splits than rows
])
def test_wgrad_nhwc_matches_oracle(N, H, Cin, ldx, Cout, ldg, dil, splits):
    W = 64
    g = np.random.default_rng(100 * N + H + dil)
    x = bf(g.normal(size=(N, Cin, H, W)))
    dy = bf(g.normal(size=(N, Cout, H, W)))
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    dw, db = U.conv_tc_wgrad_nhwc(nhwc(dy, ldg), nhwc(x, ldx), N, H, W, dil, Cout, Cin, splits=splits, err=err)
    torch.cuda.synchronize()
    assert err.item() == 0
    _, want_w, want_b = NO.conv2d_grads(x, np.zeros((Cout, Cin, 3, 3)), dy, dil)
    _, abs_w, abs_b = NO.conv2d_grads(np.abs(x), np.zeros((Cout, Cin, 3, 3)), np.abs(dy), dil)
    tol = (N * H * W / 16 + splits + 4) * 2.0 ** -23
    assert np.all(np.abs(dw.double().cpu().numpy() - want_w) <= tol * abs_w + 1e-30)
    assert np.all(np.abs(db.double().cpu().numpy() - want_b) <= 16 * tol * abs_b + 1e-30)


def test_wgrad_nhwc_refuses_what_does_not_fit():
    x = torch.zeros(64, 64, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(U.UotError):
        U.conv_tc_wgrad_nhwc(x, x, 1, 1, 64, 1, 65, 64)  # more outputs than the gradient has channels
    with pytest.raises(U.UotError):
        U.conv_tc_wgrad_nhwc(x, x, 2, 1, 32, 1, 64, 64)  # image width
    with pytest.raises(ValueError):
        U.conv_tc_wgrad_nhwc(x, x, 1, 1, 64, 1, 64, 64, part=torch.empty(10, device="cuda"))
