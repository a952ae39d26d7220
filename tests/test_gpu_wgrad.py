"""The weight gradient from NHWC operands (conv_wgrad.cu) at the edges of its
plan: pixel boxes with remainders, one and two 128-channel M tiles and a
remainder, input channels past one N tile, tap groups of one and of all,
strides, and images larger than a box; through minw_conv_train_step with alpha 0.5 and
lr small enough not to clip, against the same bf16 operands in fp64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2003_04296_gb300.inputs import DEFAULT_THR  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()
    from paper_2003_04296_gb300 import minw
    return minw


@pytest.mark.parametrize("B,C,H,W,O,kh,kw,stride,pad", [
    (64, 64, 7, 7, 16, 3, 3, 1, 1),        # 49-pixel images: boxes of 64 with padding columns
    (32, 64, 13, 6, 100, 1, 1, 1, 0),
    (64, 128, 9, 9, 129, 3, 3, 2, 1),      # second M tile of one channel, stride 2
    (64, 320, 8, 8, 200, 1, 3, 1, 0),      # two N tiles with a remainder, a 1 x 3 kernel
    (16, 64, 32, 32, 300, 3, 3, 1, 1),     # two M groups
    (64, 64, 5, 5, 64, 5, 5, 1, 2),
    (1, 64, 64, 64, 32, 3, 3, 1, 1),
    (96, 64, 24, 24, 39, 1, 1, 1, 0),      # a slice per SM: more than the update has in flight, with a remainder
    (64, 256, 8, 8, 300, 3, 3, 1, 1),      # a gradient of many elements: the update's wide blocks
])
def test_weight_gradient(M, B, C, H, W, O, kh, kw, stride, pad):
    g = torch.Generator(device="cuda").manual_seed(B + C + H + W + O)
    A = (torch.randn((B, C, H, W), generator=g, device="cuda") / (C * kh * kw) ** 0.5).contiguous()
    Wt = torch.rand((O, C, kh, kw), generator=g, device="cuda") * 1.8 - 0.9
    Ho, Wo = (H + 2 * pad - kh) // stride + 1, (W + 2 * pad - kw) // stride + 1
    G = torch.randn((B, O, Ho, Wo), generator=g, device="cuda") * 0.1
    lr, alpha = 1e-5, 0.5
    W0 = Wt.clone()
    a_out, g_in = torch.empty_like(G), torch.empty_like(A)
    ws = torch.empty(M.minw_conv_train_workspace_bytes(B, C, H, W, O, kh, kw, stride, pad), dtype=torch.uint8, device="cuda")
    q = M.quant(2, DEFAULT_THR[2])
    M.minw_conv_train_step(A, Wt, G, stride, pad, alpha, lr, q, None, a_out, g_in, ws)     # the last layer: g~ = g
    a64, g64 = A.bfloat16().double(), G.bfloat16().double()
    ref = torch.nn.grad.conv2d_weight(a64, Wt.shape, g64, stride, pad)
    absum = torch.nn.grad.conv2d_weight(a64.abs(), Wt.shape, g64.abs(), stride, pad)
    # fp32 accumulation over the pixels (2^-23 per product covers rounding or truncating adds); the step adds
    # one rounding of lr g and one of w
    n = B * Ho * Wo
    bound = lr * (n * 2.0 ** -23 * absum + 2.0 ** -23 * ref.abs()) + 2.0 ** -23 * W0.abs().double()
    err = (Wt.double() - (W0.double() - lr * ref)).abs()
    assert (err <= bound).all(), float((err / bound).max())
    assert M.minw_get_last_device_error() == M.MINW_OK


def test_short_gradients_are_not_bound_by_the_slice_sums(M):
    """A 1x1 layer's gradient has few elements, each the sum of a slice per SM:
    its step takes less than that of the 3x3 layer of the same sizes, which
    does nine times the products."""
    B, C, S, O = 96, 64, 24, 39
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn((B, C, S, S), generator=g, device="cuda") * 0.1
    G = torch.randn((B, O, S, S), generator=g, device="cuda") * 0.1
    a_out, g_in = torch.empty_like(G), torch.empty_like(A)
    q = M.quant(2, DEFAULT_THR[2])
    us = []
    for k in (1, 3):
        Wt = torch.rand((O, C, k, k), generator=g, device="cuda") * 2 - 1
        ws = torch.empty(M.minw_conv_train_workspace_bytes(B, C, S, S, O, k, k, 1, k // 2), dtype=torch.uint8, device="cuda")
        best = float("inf")
        for i in range(30):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            for _ in range(5):
                M.minw_conv_train_step(A, Wt, G, 1, k // 2, 0.75, 1e-4, q, q, a_out, g_in, ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 200 if i else best)
        us.append(best)
    assert us[0] <= 0.9 * us[1], us
