"""The bit-plane convolution on the tensor cores (conv_planes_tc.cu, what
minw_conv2d and minw_conv_block run unless the popcount path is requested):
exact accumulators against the CPU oracle at tile edges, bit-equal outputs
against the popcount kernel over the shapes both accept, and its timeout path."""
from itertools import product

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2003_04296_gb300.inputs import DEFAULT_THR, conv_problem  # noqa: E402
from tests._gpu import case_seed, dev_tensor  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()
    from paper_2003_04296_gb300 import minw
    return minw


def _operands(M, B, C, H, W, O_, k, ba, bw, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((B, C, H, W), generator=g, device="cuda")
    w = torch.randn((O_, C, k, k), generator=g, device="cuda") * 0.5
    act = torch.empty(M.packed_words(B, C, H, W, ba), dtype=torch.int32, device="cuda")
    wgt = torch.empty(M.packed_words(O_, C, k, k, bw), dtype=torch.int32, device="cuda")
    M.aqe_quantize_pack(x, M.quant(ba, DEFAULT_THR[ba]), act)
    M.minw_pack_weights(w, M.quant(bw, DEFAULT_THR[bw]), wgt)
    unit = (4.0 if ba == 3 else 1.0) * (4.0 if bw == 3 else 1.0)
    scale = (1.0 + 0.1 * torch.randn(O_, generator=g, device="cuda")) / (unit * (C * k * k * 0.3) ** 0.5)
    scale[::5] *= -1.0
    shift = 0.1 * torch.randn(O_, generator=g, device="cuda")
    return x, w, act, wgt, scale, shift


# B, C, H, W, O, k, stride, pad: words per pixel 1 .. 16 (whole chunks, remainders, one tap per
# several chunks), channel tiles of 32 / 64 / 128 with remainders, pixel tiles with remainders
SHAPES = [
    (1, 32, 1, 1, 1, 1, 1, 0),
    (2, 64, 9, 7, 70, 3, 1, 1),
    (3, 96, 13, 11, 33, 3, 2, 1),
    (1, 160, 8, 17, 130, 1, 3, 0),
    (5, 32, 16, 16, 40, 5, 1, 2),
    (4, 128, 32, 32, 128, 3, 1, 1),
    (37, 96, 32, 32, 200, 3, 1, 1),
    (9, 512, 14, 14, 300, 3, 1, 1),
    (64, 256, 8, 8, 512, 3, 2, 0),
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ba,bw", list(product([1, 2, 3], [1, 2, 3])))
def test_matches_popcount(M, shape, ba, bw):
    B, C, H, W, O_, k, s, pad = shape
    _, _, act, wgt, scale, shift = _operands(M, B, C, H, W, O_, k, ba, bw, case_seed(shape, ba, bw))
    Ho, Wo = (H + 2 * pad - k) // s + 1, (W + 2 * pad - k) // s + 1
    got = []
    for variant in (M.VARIANT_AUTO, M.VARIANT_POPC):
        acc = torch.full((B, O_, Ho, Wo), -7, dtype=torch.int32, device="cuda")
        y = torch.full((B, O_, Ho, Wo), -7.0, device="cuda")
        M.minw_conv2d(act, B, C, H, W, ba, wgt, O_, k, k, bw, s, pad, acc, scale, shift, y, variant=variant)
        bo = 1 + (ba + bw) % 3
        planes = torch.full((M.packed_words(B, O_, Ho, Wo, bo),), -1, dtype=torch.int32, device="cuda")
        yq = torch.full((B, O_, Ho, Wo), -7.0, device="cuda")
        M.minw_conv_block(act, B, C, H, W, ba, wgt, O_, k, k, bw, s, pad, 0, scale, shift,
                          M.quant(bo, DEFAULT_THR[bo]), planes, yq, variant=variant)
        got.append((acc, y, planes, yq))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert M.minw_get_last_device_error() == M.MINW_OK


@pytest.mark.parametrize("side", [2, 4, 8, 16, 32, 64])
@pytest.mark.parametrize("bo", [0, 1, 2, 3])
def test_pooled_matches_popcount(M, side, bo):
    """2x2 pooling at every output width whose windows a 128-pixel tile holds."""
    B, C, O_ = 3, 64, 72
    _, _, act, wgt, scale, shift = _operands(M, B, C, side, side, O_, 3, 2, 3, side + bo)
    h = side // 2
    got = []
    for variant in (M.VARIANT_AUTO, M.VARIANT_POPC):
        y = torch.full((B, O_, h, h), -7.0, device="cuda")
        planes = torch.full((M.packed_words(B, O_, h, h, max(bo, 1)),), -1, dtype=torch.int32, device="cuda")
        q = M.quant(bo, DEFAULT_THR[bo]) if bo else None
        M.minw_conv_block(act, B, C, side, side, 2, wgt, O_, 3, 3, 3, 1, 1, 1, scale, shift, q,
                          planes if bo else None, y, variant=variant)
        got.append((y, planes))
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("ba,bw", [(1, 1), (3, 3), (1, 3), (2, 1)])
def test_exact_against_oracle(M, ba, bw):
    """Largest magnitudes of a 512-channel 3x3 kernel, and a ragged shape, against the oracle."""
    for B, C, H, W, O_, big in ((2, 512, 6, 6, 40, True), (3, 96, 7, 9, 35, False)):
        p = conv_problem(ba * 4 + bw, B, C, H, W, O_, 3, 3, 1, 1, ba, bw, w_sigma=0.5)
        if big:
            p["x"] = np.where(p["x"] > -2.0, 1.0, -1.0).astype(np.float32)
            p["w"] = np.ones_like(p["w"])
            p["w_scale"] = np.ones_like(p["w_scale"])
        act = torch.empty(M.packed_words(B, C, H, W, ba), dtype=torch.int32, device="cuda")
        wgt = torch.empty(M.packed_words(O_, C, 3, 3, bw), dtype=torch.int32, device="cuda")
        M.aqe_quantize_pack(dev_tensor(p["x"], "cuda"), M.quant(ba, p["thr_a"]), act)
        M.minw_pack_weights(dev_tensor(p["w"], "cuda"), M.quant(bw, p["thr_w"]), wgt,
                            channel_scale=dev_tensor(p["w_scale"], "cuda"))
        acc = torch.full((B, O_, H, W), -7, dtype=torch.int32, device="cuda")
        M.minw_conv2d(act, B, C, H, W, ba, wgt, O_, 3, 3, bw, 1, 1, acc)
        ref = O.conv2d_levels(O.quantize(p["x"], ba, p["thr_a"]), O.quantize(p["w"], bw, p["thr_w"], p["w_scale"]),
                              1, 1, ba, bw)
        assert np.array_equal(acc.cpu().numpy(), ref)


def _replay_us(call):
    """Least time of a pass, 20 of them in a graph."""
    call()
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        for _ in range(20):
            call()
    best = float("inf")
    for _ in range(12):
        a, b = torch.cuda.Event(True), torch.cuda.Event(True)
        a.record()
        g.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 50)
    return best


# B, C, side, O, bits of activations, weights and outputs (0: fp32, None: raw accumulators), pool
SHORT = [
    (160, 32, 32, 64, 2, 2, 1, 1),
    (160, 32, 32, 64, 1, 1, 3, 1),
    (160, 64, 32, 96, 2, 1, 0, 1),
    (160, 32, 32, 8, 2, 1, 2, 0),
    (160, 32, 32, 16, 1, 1, 0, 0),
    (160, 64, 32, 4, 2, 2, 1, 1),
    (160, 32, 32, 64, 2, 2, None, 0),
    (40, 64, 32, 40, 2, 1, None, 0),
]


@pytest.mark.parametrize("case", SHORT)
def test_auto_is_not_slower_than_popcount(M, case):
    """1x1 layers of one or two words, where a tile's fixed cost and its
    epilogue are all there is: the kernel that the automatic choice runs takes
    at most a tenth more than the popcount kernel."""
    B, C, side, O_, ba, bw, bo, pool = case
    _, _, act, wgt, scale, shift = _operands(M, B, C, side, side, O_, 1, ba, bw, O_ + C)
    h = side >> pool
    y = torch.empty((B, O_, h, h), device="cuda")
    acc = torch.empty((B, O_, h, h), dtype=torch.int32, device="cuda")
    planes = torch.empty(M.packed_words(B, O_, h, h, bo or 1), dtype=torch.int32, device="cuda")
    q = M.quant(bo, DEFAULT_THR[bo]) if bo else None

    def call(variant):
        if bo is None:
            M.minw_conv2d(act, B, C, side, side, ba, wgt, O_, 1, 1, bw, 1, 0, acc, variant=variant)
        else:
            M.minw_conv_block(act, B, C, side, side, ba, wgt, O_, 1, 1, bw, 1, 0, pool, scale, shift, q,
                              planes if bo else None, None if bo else y, variant=variant)

    us = [_replay_us(lambda: call(v)) for v in (M.VARIANT_AUTO, M.VARIANT_POPC)]
    assert us[0] <= 1.1 * us[1], us


def test_timeout_path(M):
    """A stalled MMA issuer: the bounded waits run out, the status is reported
    once, and the next launch is correct."""
    B, C, H, W, O_ = 2, 128, 8, 8, 64
    _, _, act, wgt, _, _ = _operands(M, B, C, H, W, O_, 3, 2, 2, 3)
    acc = [torch.empty((B, O_, H, W), dtype=torch.int32, device="cuda") for _ in range(2)]
    assert M.minw_get_last_device_error() == M.MINW_OK
    M.set_plan_options(wait_cycles=1 << 20)
    try:
        M.minw_test_stall_next_launch(M.STALL_CONV_TC)
        M.minw_conv2d(act, B, C, H, W, 2, wgt, O_, 3, 3, 2, 1, 1, acc[0])
        assert M.minw_get_last_device_error() == M.MINW_ETIMEOUT
    finally:
        M.minw_test_stall_next_launch(0)
        M.set_plan_options()
    M.minw_conv2d(act, B, C, H, W, 2, wgt, O_, 3, 3, 2, 1, 1, acc[0])
    M.minw_conv2d(act, B, C, H, W, 2, wgt, O_, 3, 3, 2, 1, 1, acc[1], variant=M.VARIANT_POPC)
    assert torch.equal(acc[0], acc[1])
    assert M.minw_get_last_device_error() == M.MINW_OK
