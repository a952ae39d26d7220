"""The 3x3 convolution on tiles with their halo (conv_halo_kernel: stride 1,
pad 1, rows of 64 or 128 bytes, level outputs only, 16 x 8-pixel tiles), bit
for bit against the tile-per-tap kernel (plan option channel_major = 0) on
every image and the oracle on the first and the last: ragged images, channel
tiles of 32 to 128 and several of them, pooled and residual blocks, every
width and format of the outputs.  The residual epilogue's two rarer branches,
which both kernels share, and the halo kernel's timeout path."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2003_04296_gb300.inputs import DEFAULT_THR, conv_problem  # noqa: E402
from tests._gpu import dev_tensor, planes_view  # noqa: E402
from tests.test_gpu_e2m1 import decode_e2m1  # noqa: E402
from tests.test_gpu_tc import decode_e4m3  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()
    from paper_2003_04296_gb300 import minw
    return minw


@pytest.fixture
def restore(M):
    yield
    M.set_plan_options()
    M.minw_test_stall_next_launch(0)


def _codes(M, x, bits, thr, fp4):
    out = torch.empty((x.shape[0], x.shape[2], x.shape[3], x.shape[1] // (2 if fp4 else 1)), dtype=torch.uint8,
                      device="cuda")
    (M.aqe_quantize_codes_e2m1 if fp4 else M.aqe_quantize_codes)(dev_tensor(x, "cuda"), M.quant(bits, thr), out)
    return out


def _weights(M, p, bits, fp4):
    O_, C = p["w"].shape[:2]
    out = torch.empty((O_, 3, 3, C // (2 if fp4 else 1)), dtype=torch.uint8, device="cuda")
    (M.minw_pack_weight_codes_e2m1 if fp4 else M.minw_pack_weight_codes)(
        dev_tensor(p["w"], "cuda"), M.quant(bits, p["thr_w"]), out, dev_tensor(p["w_scale"], "cuda"))
    return out


def _unaligned(t, off):
    """The tensor's values ``off`` bytes past a 16-byte boundary."""
    raw = torch.empty(t.numel() * t.element_size() + 32, dtype=torch.uint8, device="cuda")
    v = raw[off:off + t.numel() * t.element_size()].view(t.dtype).view(t.shape)
    v.copy_(t)
    return v


def _check(M, B, C, H, W, O_, bits, fp4, pool, res, thr=None, off=0, want_y=False):
    """One block under both plans: codes of the input's format and planes
    (and the BN output before the shortcut), against each other and the oracle."""
    p = conv_problem(B + H + O_ + bits, B, C, H, W, O_, 3, 3, 1, 1, bits, bits, x_dist="normal", w_sigma=0.05)
    thr = thr or DEFAULT_THR[bits]
    act, wgt = _codes(M, p["x"], bits, p["thr_a"], fp4), _weights(M, p, bits, fp4)
    r = np.random.default_rng(O_ + H)
    kw, shortcut = {}, np.float32(0.0)
    if res == "codes":
        xs = (r.standard_normal((B, O_, H, W)) * 0.7).astype(np.float32)
        shortcut = O.quantize(xs, bits, DEFAULT_THR[bits]).astype(np.float32)
        rc = _codes(M, xs, bits, DEFAULT_THR[bits], fp4)
        kw = dict(res_codes=_unaligned(rc, off) if off else rc, res_bits=bits, res_format=int(fp4))
    elif res == "f32":
        shortcut = (r.standard_normal((B, O_, H, W)) * 0.5).astype(np.float32)
        rf = dev_tensor(shortcut.transpose(0, 2, 3, 1), "cuda")
        kw = dict(res_f32=_unaligned(rf, off) if off else rf)
    Ho, Wo = H >> pool, W >> pool
    got = []
    for plan in (1, 0):
        M.set_plan_options(channel_major=plan)
        codes = torch.full((B, Ho, Wo, O_ // (2 if fp4 else 1)), 0x77, dtype=torch.uint8, device="cuda")
        planes = torch.full((M.packed_words(B, O_, Ho, Wo, bits),), -1, dtype=torch.int32, device="cuda")
        y = torch.empty((B, H, W, O_), device="cuda") if want_y else None
        M.minw_conv_block_codes_ex(act, B, C, H, W, bits, wgt, O_, 3, 3, bits, 1, 1, pool, dev_tensor(p["scale"], "cuda"),
                                   dev_tensor(p["shift"], "cuda"), q_out=M.quant(bits, thr), codes_out=codes,
                                   planes_out=planes, in_format=int(fp4), out_format=int(fp4), y_nhwc=y, **kw)
        assert M.minw_get_last_device_error() == M.MINW_OK
        got.append((codes, planes))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    pick = sorted({0, B - 1})
    acc = O.conv2d_levels(O.quantize(p["x"][pick], bits, p["thr_a"]),
                          O.quantize(p["w"], bits, p["thr_w"], p["w_scale"]), 1, 1, bits, bits)
    if pool:
        acc = O.maxpool_i32(acc, 2, 2)
    bn = O.affine(acc, p["scale"], p["shift"])
    lv = O.quantize(O.hardtanh((bn + (shortcut[pick] if res else shortcut)).astype(np.float32)), bits, thr)
    values = (decode_e2m1(got[0][0].cpu().numpy(), O_) if fp4 else decode_e4m3(got[0][0].cpu().numpy()))[pick]
    assert np.array_equal(values, lv.transpose(0, 2, 3, 1) * 2.0 ** O.units_shift(bits))
    assert np.array_equal(planes_view(got[0][1], B, Ho, Wo, bits, O_)[pick], O.pack(lv, bits))
    if want_y:
        assert np.array_equal(y.cpu().numpy()[pick], bn.transpose(0, 2, 3, 1))


# B, C, H, W, O, E2M1: rows of C or C / 2 bytes; tiles that cover 0.6 of their pixels or more, or
# (a tile per SM at most) 0.45
SHAPES = [
    (1, 64, 16, 8, 64, False),          # one whole tile
    (3, 64, 30, 28, 32, False),         # a ragged last row and column of tiles, the narrowest channel tile
    (2, 128, 18, 24, 96, False),        # covered 0.56 in 12 tiles, 96 channels
    (3, 128, 20, 14, 160, True),        # O with no even split into tiles of 32: not this kernel's
    (5, 128, 34, 40, 192, True),        # two channel tiles of 96
    (40, 256, 12, 14, 512, True),       # four channel tiles of 128, 80 pixel tiles
    (60, 128, 28, 26, 128, True),       # several tiles per CTA: buffers and accumulators in turn
]


@pytest.mark.parametrize("bits", [1, 2, 3])
@pytest.mark.parametrize("mode", ["plain", "pool", "codes", "f32"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_halo_levels(M, restore, shape, mode, bits):
    B, C, H, W, O_, fp4 = shape
    _check(M, B, C, H, W, O_, bits, fp4, int(mode == "pool"), mode if mode in ("codes", "f32") else None)


@pytest.mark.parametrize("bits", [1, 3])
@pytest.mark.parametrize("shape", [(2, 64, 13, 9, 64, False), (3, 128, 29, 31, 96, True)],
                         ids=lambda s: "x".join(map(str, s)))
def test_halo_odd_images(M, restore, shape, bits):
    _check(M, *shape[:5], bits, shape[5], 0, None)


@pytest.mark.parametrize("res", ["codes", "f32"])
@pytest.mark.parametrize("fp4", [False, True])
def test_breakpoints_that_do_not_mirror(M, restore, res, fp4):
    """A 3-bit quantizer whose top level no output reaches (a threshold of 1
    after HardTanh): its breakpoints are infinite there, and the residual
    epilogue compares with all six."""
    _check(M, 5, 128, 16, 24, 64, 3, fp4, 0, res, thr=(1.0, 0.375, 0.125))


@pytest.mark.parametrize("res,off", [("codes", 4), ("codes", 1), ("f32", 4), ("f32", 8)])
def test_unaligned_shortcut(M, restore, res, off):
    """A shortcut that does not start on 16 bytes is read element by element."""
    _check(M, 3, 64, 16, 16, 64, 3, False, 0, res, off=off)


@pytest.mark.parametrize("res", ["codes", "f32", None])
def test_residual_with_bn_output(M, restore, res):
    """The BN output before the shortcut (or without one) as fp32 NHWC beside the levels."""
    _check(M, 3, 128, 14, 14, 96, 2, False, 0, res, want_y=True)


def test_halo_timeout(M, restore):
    """A stalled MMA issuer: MINW_ETIMEOUT once, then a correct run and MINW_OK."""
    B, C, S, O_ = 4, 64, 32, 64
    p = conv_problem(9, B, C, S, S, O_, 3, 3, 1, 1, 1, 1, x_dist="normal", w_sigma=0.05)
    act, wgt = _codes(M, p["x"], 1, p["thr_a"], False), _weights(M, p, 1, False)
    codes = torch.empty((B, S, S, O_), dtype=torch.uint8, device="cuda")

    def call():
        M.minw_conv_block_codes(act, B, C, S, S, 1, wgt, O_, 3, 3, 1, 1, 1, 0, dev_tensor(p["scale"], "cuda"),
                                dev_tensor(p["shift"], "cuda"), q_out=M.quant(1, DEFAULT_THR[1]), codes_out=codes)

    assert M.minw_get_last_device_error() == M.MINW_OK
    M.set_plan_options(wait_cycles=1 << 20)
    M.minw_test_stall_next_launch(M.STALL_CONV_TC)
    call()
    assert M.minw_get_last_device_error() == M.MINW_ETIMEOUT
    assert M.minw_get_last_device_error() == M.MINW_OK
    call()
    assert M.minw_get_last_device_error() == M.MINW_OK
    acc = O.conv2d_levels(O.quantize(p["x"], 1, p["thr_a"]), O.quantize(p["w"], 1, p["thr_w"], p["w_scale"]), 1, 1, 1, 1)
    lv = O.quantize(O.hardtanh(O.affine(acc, p["scale"], p["shift"])), 1, DEFAULT_THR[1])
    assert np.array_equal(decode_e4m3(codes.cpu().numpy()), lv.transpose(0, 2, 3, 1))
