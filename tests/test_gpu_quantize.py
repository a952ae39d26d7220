"""quantize_kernel (aqe_quantize_pack and the level-code quantizers) at the
edges of its tiles: 32 / 64 / 128-pixel runs, channel groups with remainders,
rows whose length is no multiple of 4 or 32, inputs off a 16-byte boundary,
special values, and graph capture behind copies and fills."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2003_04296_gb300.inputs import DEFAULT_THR  # noqa: E402
from tests._gpu import assert_close, dev_tensor, planes_view, words  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()
    from paper_2003_04296_gb300 import minw
    return minw


def _values(shape, bits, seed):
    """N(0, 1.2) with thresholds, their neighbours, zeros, infinities and NaN mixed in."""
    r = np.random.default_rng(seed)
    x = (r.standard_normal(shape) * 1.2).astype(np.float32)
    sp = np.array([0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, 3.4e38, 1e-45], np.float32)
    t = np.array(DEFAULT_THR[bits], np.float32)
    sp = np.concatenate([sp, t, -t, np.nextafter(t, np.float32(9)), np.nextafter(t, np.float32(-9)),
                         np.nextafter(np.float32([1.0]), np.float32(9))])
    at = r.integers(0, x.size, min(x.size, 200))
    x.ravel()[at] = r.choice(sp, at.size)
    return x


def _mask_bits(x):
    flat = np.abs(x.ravel()) <= 1.0
    pad = np.zeros((-flat.size) % 32, bool)
    return np.packbits(np.concatenate([flat, pad]), bitorder="little").view(np.uint32)


def _at_offset(x, off):
    buf = torch.empty(x.size + off, dtype=torch.float32, device="cuda")
    v = buf[off:].view(x.shape)
    v.copy_(torch.from_numpy(x))
    return v


SHAPES = [(1, 1, 1, 1), (2, 3, 7, 9), (3, 33, 2, 2), (2, 64, 14, 14), (1, 65, 8, 8), (2, 40, 16, 10), (1, 130, 12, 11),
          (2, 160, 6, 6), (1, 512, 14, 14), (2, 96, 33, 4),
          # up to 16 channels, few blocks of one warp a group
          (2, 4, 32, 32), (3, 3, 33, 32), (2, 7, 13, 9), (1, 8, 50, 40), (1, 12, 40, 28), (2, 16, 29, 21), (1, 1, 47, 45),
          # and many, in one to four groups: whole and ragged runs of 1024, 512 and 256 pixels (scalar: a quarter)
          (40, 4, 32, 32), (3, 3, 65, 63), (1, 7, 99, 101), (1, 8, 201, 200), (1, 12, 280, 281), (2, 16, 141, 141),
          (2, 1, 161, 160), (77, 5, 16, 32), (610, 9, 4, 6), (310, 2, 5, 5),
          # images of up to 16 pixels with as few lanes, many channels
          (4, 100, 1, 1), (3, 1030, 1, 1), (2, 70, 3, 3), (33, 40, 1, 2), (1, 5, 3, 5), (2, 600, 1, 11)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bits", [1, 2, 3])
@pytest.mark.parametrize("off", [0, 1])
def test_planes_mask_forward(M, shape, bits, off):
    B, C, H, W = shape
    x = _values(shape, bits, sum(shape) + bits)
    xd = _at_offset(x, off)
    planes = torch.full((M.packed_words(B, C, H, W, bits),), -1, dtype=torch.int32, device="cuda")
    y = torch.empty(shape, device="cuda")
    n = x.size
    mask = torch.full(((n + 31) // 32,), -1, dtype=torch.int32, device="cuda")
    M.aqe_quantize_pack(xd, M.quant(bits, DEFAULT_THR[bits]), planes, alpha=0.6, y=y, mask=mask)
    lv = O.quantize(x, bits, DEFAULT_THR[bits])
    assert np.array_equal(planes_view(planes, B, H, W, bits, C), O.pack(lv, bits))
    assert np.array_equal(words(mask), _mask_bits(x))
    fin = np.isfinite(x)
    assert_close(y.cpu().numpy()[fin], O.aqe_forward(x, 0.6, bits, DEFAULT_THR[bits])[fin])
    planes2 = torch.full_like(planes, -1)
    M.aqe_quantize_pack(xd, M.quant(bits, DEFAULT_THR[bits]), planes2)
    assert torch.equal(planes, planes2)


@pytest.mark.parametrize("bits", [1, 2, 3])
@pytest.mark.parametrize("shape,off", [((2, 16, 5, 5), 0), ((1, 48, 4, 4), 0), ((2, 64, 14, 14), 0), ((1, 96, 9, 9), 0),
                                       ((2, 160, 8, 8), 1), ((1, 512, 7, 7), 0), ((3, 32, 12, 11), 1),
                                       ((1, 16, 64, 44), 0), ((2, 16, 20, 20), 1), ((1, 16, 280, 281), 0), ((2, 16, 141, 141), 0),
                                       ((3, 16, 3, 3), 0), ((3, 32, 1, 1), 0),
                                       ((2, 1056, 1, 1), 0), ((2, 64, 1, 5), 0)])
def test_codes(M, shape, bits, off):
    B, C, H, W = shape
    x = _values(shape, bits, sum(shape) + bits)
    xd = _at_offset(x, off)
    lv = O.quantize(x, bits, DEFAULT_THR[bits]) * (4 if bits == 3 else 1)
    lv = np.rint(lv).astype(np.int64).transpose(0, 2, 3, 1)
    e4 = np.vectorize({0: 0, 1: 0x38, 2: 0x40, 4: 0x48, -1: 0xB8, -2: 0xC0, -4: 0xC8}.get)(lv).astype(np.uint8)
    codes = torch.full((B, H, W, C), 0x77, dtype=torch.uint8, device="cuda")
    M.aqe_quantize_codes(xd, M.quant(bits, DEFAULT_THR[bits]), codes)
    assert np.array_equal(codes.cpu().numpy(), e4)
    if C % 32 == 0:
        nib = np.vectorize({0: 0, 1: 2, 2: 4, 4: 6, -1: 10, -2: 12, -4: 14}.get)(lv).astype(np.uint8)
        codes = torch.full((B, H, W, C // 2), 0x77, dtype=torch.uint8, device="cuda")
        M.aqe_quantize_codes_e2m1(xd, M.quant(bits, DEFAULT_THR[bits]), codes)
        assert np.array_equal(codes.cpu().numpy(), nib[..., 0::2] | (nib[..., 1::2] << 4))


def test_few_channels_keep_the_threads_busy(M):
    """Three-channel images take the time of their bytes: at most twice that
    of as many 96-channel values."""
    us = []
    for shape in ((64, 3, 224, 224), (64, 96, 49, 32)):
        x = torch.zeros(shape, device="cuda")
        planes = torch.empty(M.packed_words(*shape, 1), dtype=torch.int32, device="cuda")
        best = float("inf")
        for i in range(20):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            for _ in range(5):
                M.aqe_quantize_pack(x, M.quant(1, DEFAULT_THR[1]), planes)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 200 if i else best)
        us.append(best)
    assert us[0] <= 2 * us[1], us


def test_capture_behind_copies_and_fills(M):
    """The launches overlap their predecessor (programmatic serialization); behind a copy or a
    fill, in a captured graph as in a stream, they wait for it."""
    shape = (2, 64, 14, 14)
    x = _values(shape, 2, 5)
    host = torch.from_numpy(x).pin_memory()
    xd = torch.zeros(shape, device="cuda")
    planes = torch.zeros(M.packed_words(*shape, 2), dtype=torch.int32, device="cuda")
    mask = torch.zeros((x.size + 31) // 32, dtype=torch.int32, device="cuda")
    codes = torch.zeros((2, 14, 14, 64), dtype=torch.uint8, device="cuda")
    y = torch.empty(shape, device="cuda")
    q = M.quant(2, DEFAULT_THR[2])

    def work():
        xd.copy_(host, non_blocking=True)
        M.aqe_quantize_codes(xd, q, codes)
        planes.zero_()
        M.aqe_quantize_pack(xd, q, planes, alpha=0.6, y=y, mask=mask)

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        work()
    s.synchronize()
    want = [t.clone() for t in (planes, mask, codes, y)]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        work()
    for t in (planes, mask, codes, y):
        t.fill_(1)
    g.replay()
    torch.cuda.synchronize()
    for a, b in zip((planes, mask, codes, y), want):
        assert a.equal(b) or (a.isnan() == b.isnan()).all() and a.nan_to_num().equal(b.nan_to_num())
    assert np.array_equal(planes_view(planes, 2, 14, 14, 2, 64), O.pack(O.quantize(x, 2, DEFAULT_THR[2]), 2))
