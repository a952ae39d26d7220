"""The one-kernel forward of the weight-only residual network (wres_fused.cu)
at the image sizes where its tiles have remainders (8 x 16-pixel tiles of 8 .. 28-pixel
images) and one size above its range (layer by layer), every stage against
the oracle; and the layer-by-layer forward that per-op timing takes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import network as N  # noqa: E402
from oracle import oracle as O  # noqa: E402
from paper_2003_04296_gb300.inputs import wresnet_input, wresnet_params  # noqa: E402
from tests._gpu import dev_tensor  # noqa: E402
from tests.test_gpu_wresnet import M, _check_block, _run, dev  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hw,n,B", [(8, 1, 3), (12, 2, 2), (20, 1, 2), (24, 1, 1), (28, 1, 2), (36, 1, 1)])
def test_image_sizes(dev, M, hw, n, B):  # noqa: F811
    bits = 1 + hw % 3
    net_p = wresnet_params(hw + n, n=n, bits_w=bits, classes=37, hw=hw)
    x = wresnet_input(hw, B, hw=hw)
    logits, acts = _run(dev, M, net_p, x)
    st = net_p["stem"]
    assert np.array_equal(acts[0], O.hardtanh(O.affine(O.conv2d_f32_seq(x, st["w"], 1, 1), st["scale"], st["shift"])))
    for i, blk in enumerate(net_p["blocks"]):
        _check_block(blk, acts[i], acts[i + 1], bits, net_p["thr_w"])
    assert np.array_equal(logits, N.wresnet_head(net_p, acts[-1]))


def test_batch_above_the_sm_count_and_timing(dev, M):  # noqa: F811
    """More images than SMs (several CTAs in turn per SM); each image's logits do not depend on the
    batch; with timing on, the layer-by-layer path gives the same activations within its own bound."""
    net_p = wresnet_params(5, n=1, bits_w=3, classes=10, hw=32)
    x = wresnet_input(6, 200, hw=32)
    big, _ = _run(dev, M, net_p, x, keep=False)
    small, _ = _run(dev, M, net_p, x[190:193], keep=False)
    assert np.array_equal(big[190:193], small)
    net = M.Net.wresnet(net_p, 2, dev, keep_activations=True)
    logits = torch.empty((2, 10), device=dev)
    net.enable_timing(True)
    net.forward(dev_tensor(x[:2], dev), logits)
    assert len(net.layer_times()) == net.launches
    acts = []
    for i, sh in enumerate([(2, 16, 32, 32), (2, 16, 32, 32), (2, 32, 16, 16), (2, 64, 8, 8)]):
        t = torch.empty(sh, device=dev)
        net.wresnet_activation(i, t)
        acts.append(t.cpu().numpy())
    for i, blk in enumerate(net_p["blocks"]):
        _check_block(blk, acts[i], acts[i + 1], 3, net_p["thr_w"])
    assert np.array_equal(logits.cpu().numpy(), N.wresnet_head(net_p, acts[-1]))
    net.close()
