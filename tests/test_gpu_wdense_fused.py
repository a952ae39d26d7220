"""The one-kernel forward of the weight-only DenseNet-BC (wdense_fused.cu): the
growths it covers, image sizes whose tiles and feature stages have
remainders, and sizes just outside its range, every layer against the oracle;
its features next to a layer-by-layer forward's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2003_04296_gb300.inputs import wdense_params, wresnet_input  # noqa: E402
from tests._gpu import dev_tensor  # noqa: E402
from tests.test_gpu_wdense import M, _check_net, _finals, _pad64, _run, dev  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,growth,hw,B", [
    (1, 4, 8, 2),      # smallest
    (3, 4, 12, 2), (4, 8, 20, 1), (5, 12, 24, 2), (2, 12, 28, 1),
    (7, 12, 32, 2),    # odd channel multiples: features off a 4-channel boundary
    (20, 12, 16, 1),   # weights above the buffers: layer by layer
    (1, 12, 36, 1)])   # images above 32 x 32: layer by layer
def test_shapes(dev, M, layers, growth, hw, B):  # noqa: F811
    bits = 1 + (layers + hw) % 3
    net_p = wdense_params(layers + growth + hw, layers=layers, growth=growth, bits_w=bits, classes=37, hw=hw)
    x = wresnet_input(hw, B, hw=hw)
    logits, feats = _run(dev, M, net_p, x)
    _check_net(net_p, x, logits, feats, list(range(B)))


def test_batches_and_timing(dev, M):  # noqa: F811
    """More images than SMs, each image independent of the batch; a timed (layer-by-layer) forward and
    a replay in turn, with the features of whichever ran last."""
    net_p = wdense_params(7, layers=3, growth=12, bits_w=3, classes=10, hw=32)
    x = wresnet_input(8, 200, hw=32)
    big, _ = _run(dev, M, net_p, x)
    small, feats = _run(dev, M, net_p, x[190:193])
    assert np.array_equal(big[190:193], small)
    net = M.Net.wdense(net_p, 3, dev)
    xd = dev_tensor(x[190:193], dev)
    logits = torch.empty((3, 10), device=dev)

    def features():
        out = []
        for b, cf in enumerate(_finals(net_p)):
            h = 32 >> b
            t = torch.empty(3 * h * h * _pad64(cf), dtype=torch.int16, device=dev)
            net.wdense_features(b, t)
            u = t.cpu().numpy().view(np.uint16).astype(np.uint32) << 16
            out.append(np.ascontiguousarray(u.view(np.float32).reshape(3, h, h, -1)[..., :cf].transpose(0, 3, 1, 2)))
        return out

    for timed in (False, True, False, False, True):
        net.enable_timing(timed)
        net.forward(xd, logits)
        f = features()
        if timed:
            assert len(net.layer_times()) == net.launches
            _check_net(net_p, x[190:193], logits.cpu().numpy(), f, [0, 1, 2])
        else:
            assert np.array_equal(logits.cpu().numpy(), small)
            assert all(np.array_equal(a, b) for a, b in zip(f, feats))
    net.close()
