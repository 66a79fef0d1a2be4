"""GPU parity of depthwise layers that run in the launch of the pointwise layer before them: both tensors against the oracle's walker,
at map sizes around a block's tile (32 to 256 positions of the padded map), strides, unpadded and rectangular kernels, channel counts
that do not fill the last block."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import forward as oracle_forward
from workloads import gen, models
from parity import assert_close_f32, NET_FLOOR

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _tensor(B, net, slot, shape):
    """A channel-planar feature map with its border of one pixel, as NHWC."""
    n, h, w, c = shape
    ptr, nbytes = B.cadnn_net_slot(net, slot)
    raw = np.empty(nbytes // 4, np.float32)
    assert ctypes.CDLL("libcudart.so").cudaMemcpy(ctypes.c_void_p(raw.ctypes.data), ctypes.c_void_p(ptr), ctypes.c_size_t(nbytes), 2) == 0
    pitch = ((h + 2) * (w + 2) + 3) // 4 * 4
    grid = raw[:n * c * pitch].reshape(n, c, pitch)[:, :, :(h + 2) * (w + 2)].reshape(n, c, h + 2, w + 2)
    assert np.count_nonzero(grid) == np.count_nonzero(grid[:, :, 1:h + 1, 1:w + 1]), "a plane's border was written"
    return grid[:, :, 1:h + 1, 1:w + 1].transpose(0, 2, 3, 1)


def _add(m, g, name, src, c_in, c_out, kh, kw, stride, pad, pad_w, hw, act, density, groups=1):
    w = gen.he_weights(g, c_out, kh, kw, c_in // groups)
    mask = None if density >= 1.0 else gen.random_mask(g, w.shape, density)
    scale, bias = gen.folded_bn(g, c_out, gain=1.0)
    ho = ((hw[0] + 2 * pad - kh) // stride + 1, (hw[1] + 2 * pad_w - kw) // stride + 1)
    m.ops.append(models.Op("conv", name, src, m.new_slot(), -1, c_in, c_out, kh, stride, pad, groups, act, w, mask, scale, bias, "f32",
                           density, hw, ho, pad_w=pad_w))
    return m.ops[-1].dst, ho


@pytest.mark.parametrize("hw,c,kernel,stride,pad,batch,schedule", [
    ((1, 2), 24, (3, 3), 1, 1, 2, "nw=4,ks=1,rpw=1"),
    ((2, 13), 40, (3, 3), 2, 1, 1, "nw=8,ks=2,rpw=2"),
    ((7, 7), 100, (3, 3), 1, 1, 3, "nw=4,ks=4,rpw=1"),
    ((7, 7), 960, (3, 3), 1, 1, 1, "nw=4,ks=1,rpw=2"),
    ((8, 6), 36, (2, 2), 1, 0, 1, "nw=8,ks=1,rpw=4"),
    ((9, 5), 33, (2, 3), 1, 1, 2, "nw=4,ks=2,rpw=2,chunks=2,stages=2"),
    ((11, 14), 20, (1, 2), 2, 0, 1, "nw=16,ks=2,rpw=1"),
    ((14, 14), 384, (3, 3), 1, 1, 1, "nw=4,ks=1,rpw=1"),
    ((14, 14), 64, (3, 3), 2, 1, 5, "nw=8,ks=1,rpw=2,chunks=4,stages=2"),
    ((16, 14), 48, (3, 3), 3, 1, 1, "nw=4,ks=1,rpw=1"),
    ((15, 15), 48, (3, 3), 1, 1, 1, "nw=4,ks=1,rpw=1"),
    ((28, 28), 48, (3, 3), 2, 1, 1, "nw=4,ks=1,rpw=1"),
])
def test_depthwise_behind_pointwise(hw, c, kernel, stride, pad, batch, schedule, monkeypatch):
    from paper_1905_00571_b200 import binding as B
    from paper_1905_00571_b200.network import PackedModel
    monkeypatch.setenv("CADNN_FORCE_PLANAR", "1")
    monkeypatch.setenv("CADNN_PERSIST", "0")
    # positions a block has to cover: from the first interior one (rounded down to 16 bytes) to the last
    span = hw[0] * (hw[1] + 2) + hw[1] + 1 - (hw[1] + 3) // 4 * 4
    bands = next((t for t in (1, 2, 4, 8) if 32 * t >= span), 8)
    monkeypatch.setenv("CADNN_PLANAR_SCHEDULE", "t=%d,tma=1,kc=1,chunks=1,stages=1,%s" % (bands, schedule) if "chunks" not in schedule
                       else "t=%d,tma=1,kc=1,%s" % (bands, schedule))
    g = gen.rng(71)
    m = models.Model("dw_tail", "f32", (2 * hw[0], 2 * hw[1], 3), seed=71)
    stem, at = _add(m, g, "stem", 0, 3, 16, 3, 3, 2, 1, 1, m.in_shape[:2], "relu", 1.0)
    assert at == hw
    a, _ = _add(m, g, "expand", stem, 16, c, 1, 1, 1, 0, 0, hw, "relu6", 0.3)
    b, hw2 = _add(m, g, "dw", a, c, c, kernel[0], kernel[1], stride, pad, pad, hw, "relu6", 1.0, groups=c)
    d, _ = _add(m, g, "project", b, c, 24, 1, 1, 1, 0, 0, hw2, "none", 0.3)
    pool = m.new_slot()
    m.ops.append(models.Op("gavgpool", "pool", d, pool, c_in=24, c_out=24, in_hw=hw2, out_hw=(1, 1)))
    m.ops.append(models.Op("fc", "fc", pool, m.new_slot(), -1, 24, 10, 1, 1, 0, 1, "none", gen.he_weights(g, 10, 1, 1, 24), None,
                           np.ones(10, np.float32), np.zeros(10, np.float32), "f32", 1.0, (1, 1), (1, 1)))
    x = models.make_input(m, batch)
    pm = PackedModel(m, batch, DEV)
    assert B.cadnn_net_layout(pm.net)["planar"]
    assert pm.launches_per_forward() == len(m.ops) - (32 * bands >= span)
    xd = torch.from_numpy(x).to(DEV)
    y = pm.new_output()
    want, slots = oracle_forward.forward(m, x)
    for use_graph in (False, True):
        y.zero_()
        pm.forward(xd, y, use_graph=use_graph)
        torch.cuda.synchronize()
        for slot in (a, b, d):
            assert_close_f32(_tensor(B, pm.net, slot, slots[slot].shape), slots[slot], "slot %d" % slot, floor=NET_FLOOR)
        assert_close_f32(y.cpu().numpy(), want, "logits", floor=NET_FLOOR)
