"""GPU parity of 2 x 2 max pools that run in the launch of the int8 layer before them: the layer's output, the pool's and the next
layer's, byte for byte, over block shapes, cluster splits, ragged tiles and rectangular maps."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import forward as oracle_forward
from workloads import gen, models
from parity import assert_exact, launches_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _add(m, g, name, src, c_in, c_out, k, stride, hw, pad=None):
    w = np.clip(np.rint(g.standard_normal((c_out, k, k, c_in)) * 40), -127, 127).astype(np.int8)
    mask = gen.random_mask(g, w.shape, 0.3)
    # (negative multipliers too: the pool takes the maximum of finished values)
    scale = (g.uniform(-1.0, 1.5, c_out) * 1.5 / np.sqrt(0.3 * k * k * c_in) / 40).astype(np.float32)
    bias = (g.standard_normal(c_out) * 10).astype(np.float32)
    pad = k // 2 if pad is None else pad
    ho = tuple((d + 2 * pad - k) // stride + 1 for d in hw)
    m.ops.append(models.Op("conv", name, src, m.new_slot(), -1, c_in, c_out, k, stride, pad, 1, "none", w, mask, scale, bias, "s8", 0.3, hw, ho))
    return m.ops[-1].dst, ho


@pytest.mark.parametrize("hw,c_in,c_out,k,stride,batch,shape,fused", [
    ((2, 2), 16, 16, 1, 1, 1, "16,128,1", True),
    ((4, 10), 16, 48, 3, 1, 3, "128,64,1", True),
    ((14, 12), 48, 80, 3, 1, 2, "128,64,4", True),
    ((14, 12), 48, 144, 3, 1, 2, "64,128,1", True),
    ((6, 18), 32, 128, 3, 1, 2, "16,128,16", True),     # 16 pixels over 16 blocks: fewer blocks, so that each has whole windows
    ((12, 20), 32, 160, 3, 1, 1, "112,128,4", True),
    ((20, 8), 24, 64, 3, 1, 2, "48,128,2", True),       # 24 input channels: gathered in runs
    ((26, 34), 3, 32, 3, 1, 1, "128,64,1", True),
    ((28, 28), 64, 96, 5, 2, 2, "128,128,2", True),
    ((28, 30), 32, 64, 1, 1, 1, "256,128,1", True),
    ((15, 14), 16, 32, 3, 1, 1, "128,64,1", False),     # odd rows, channels that are no whole pieces: pools of their own
    ((14, 14), 16, 36, 3, 1, 1, "128,64,1", False),
])
def test_pool_behind_int8_layer(hw, c_in, c_out, k, stride, batch, shape, fused, monkeypatch):
    _check(hw, c_in, c_out, k, stride, batch, shape, fused, monkeypatch)


@pytest.mark.parametrize("hw,c_in,c_out,k,stride,pad,batch,shape", [
    ((14, 12), 64, 80, 3, 1, 1, 3, "32,128,1"),       # 42 windows an image: tiles of 8 run over rows and images, the last one is ragged
    ((14, 12), 192, 96, 3, 1, 1, 3, "96,128,1"),      # 27 halves of a stage: the last stage has one
    ((10, 6), 64, 48, 1, 1, 0, 5, "192,128,1"),       # one stage of one half; a tile holds three images
    ((20, 14), 64, 64, 5, 1, 2, 2, "256,128,1"),
    ((22, 10), 128, 64, 3, 1, 1, 2, "128,64,1"),
    ((24, 20), 64, 96, 3, 2, 1, 3, "64,128,1"),       # windows 4, 6 and 8 positions apart
    ((18, 30), 64, 48, 3, 3, 1, 2, "128,128,1"),
    ((32, 24), 128, 64, 5, 4, 2, 3, "32,128,1"),
    ((16, 12), 64, 32, 3, 1, 0, 3, "160,128,1"),      # no padding
    ((9, 13), 64, 64, 4, 1, 3, 2, "96,128,1"),        # more padding than the window's middle, odd maps
    ((2, 2), 64, 16, 3, 1, 1, 9, "32,128,1"),         # one window an image
    ((56, 40), 64, 160, 3, 1, 1, 2, None),
])
def test_pool_behind_int8_layer_gathered_by_the_copy_engine(hw, c_in, c_out, k, stride, pad, batch, shape, monkeypatch):
    """Unsplit tiles of whole 64-channel rows, a quarter of a tile's rows for each place in a window."""
    _check(hw, c_in, c_out, k, stride, batch, shape, True, monkeypatch, pad, True)


def _check(hw, c_in, c_out, k, stride, batch, shape, fused, monkeypatch, pad=None, engine=False):
    from paper_1905_00571_b200 import binding as B
    from paper_1905_00571_b200.network import PackedModel
    if shape:
        monkeypatch.setenv("CADNN_TCV", shape)
    g = gen.rng(83)
    m = models.Model("pool_tail", "s8", (hw[0], hw[1], c_in), seed=83)
    a, at = _add(m, g, "conv", 0, c_in, c_out, k, stride, hw, pad)
    pooled = m.new_slot()
    half = (at[0] // 2, at[1] // 2)
    m.ops.append(models.Op("maxpool", "pool", a, pooled, k=2, stride=2, pad=0, c_in=c_out, c_out=c_out, out="s8", in_hw=at, out_hw=half))
    _add(m, g, "next", pooled, c_out, 32, 1, 1, half)
    x = models.make_input(m, batch)
    pm = PackedModel(m, batch, DEV)
    assert pm.launches_per_forward() == (2 if fused else 3)
    want, slots = oracle_forward.forward(m, x)
    xd = torch.from_numpy(x).to(DEV)
    y = pm.new_output()
    name, _ = launches_of(lambda: pm.forward(xd, y, use_graph=False))[0]
    assert "tcconv_kernel" in name and ("6GatherE2ELb1" in name) == engine, name   # (the copy engine's kernel, with a pool)
    for use_graph in (False, True):
        y.zero_()
        pm.forward(xd, y, use_graph=use_graph)
        torch.cuda.synchronize()
        for slot in (a, pooled):
            ptr, nbytes = B.cadnn_net_slot(pm.net, slot)
            got = np.empty(nbytes, np.int8)
            assert ctypes.CDLL("libcudart.so").cudaMemcpy(ctypes.c_void_p(got.ctypes.data), ctypes.c_void_p(ptr), ctypes.c_size_t(nbytes), 2) == 0
            assert_exact(got.reshape(slots[slot].shape), slots[slot], "slot %d" % slot)
        assert_exact(y.cpu().numpy(), want, "output")
