"""Timed packs and the dense tensor-core route: the packer times that kernel too, a handle keeps the dense image where it was
the faster one, and a network's layout follows from the times of the kernels that would run."""
import struct

import numpy as np
import pytest
import torch

from oracle import forward as oracle_forward
from oracle import ref
from workloads import gen, models
from parity import assert_close_f32, assert_exact, NET_FLOOR
from test_gpu_parity_planes import _conv

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_a_timed_network_takes_the_dense_route_where_it_is_faster():
    """Two 3x3 layers that keep 40 % on 28 x 28 maps of 32 images: several times faster on the tensor cores than on either sparse
    kernel, so the network runs NHWC whether its schedules were timed or not."""
    from paper_1905_00571_b200 import binding as B
    from paper_1905_00571_b200.network import PackedModel
    g = gen.rng(71)
    m = models.Model("timed_dense", "f32", (56, 56, 3), seed=71)
    stem, hw = _conv(m, g, "stem", 0, 3, 64, 3, 2, 1, (56, 56), "relu", 1.0)
    a, _ = _conv(m, g, "a", stem, 64, 128, 3, 1, 1, hw, "relu", 0.4)
    b, _ = _conv(m, g, "b", a, 128, 128, 3, 1, 1, hw, "relu", 0.4)
    pool = m.new_slot()
    m.ops.append(models.Op("gavgpool", "pool", b, pool, c_in=128, c_out=128, in_hw=hw, out_hw=(1, 1)))
    w = gen.he_weights(g, 10, 1, 1, 128)
    m.ops.append(models.Op("fc", "fc", pool, m.new_slot(), -1, 128, 10, 1, 1, 0, 1, "none", w, None,
                           np.ones(10, np.float32), np.zeros(10, np.float32), "f32", 1.0, (1, 1), (1, 1)))
    x = models.make_input(m, 32)
    want, _ = oracle_forward.forward(m, x)
    for autotune in (False, True):
        pm = PackedModel(m, 32, DEV, autotune=autotune)
        assert not B.cadnn_net_layout(pm.net)["planar"], autotune
        y = pm.new_output()
        pm.forward(torch.from_numpy(x).to(DEV), y)
        torch.cuda.synchronize()
        assert_close_f32(y.cpu().numpy(), want, "logits, autotune %s" % autotune, floor=NET_FLOOR)


@pytest.mark.parametrize("batch", [1, 2])
def test_a_timed_network_takes_the_layout_of_the_lower_sum(batch, tmp_path, monkeypatch):
    """The times of a cache record's layer (its last four numbers: the two planar kernels, the NHWC sparse and the dense kernel) written
    on both sides of each other: the network's layout follows the sums, a single image's as well."""
    from paper_1905_00571_b200 import binding as B
    from paper_1905_00571_b200.network import PackedModel
    cache = tmp_path / "tune.cache"
    monkeypatch.setenv("CADNN_TUNE_CACHE", str(cache))
    g = gen.rng(75)
    m = models.Model("timed_layout", "f32", (28, 28, 3), seed=75)
    stem, hw = _conv(m, g, "stem", 0, 3, 32, 3, 2, 1, (28, 28), "relu", 1.0)
    a, _ = _conv(m, g, "a", stem, 32, 96, 3, 1, 1, hw, "relu", 0.2)
    b, _ = _conv(m, g, "b", a, 96, 80, 1, 1, 0, hw, "relu", 0.2)
    pool = m.new_slot()
    m.ops.append(models.Op("gavgpool", "pool", b, pool, c_in=80, c_out=80, in_hw=hw, out_hw=(1, 1)))
    m.ops.append(models.Op("fc", "fc", pool, m.new_slot(), -1, 80, 10, 1, 1, 0, 1, "none", gen.he_weights(g, 10, 1, 1, 80), None,
                           np.ones(10, np.float32), np.zeros(10, np.float32), "f32", 1.0, (1, 1), (1, 1)))
    x = models.make_input(m, batch)
    want, _ = oracle_forward.forward(m, x)
    PackedModel(m, batch, DEV, autotune=True)
    records = [line.split() for line in cache.read_text().splitlines()]
    assert records
    for dense_us, planar in ((9.5, False), (7.0, False), (10.5, True)):
        cache.write_text("".join("%s %s\n" % (key, r[:-32] + struct.pack("<4f", 10.0, 10.0, 20.0, dense_us).hex()) for key, r in records))
        pm = PackedModel(m, batch, DEV, autotune=True)
        assert B.cadnn_net_layout(pm.net)["planar"] == planar, (dense_us, planar)
        y = pm.new_output()
        pm.forward(torch.from_numpy(x).to(DEV), y)
        torch.cuda.synchronize()
        assert_close_f32(y.cpu().numpy(), want, "logits, dense layers of %g us" % dense_us, floor=NET_FLOOR)


@pytest.mark.parametrize("dtype", ["f32", "s8"])
def test_a_timed_handle_keeps_the_dense_image_only_where_it_was_faster(dtype, tmp_path, monkeypatch):
    """The cache record's last number is the dense kernel's time: with a long one the handle holds no dense image and calls run the
    sparse kernel, with a short one it does; a record without the time is completed; results are the layer's in each case."""
    from paper_1905_00571_b200 import binding as B
    cache = tmp_path / "tune.cache"
    monkeypatch.setenv("CADNN_TUNE_CACHE", str(cache))
    g = gen.rng(73)
    x = gen.int8_relu_activation(g, (2, 9, 10, 72)) if dtype == "s8" else gen.relu_normal_input(g, (2, 9, 10, 72))
    w = gen.int8_weights(g, (70, 3, 3, 72)) if dtype == "s8" else gen.he_weights(g, 70, 3, 3, 72)
    mask = gen.random_mask(g, w.shape, 0.2)
    want = ref.conv2d_s8(x, w, mask, 1, 1, out="s32") if dtype == "s8" else ref.conv2d_f32(x, w, mask, 1, 1, act="relu")
    d = B.make_desc(72, 70, 3, 3, 1, 1, 1, 9, 10, 2, dtype, autotune=True)
    pack = B.cadnn_pack_q8 if dtype == "s8" else B.cadnn_pack
    dense = 128 * 9 * 72 * (1 if dtype == "s8" else 6)

    def check(wh, what):
        y = torch.zeros(want.shape, dtype=torch.int32 if dtype == "s8" else torch.float32, device=DEV)
        if dtype == "s8":
            B.cadnn_conv2d(wh, torch.from_numpy(x).to(DEV), y, out_dtype="s32")
        else:
            B.cadnn_conv2d(wh, torch.from_numpy(x).to(DEV), y, act="relu")
        torch.cuda.synchronize()
        (assert_exact if dtype == "s8" else assert_close_f32)(y.cpu().numpy(), want, what)
        return B.cadnn_weights_info(wh)["packed_bytes"]

    check(pack(d, w, mask), "timed")
    key, record = cache.read_text().split()
    told = {}
    for us in (1e6, 1e-3):
        cache.write_text("%s %s\n" % (key, record[:-8] + struct.pack("<f", us).hex()))
        told[us] = check(pack(d, w, mask), "%g us" % us)
        assert len(cache.read_text().splitlines()) == 1
    assert told[1e-3] - told[1e6] >= dense
    cache.write_text("%s %s\n" % (key, record[:-8] + struct.pack("<f", -1.0).hex()))
    check(pack(d, w, mask), "no time recorded")
    again = cache.read_text().split()
    assert again[2] == key and struct.unpack("<f", bytes.fromhex(again[3][-8:]))[0] > 0.0


def test_records_of_earlier_kernels_are_timed_again(tmp_path, monkeypatch):
    """A record under the key of the kernels before (the same hash without their generation), with a dense time that would drop the dense
    image: the pack does not take it, times the layer itself and adds a record of its own, which the next pack takes."""
    from paper_1905_00571_b200 import binding as B
    cache = tmp_path / "tune.cache"
    monkeypatch.setenv("CADNN_TUNE_CACHE", str(cache))
    g = gen.rng(77)
    c_in, c_out, h, wd, n = 72, 70, 9, 10, 2
    w = gen.he_weights(g, c_out, 3, 3, c_in)
    mask = gen.random_mask(g, w.shape, 0.2)
    d = B.make_desc(c_in, c_out, 3, 3, 1, 1, 1, h, wd, n, "f32", autotune=True)
    B.cadnn_pack(d, w, mask)
    key, record = cache.read_text().split()
    assert len(record) == 2 * (100 + 100 + 6 * 4 + 4 * 4)
    rows = [int(k) for k in mask.reshape(c_out, -1).astype(bool).sum(1)]

    def digest(*generation):
        v = 1469598103934665603
        for byte in struct.pack("<%dq" % (15 + len(generation) + c_out), c_in, c_out, 3, 3, 1, 1, 1, 1, h, wd, n, d.dtype, 100, 100, 240, *generation, *rows):
            v = (v ^ byte) * 1099511628211 % 2 ** 64
        return "%016x" % v

    old = digest()
    assert key != old and key in [digest(i) for i in range(2, 100)]
    slow = record[:-8] + struct.pack("<f", 1e6).hex()
    cache.write_text("%s %s\n" % (old, slow))
    B.cadnn_pack(d, w, mask)
    lines = [line.split() for line in cache.read_text().splitlines()]
    assert [k for k, _ in lines] == [old, key]
    assert 0.0 < struct.unpack("<f", bytes.fromhex(lines[1][1][-8:]))[0] < 1e3
    cache.write_text("%s %s\n" % (key, slow))
    B.cadnn_pack(d, w, mask)
    assert len(cache.read_text().splitlines()) == 1
