"""Dense tensor-core route (csrc/tcconv.cu): every block shape and reduction split at the sizes where it can go wrong -
ragged last tiles of pixels and channels, one pipeline stage and more stages than the ring holds, channels that are not a
multiple of 16 bytes, padding, strides - against the oracle."""
import numpy as np
import pytest
import torch

from oracle import forward as oracle_forward, ref
from workloads import gen, models
from parity import NET_FLOOR, assert_close_f32, assert_close_or_bounded, assert_exact, launches_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (pixels, channels, split) of a block; None = the library's own choice
SHAPES = ["128,64,1", "128,64,4", "16,128,1", "48,128,8", "64,128,1", "64,128,16", "80,128,2", "128,128,1", "128,128,4", "256,128,1", None]
# n, h, w, c_in, c_out, k, stride, pad
LAYERS = [(1, 7, 7, 32, 64, 1, 1, 0), (2, 9, 11, 40, 130, 3, 1, 1), (1, 14, 13, 67, 65, 3, 2, 1), (3, 10, 6, 3, 70, 5, 1, 2),
          (1, 13, 13, 304, 129, 3, 1, 0), (17, 1, 1, 1027, 200, 1, 1, 0)]


def _pack(B, monkeypatch, shape, dtype, layer, w, mask):
    n, h, wd, c_in, c_out, k, stride, pad = layer
    if shape:
        monkeypatch.setenv("CADNN_TCV", shape)
    d = B.make_desc(c_in, c_out, k, k, stride, pad, 1, h, wd, n, dtype)
    return (B.cadnn_pack_q8 if dtype == "s8" else B.cadnn_pack)(d, w, mask)


@pytest.mark.parametrize("layer", LAYERS)
@pytest.mark.parametrize("shape", SHAPES)
def test_float_layers(shape, layer, monkeypatch):
    from paper_1905_00571_b200 import binding as B
    n, h, wd, c_in, c_out, k, stride, pad = layer
    g = gen.rng(41 + c_in)
    x = gen.normal_input(g, (n, h, wd, c_in))
    w = gen.he_weights(g, c_out, k, k, c_in)
    mask = gen.random_mask(g, w.shape, 0.2)
    scale, bias = gen.folded_bn(g, c_out)
    res = gen.normal_input(g, ref.conv2d_f32(x, w, mask, stride, pad).shape)
    want = ref.conv2d_f32(x, w, mask, stride, pad, 1, scale, bias, res, "relu")
    wh = _pack(B, monkeypatch, shape, "f32", layer, w, mask)
    y = torch.full(want.shape, -1.0, device=DEV)
    dev = lambda a: torch.from_numpy(a).to(DEV)
    B.cadnn_conv2d(wh, dev(x), y, dev(scale), dev(bias), dev(res), "relu")
    torch.cuda.synchronize()
    s_abs = ref.conv2d_f32(np.abs(x), np.abs(w) * mask, None, stride, pad, 1, np.abs(scale), np.abs(bias), np.abs(res), "none")
    assert_close_or_bounded(y.cpu().numpy(), want, s_abs, int(mask.reshape(c_out, -1).sum(1).max()) + 4, "%s %s" % (layer, shape))
    assert B.cadnn_device_status()["copy_timeouts"] == 0


@pytest.mark.parametrize("shape", SHAPES)
def test_all_terms_of_the_float_products_arrive(shape, monkeypatch):
    """The smallest of the split products weigh 2^-18: a result that misses them is off by 5e-6 (2-norm), one with all of them
    by about 1e-7."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(45)
    layer = (2, 12, 13, 64, 130, 3, 1, 1)
    n, h, wd, c_in, c_out, k, stride, pad = layer
    x = gen.relu_normal_input(g, (n, h, wd, c_in))
    w = gen.he_weights(g, c_out, k, k, c_in)
    mask = gen.random_mask(g, w.shape, 0.2)
    want = ref.conv2d_f32(x, w, mask, stride, pad).astype(np.float64)
    wh = _pack(B, monkeypatch, shape, "f32", layer, w, mask)
    y = torch.zeros(want.shape, device=DEV)
    B.cadnn_conv2d(wh, torch.from_numpy(x).to(DEV), y)
    torch.cuda.synchronize()
    assert np.linalg.norm(y.cpu().numpy() - want) < 5e-7 * np.linalg.norm(want)


@pytest.mark.parametrize("layer", LAYERS)
@pytest.mark.parametrize("shape", SHAPES)
def test_int8_layers_bit_exact(shape, layer, monkeypatch):
    from paper_1905_00571_b200 import binding as B
    n, h, wd, c_in, c_out, k, stride, pad = layer
    g = gen.rng(43 + c_in)
    x = gen.int8_relu_activation(g, (n, h, wd, c_in))
    q = gen.int8_weights(g, (c_out, k, k, c_in))
    mask = gen.random_mask(g, q.shape, 0.2)
    m = (g.uniform(0.5, 1.5, size=c_out) * 2e-4).astype(np.float32)
    b = (g.standard_normal(c_out) * 3).astype(np.float32)
    dev = lambda a: torch.from_numpy(a).to(DEV)
    wh = _pack(B, monkeypatch, shape, "s8", layer, q, mask)
    r = gen.int8_relu_activation(g, ref.conv2d_s8(x, q, mask, stride, pad, out="s32").shape)
    for out, dt, res in (("s8", torch.int8, r), ("f32", torch.float32, None), ("s32", torch.int32, None)):
        want = ref.conv2d_s8(x, q, mask, stride, pad, 1, m, b, "relu", out, res, 0.4) if out != "s32" else \
            ref.conv2d_s8(x, q, mask, stride, pad, out="s32")
        y = torch.full(want.shape, 5, dtype=dt, device=DEV)
        B.cadnn_conv2d(wh, dev(x), y, dev(m), dev(b), None if res is None else dev(res), "relu", out_dtype=out, residual_scale=0.4)
        torch.cuda.synchronize()
        assert_exact(y.cpu().numpy(), want, "%s %s %s" % (layer, shape, out))
    assert B.cadnn_device_status()["copy_timeouts"] == 0


@pytest.mark.parametrize("c_off", [0, 12])
def test_channel_window_of_a_concatenation(c_off):
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(47)
    x = gen.relu_normal_input(g, (2, 8, 9, 48))
    w = gen.he_weights(g, 68, 3, 3, 48)
    mask = gen.random_mask(g, w.shape, 0.3)
    want = ref.conv2d_f32(x, w, mask, 1, 1, act="relu")
    wh = B.cadnn_pack(B.make_desc(48, 68, 3, 3, 1, 1, 1, 8, 9, 2, "f32"), w, mask)
    y = torch.full((2, 8, 9, 96), 3.0, device=DEV)
    B.cadnn_conv2d(wh, torch.from_numpy(x).to(DEV), y, act="relu", out_c_total=96, out_c_off=c_off)
    torch.cuda.synchronize()
    got = y.cpu().numpy()
    s_abs = ref.conv2d_f32(np.abs(x), np.abs(w) * mask, None, 1, 1)
    assert_close_or_bounded(got[..., c_off:c_off + 68], want, s_abs, 48 * 9, "window")
    assert (got[..., :c_off] == 3.0).all() and (got[..., c_off + 68:] == 3.0).all()


@pytest.mark.parametrize("dtype", ["f32", "s8"])
def test_small_batch_fc_takes_the_dense_route_where_it_pays(dtype):
    """Packed for a batch of 8 (row CSR): 7 images run dense, one image sparse, both against the oracle."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(49)
    c_in, c_out = 1027, 1201
    mask = gen.random_mask(g, (c_out, 1, 1, c_in), 0.5)
    dev = lambda a: torch.from_numpy(a).to(DEV)
    d = B.make_desc(c_in, c_out, batch_hint=8, dtype=dtype)
    for n in (7, 1):
        if dtype == "s8":
            x = gen.int8_relu_activation(g, (n, c_in))
            q = gen.int8_weights(g, (c_out, 1, 1, c_in))
            m = (g.uniform(0.5, 1.5, size=c_out) * 2e-4).astype(np.float32)
            b = (g.standard_normal(c_out) * 3).astype(np.float32)
            want = ref.fc_s8(x, q.reshape(c_out, c_in), mask.reshape(c_out, c_in), m, b, "relu", "s8")
            y = torch.zeros((n, c_out), dtype=torch.int8, device=DEV)
            B.cadnn_fc(B.cadnn_pack_q8(d, q, mask), dev(x), y, dev(m), dev(b), act="relu")
            torch.cuda.synchronize()
            assert_exact(y.cpu().numpy(), want, "fc s8, batch %d" % n)
        else:
            x = gen.normal_input(g, (n, 1, 1, c_in))
            w = gen.he_weights(g, c_out, 1, 1, c_in)
            want = ref.conv2d_f32(x, w, mask).reshape(n, c_out)
            s_abs = ref.conv2d_f32(np.abs(x), np.abs(w) * mask, None).reshape(n, c_out)
            y = torch.zeros((n, c_out), device=DEV)
            B.cadnn_fc(B.cadnn_pack(d, w, mask), dev(x.reshape(n, c_in)), y)
            torch.cuda.synchronize()
            assert_close_or_bounded(y.cpu().numpy(), want, s_abs, c_in, "fc f32, batch %d" % n)


@pytest.mark.parametrize("shape", ["128,64,1", "16,128,1", "128,128,1", "256,128,1", None])
@pytest.mark.parametrize("h,w,c_in,k", [(5, 5, 1, 3), (3, 5, 3, 3), (7, 3, 7, 1), (5, 7, 9, 3), (9, 1, 35, 1), (6, 7, 3, 5)])
def test_int8_tensors_that_end_inside_a_word(h, w, c_in, k, shape, monkeypatch):
    """Sizes of 1, 2 and 3 modulo 4 bytes: the last bytes are fetched one by one, nothing behind the tensor is read, and they
    take part in the result (bytes of another value follow them here)."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(59 + c_in)
    size = h * w * c_in
    x = np.ascontiguousarray(gen.int8_image(g, (1, h, w, c_in)))
    q = gen.int8_weights(g, (70, k, k, c_in))
    want = ref.conv2d_s8(x, q, None, 1, k // 2, out="s32")
    wh = _pack(B, monkeypatch, shape, "s8", (1, h, w, c_in, 70, k, 1, k // 2), q, None)
    flat = torch.full((size + 64,), 77, dtype=torch.int8, device=DEV)
    flat[:size] = torch.from_numpy(x.reshape(-1)).to(DEV)
    y = torch.zeros(want.shape, dtype=torch.int32, device=DEV)
    B.cadnn_conv2d(wh, flat[:size].view(1, h, w, c_in), y, out_dtype="s32")
    torch.cuda.synchronize()
    assert_exact(y.cpu().numpy(), want, "%d bytes" % size)


def test_no_memory_for_the_dense_image_leaves_the_sparse_route():
    """The dense image (200 MB here) is optional: with 100 MB of device memory left the layer packs all the same, and computes
    what it computes with the image."""
    from paper_1905_00571_b200 import binding as B
    g = np.random.default_rng(63)
    n, c_in, c_out = 16, 8192, 4096
    w = g.standard_normal((c_out, 1, 1, c_in), dtype=np.float32) * np.float32(0.02)
    mask = (g.random(w.shape, dtype=np.float32) < 0.03).astype(np.uint8)
    x = torch.from_numpy(g.standard_normal((n, c_in), dtype=np.float32)).to(DEV)
    d = B.make_desc(c_in, c_out, batch_hint=n)
    y = [torch.zeros((n, c_out), device=DEV) for _ in range(2)]
    B.cadnn_fc(B.cadnn_pack(d, w, mask), x, y[0])
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (100 << 20), dtype=torch.uint8, device=DEV)
    try:
        wh = B.cadnn_pack(d, w, mask)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert B.cadnn_weights_info(wh)["packed_bytes"] < 100 << 20
    B.cadnn_fc(wh, x, y[1])
    torch.cuda.synchronize()
    # two sums of at most 330 products in different orders: each within 330 * 2^-24 of sum |w x|
    s_abs = x.abs().cpu().numpy().astype(np.float64) @ np.abs(w * mask).reshape(c_out, c_in).astype(np.float64).T
    terms = int(mask.reshape(c_out, -1).sum(1).max())
    assert (np.abs(y[0].cpu().numpy().astype(np.float64) - y[1].cpu().numpy()) <= 2 * terms * 2.0 ** -24 * s_abs).all()


@pytest.mark.parametrize("kind", ["conv f32", "conv stride 2", "conv s8", "fc f32", "fc s8, small batch"])
def test_reported_bytes_cover_the_device_memory_of_a_handle(kind):
    """packed_bytes against the fall of the device's free memory over twenty handles.  An allocation
    takes at most 2 MB more than asked for, and a handle has three: its images, its dense image, its parity form."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(65)
    s8 = "s8" in kind
    if kind.startswith("fc"):
        d, shape = B.make_desc(2048, 1000, batch_hint=8 if "small" in kind else 32, dtype="s8" if s8 else "f32"), (1000, 1, 1, 2048)
    else:
        d, shape = B.make_desc(256, 250, 3, 3, 2 if "2" in kind.split()[-1] else 1, 1, 1, 14, 14, 1, "s8" if s8 else "f32"), (250, 3, 3, 256)
    w = gen.int8_weights(g, shape) if s8 else gen.he_weights(g, *shape)
    mask = gen.random_mask(g, shape, 0.3)
    pack = B.cadnn_pack_q8 if s8 else B.cadnn_pack
    first = pack(d, w, mask)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    n = 20
    handles = [pack(d, w, mask) for _ in range(n)]
    used = (free - torch.cuda.mem_get_info()[0]) / n
    told = B.cadnn_weights_info(handles[0])["packed_bytes"]
    assert told == B.cadnn_weights_info(first)["packed_bytes"]
    dense = (250 + 63) // 64 * 64 * 9 * 256 * (1 if s8 else 6) if kind.startswith("conv") else 1024 * 2048 * (1 if s8 else 6)
    assert told >= dense, (told, dense)
    assert told <= used + 2 ** 21 and used <= told + 3 * 2 ** 21, (told, used)


@pytest.mark.parametrize("dtype", ["f32", "s8"])
@pytest.mark.parametrize("shape", ["48,128,16", "16,128,16", "112,128,16", "32,128,4", "128,64,2"])
def test_shares_of_a_split_tile(shape, dtype, monkeypatch):
    """A split tile's blocks finish 3, 1, 7, 8 and 64 pixels each (sums sent one, four, ... at a time, a block's own share stored),
    with a residual that they ask for ahead, on a map whose last tile is ragged."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(53)
    layer = (2, 11, 7, 64, 136, 3, 1, 1)
    n, h, wd, c_in, c_out, k, stride, pad = layer
    dev = lambda a: torch.from_numpy(a).to(DEV)
    mask = gen.random_mask(g, (c_out, k, k, c_in), 0.2)
    if dtype == "s8":   # 18 x 128 values of K: 64-channel stages of two taps
        layer = (2, 11, 7, 256, 136, 3, 1, 1)
        c_in, mask = 256, gen.random_mask(g, (c_out, k, k, 256), 0.2)
        x, q = gen.int8_relu_activation(g, (n, h, wd, c_in)), gen.int8_weights(g, (c_out, k, k, c_in))
        m = (g.uniform(0.5, 1.5, size=c_out) * 2e-4).astype(np.float32)
        b = (g.standard_normal(c_out) * 3).astype(np.float32)
        r = gen.int8_relu_activation(g, (n, h, wd, c_out))
        want = ref.conv2d_s8(x, q, mask, stride, pad, 1, m, b, "relu", "s8", r, 0.4)
        wh = _pack(B, monkeypatch, shape, dtype, layer, q, mask)
        y = torch.full(want.shape, 5, dtype=torch.int8, device=DEV)
        B.cadnn_conv2d(wh, dev(x), y, dev(m), dev(b), dev(r), "relu", out_dtype="s8", residual_scale=0.4)
        torch.cuda.synchronize()
        assert_exact(y.cpu().numpy(), want, shape)
    else:
        x, w = gen.relu_normal_input(g, (n, h, wd, c_in)), gen.he_weights(g, c_out, k, k, c_in)
        scale, bias = gen.folded_bn(g, c_out)
        r = gen.normal_input(g, (n, h, wd, c_out))
        want = ref.conv2d_f32(x, w, mask, stride, pad, 1, scale, bias, r, "relu")
        wh = _pack(B, monkeypatch, shape, dtype, layer, w, mask)
        y = torch.full(want.shape, -1.0, device=DEV)
        B.cadnn_conv2d(wh, dev(x), y, dev(scale), dev(bias), dev(r), "relu")
        torch.cuda.synchronize()
        s_abs = ref.conv2d_f32(np.abs(x), np.abs(w) * mask, None, stride, pad, 1, np.abs(scale), np.abs(bias), np.abs(r), "none")
        assert_close_or_bounded(y.cpu().numpy(), want, s_abs, int(mask.reshape(c_out, -1).sum(1).max()) + 4, shape)
    assert B.cadnn_device_status()["copy_timeouts"] == 0


# n, h, w, c_in, c_out, kh, kw, stride, pad, pad_w
ENGINE_LAYERS = [(3, 9, 7, 64, 80, 3, 3, 1, 1, 1), (2, 13, 10, 192, 96, 1, 7, 1, 0, 3), (2, 10, 13, 64, 130, 7, 1, 1, 3, 0), (3, 15, 12, 128, 64, 3, 3, 2, 1, 1),
                 (2, 17, 20, 64, 48, 3, 5, 3, 1, 2), (2, 23, 21, 128, 72, 7, 7, 4, 6, 5), (1, 12, 9, 64, 80, 1, 9, 1, 0, 8),
                 (5, 9, 11, 64, 64, 1, 1, 2, 0, 0), (1, 8, 8, 64, 48, 5, 5, 1, 0, 0), (2, 6, 5, 128, 70, 3, 5, 1, 2, 0), (33, 1, 1, 320, 200, 1, 1, 1, 0, 0)]


@pytest.mark.parametrize("shape", ["128,64,1", "48,128,1", "128,128,2", "256,128,1", None])
@pytest.mark.parametrize("layer", ENGINE_LAYERS)
def test_int8_rows_by_the_copy_engine(layer, shape, monkeypatch):
    """Layers of whole 64-channel rows: tiles that begin and end inside a row of the map and run over images, rectangular windows with
    different paddings, strides of up to four, a last stage of one half, against float64 sums and against the general gather (one channel
    more); the kernels' names tell which ran."""
    from paper_1905_00571_b200 import binding as B
    n, h, wd, c_in, c_out, kh, kw, stride, pad, pad_w = layer
    g = gen.rng(59 + c_in + kw)
    x, q = gen.int8_relu_activation(g, (n, h, wd, c_in)), gen.int8_weights(g, (c_out, kh, kw, c_in))
    mask = gen.random_mask(g, q.shape, 0.2)
    if shape:
        monkeypatch.setenv("CADNN_TCV", shape)
    dev = lambda a: torch.from_numpy(a).to(DEV)
    outs = []
    for extra in (0, 1):   # an odd number of channels takes the general gather
        xs, qs, ms = (np.pad(a, [(0, 0)] * 3 + [(0, extra)]) for a in (x, q, mask))
        # (whole numbers below 2^53 in double: exact; the int8 oracle has one padding for both axes)
        want = torch.nn.functional.conv2d(torch.from_numpy(xs).double().permute(0, 3, 1, 2), torch.from_numpy(qs * ms).double().permute(0, 3, 1, 2), None,
                                          stride, (pad, pad_w)).permute(0, 2, 3, 1).to(torch.int32).numpy()
        wh = B.cadnn_pack_q8(B.make_desc(c_in + extra, c_out, kh, kw, stride, pad, 1, h, wd, n, "s8", pad_w=pad_w), qs, ms)
        y = torch.full(want.shape, 5, dtype=torch.int32, device=DEV)
        xd = dev(xs)
        names = launches_of(lambda: B.cadnn_conv2d(wh, xd, y, out_dtype="s32"))
        own = "6GatherE0" if extra else "6GatherE2" if shape else "6GatherE1"   # (small layers that do not overlap, as in a graph: the gather)
        assert len(names) == 1 and "tcconv_kernel" in names[0][0] and own in names[0][0], names
        assert_exact(y.cpu().numpy(), want, "%s %s" % (layer, shape))
        outs.append(y.cpu().numpy())
    assert (outs[0] == outs[1]).all()
    assert B.cadnn_device_status()["copy_timeouts"] == 0


@pytest.mark.parametrize("c_out,density,dense", [(16, 0.03, False), (64, 0.03, False), (64, 0.055, False), (64, 0.065, True), (65, 0.03, True), (65, 0.02, False)])
def test_float_layers_of_up_to_64_channels_take_the_dense_route_from_six_per_cent_on(c_out, density, dense):
    """Below, the sparse kernels' sums keep every bit of activations of any magnitude (the split products lose bits below 8e-34)."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(61)
    x, w = gen.relu_normal_input(g, (2, 9, 8, 72)), gen.he_weights(g, c_out, 3, 3, 72)
    mask = gen.random_mask(g, w.shape, density)
    wh = B.cadnn_pack(B.make_desc(72, c_out, 3, 3, 1, 1, 1, 9, 8, 2, "f32"), w, mask)
    assert (B.cadnn_weights_info(wh)["packed_bytes"] > 6 * w.size) == dense
    terms = int(mask.reshape(c_out, -1).sum(1).max()) + 4
    for xs in (x,) if dense else (x, x * np.float32(1e-35)):
        want = ref.conv2d_f32(xs, w, mask, 1, 1, act="relu")
        y = torch.zeros(want.shape, device=DEV)
        B.cadnn_conv2d(wh, torch.from_numpy(xs).to(DEV), y, act="relu")
        torch.cuda.synchronize()
        got, s_abs = y.cpu().numpy(), ref.conv2d_f32(np.abs(xs), np.abs(w) * mask, None, 1, 1)
        assert_close_or_bounded(got, want, s_abs, terms, "%d %g" % (c_out, density))
        # fewer than `terms` fused multiply-adds, each within 2^-24 of a sum that the magnitudes bound, and the oracle's own rounding
        assert dense or (np.abs(got.astype(np.float64) - want) <= (terms + 1) * 2.0 ** -24 * s_abs.astype(np.float64)).all()


@pytest.mark.parametrize("batch,c,planar", [(2, 304, True), (2, 528, True), (2, 576, False), (1, 1152, False)])
def test_layout_of_networks_with_depthwise_layers(batch, c, planar):
    """A pointwise, a depthwise and a pointwise layer, with kept multiply-adds on both sides of the line: up to it the planar kernels' 32-bit
    sums, whatever the batch."""
    from paper_1905_00571_b200 import binding as B
    from paper_1905_00571_b200.network import PackedModel
    from test_gpu_fused_depthwise import _add
    g = gen.rng(63)
    hw = (48, 48)
    m = models.Model("dw_layout", "f32", (96, 96, 3), seed=63)
    stem, at = _add(m, g, "stem", 0, 3, 40, 3, 3, 2, 1, 1, m.in_shape[:2], "relu", 1.0)
    assert at == hw
    a, _ = _add(m, g, "expand", stem, 40, c, 1, 1, 1, 0, 0, hw, "relu6", 0.99)
    b, hw2 = _add(m, g, "dw", a, c, c, 3, 3, 1, 1, 1, hw, "relu6", 1.0, groups=c)
    d, _ = _add(m, g, "project", b, c, 20, 1, 1, 1, 0, 0, hw2, "none", 0.99)
    pool = m.new_slot()
    m.ops.append(models.Op("gavgpool", "pool", d, pool, c_in=20, c_out=20, in_hw=hw2, out_hw=(1, 1)))
    m.ops.append(models.Op("fc", "fc", pool, m.new_slot(), -1, 20, 10, 1, 1, 0, 1, "none", gen.he_weights(g, 10, 1, 1, 20), None,
                           np.ones(10, np.float32), np.zeros(10, np.float32), "f32", 1.0, (1, 1), (1, 1)))
    kept = batch * sum(int(op.mask.sum()) * op.out_hw[0] * op.out_hw[1] for op in m.ops if op.mask is not None)
    assert planar == (kept <= 150e6) and 0.54 < kept / 150e6 < 1.12
    x = models.make_input(m, batch)
    pm = PackedModel(m, batch, DEV)
    assert B.cadnn_net_layout(pm.net)["planar"] == planar
    y = pm.new_output()
    pm.forward(torch.from_numpy(x).to(DEV), y)
    torch.cuda.synchronize()
    want, _ = oracle_forward.forward(m, x)
    assert_close_f32(y.cpu().numpy(), want, "logits", floor=NET_FLOOR)


@pytest.mark.parametrize("shape", ["128,64,1", "32,128,1", "64,128,2"])
@pytest.mark.parametrize("act", ["none", "relu", "relu6"])
def test_float_epilogue_of_nan_infinities_and_zeros(act, shape, monkeypatch):
    """The activation as act_f32 defines it (z > 0 ? z : 0, then at most 6), whatever joins through the residual."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(67)
    w = gen.he_weights(g, 72, 1, 1, 64)
    monkeypatch.setenv("CADNN_TCV", shape)
    wh = B.cadnn_pack(B.make_desc(64, 72, 1, 1, 1, 0, 1, 5, 7, 1, "f32"), w, gen.random_mask(g, w.shape, 0.2))
    r = np.resize(np.array([np.nan, np.inf, -np.inf, -0.0, 0.0, 3.0, -3.0, 7.0, 6.0, 1e-40], np.float32), (1, 5, 7, 72))
    for scale in (1.0, -1.0):   # with -1 the sum is -0 before the residual joins
        y = torch.full(r.shape, 9.0, device=DEV)
        B.cadnn_conv2d(wh, torch.zeros((1, 5, 7, 64), device=DEV), y, torch.full((72,), scale, device=DEV), torch.full((72,), -0.0, device=DEV),
                       torch.from_numpy(r).to(DEV), act)
        torch.cuda.synchronize()
        want = r + (np.float32(0.0) * np.float32(scale) + np.float32(-0.0))
        if act != "none":
            want = np.where(want > 0, want, np.float32(0.0))
        if act == "relu6":
            want = np.minimum(want, np.float32(6.0))
        got = y.cpu().numpy()
        assert np.array_equal(got, want, equal_nan=True)
        assert (np.signbit(got) == np.signbit(want))[want == 0].all() and (want[r == 0] == 0).all()


@pytest.mark.parametrize("act", ["none", "relu"])
def test_int8_epilogue_of_nan_infinities_and_ties(act):
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(69)
    b = np.resize(np.array([np.nan, np.inf, -np.inf, 0.5, 1.5, -0.5, -2.5, 126.5, 127.5, -126.5, -200.0, 1e30], np.float32), 96)
    q = gen.int8_weights(g, (96, 1, 1, 64))
    wh = B.cadnn_pack_q8(B.make_desc(64, 96, 1, 1, 1, 0, 1, 5, 7, 1, "s8"), q, gen.random_mask(g, q.shape, 0.2))
    r = gen.int8_weights(g, (1, 5, 7, 96))
    for res in (None, r):
        y = torch.full(r.shape, 9, dtype=torch.int8, device=DEV)
        B.cadnn_conv2d(wh, torch.zeros((1, 5, 7, 64), dtype=torch.int8, device=DEV), y, torch.ones(96, device=DEV), torch.from_numpy(b).to(DEV),
                       None if res is None else torch.from_numpy(res).to(DEV), act, out_dtype="s8", residual_scale=1.0)
        torch.cuda.synchronize()
        t = np.broadcast_to(b, r.shape) if res is None else (b + res.astype(np.float32))   # (sums of halves: exact, or beyond the clamp)
        t = np.where(t > 0, t, np.float32(0.0)) if act == "relu" else t
        want = np.rint(np.fmin(np.fmax(t, np.float32(-127.0)), np.float32(127.0))).astype(np.int8)
        assert (y.cpu().numpy() == want).all()


def test_one_handle_with_and_without_a_residual():
    """The residual tile of an int8 layer takes shared memory, so the block shape may differ: whichever call comes first, each runs the
    shape that a handle of its own would."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(71)
    n, hw, c_in, c_out = 4, 56, 512, 64
    x, q = gen.int8_relu_activation(g, (n, hw, hw, c_in)), gen.int8_weights(g, (c_out, 3, 3, c_in))
    mask = gen.random_mask(g, q.shape, 0.1)
    r = torch.from_numpy(gen.int8_relu_activation(g, (n, hw, hw, c_out))).to(DEV)
    xd, m, b = torch.from_numpy(x).to(DEV), torch.full((c_out,), 3e-4, device=DEV), torch.zeros(c_out, device=DEV)
    ran = {}
    for order in ((False, True), (True, False)):
        wh = B.cadnn_pack_q8(B.make_desc(c_in, c_out, 3, 3, 1, 1, 1, hw, hw, n, "s8"), q, mask)
        for res in order:
            y = torch.zeros((n, hw, hw, c_out), dtype=torch.int8, device=DEV)
            call = lambda: B.cadnn_conv2d(wh, xd, y, m, b, r if res else None, "relu", out_dtype="s8", residual_scale=0.5)
            names = launches_of(call)
            assert len(names) == 1 and "tcconv_kernel" in names[0][0], names
            ran.setdefault(res, []).append((names, y.cpu().numpy()))
    for res in (False, True):
        (first, a), (second, c) = ran[res]
        assert first == second, (res, first, second)
        assert (a == c).all()
    assert ran[False][0][0] != ran[True][0][0]   # (the layer is one where the two choices differ)


@pytest.mark.parametrize("n,hw,c_in,c_out,k,engine", [(1, 7, 64, 64, 1, False), (16, 1, 2048, 1000, 1, False), (1, 28, 128, 320, 1, False), (1, 28, 128, 384, 1, True),
                                                      (1, 14, 512, 576, 3, False), (1, 14, 512, 704, 3, True)])
def test_small_int8_layers_that_overlap_nothing_run_on_the_gather(n, hw, c_in, c_out, k, engine):
    """On both sides of the two lines, 300 thousand outputs and 600 million multiply-adds, in a captured graph, and called one by one, where a
    layer's start overlaps the one before it and the copy engine takes them all: the same bytes."""
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(79)
    x, q = gen.int8_relu_activation(g, (n, hw, hw, c_in)), gen.int8_weights(g, (c_out, k, k, c_in))
    mask = gen.random_mask(g, q.shape, 0.1)
    wh = B.cadnn_pack_q8(B.make_desc(c_in, c_out, k, k, 1, k // 2, 1, hw, hw, n, "s8"), q, mask)
    want = ref.conv2d_s8(x, q, mask, 1, k // 2, out="s32")
    y, xd = torch.zeros(want.shape, dtype=torch.int32, device=DEV), torch.from_numpy(x).to(DEV)
    B.cadnn_conv2d(wh, xd, y, out_dtype="s32")
    torch.cuda.synchronize()
    assert_exact(y.cpu().numpy(), want, "called")
    y.zero_()
    names = launches_of(lambda: B.cadnn_conv2d(wh, xd, y, out_dtype="s32"))
    assert len(names) == 1 and ("6GatherE2" if engine else "6GatherE1") in names[0][0], names
    assert_exact(y.cpu().numpy(), want, "captured")
