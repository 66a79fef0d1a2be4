"""The sparse kernels on everything they still run for - layers below the dense route's densities, batches beyond its index ranges,
handles without memory for its image, timed packs: the layer and network tests once more with the dense route left out, so that
sconv_kernel and the planar kernels compute what tcconv_kernel does by default (int8 residuals, channel windows and whole int8
networks among them)."""
import numpy as np
import pytest
import torch

from oracle import forward as oracle_forward
from workloads import gen, models
from parity import assert_close_f32, NET_FLOOR
from test_gpu_layers import (test_identity_1x1_is_a_copy_on_gpu, test_int8_pack_from_float_weights_matches_oracle_quantizer,  # noqa: F401
                             test_schedule_hint_does_not_change_results, test_skewed_and_empty_filters, test_sparse_1x1_conv_f32,
                             test_sparse_conv_f32, test_sparse_conv_s8_bit_exact, test_sparse_fc_f32, test_sparse_fc_s8_bit_exact)
from test_gpu_inception import (test_conv_writes_a_channel_window, test_inception_v3_reduced,  # noqa: F401
                                test_int8_conv_with_int8_residual_bit_exact, test_mobilenet_v1_reduced, test_rectangular_kernel_int8_bit_exact,
                                test_rectangular_kernels_f32, test_resnet50_int8_full_batch1, test_resnet50_int8_reduced)
from test_gpu_networks import (test_general_graph_scheduler_on_residual_networks, test_graph_with_parallel_branches_matches_layer_by_layer,  # noqa: F401
                               test_mobilenet_v2_reduced, test_resnet50_full_batch1, test_resnet50_reduced, test_vgg16_int8_full_batch1_bit_exact,
                               test_vgg16_int8_reduced_bit_exact)

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(autouse=True)
def no_dense_route(monkeypatch):
    monkeypatch.setenv("CADNN_NO_TCV", "1")


@pytest.mark.parametrize("dtype", ["f32", "s8"])
def test_no_handle_has_a_dense_image_here(dtype):
    from paper_1905_00571_b200 import binding as B
    g = gen.rng(81)
    w = gen.int8_weights(g, (128, 3, 3, 64)) if dtype == "s8" else gen.he_weights(g, 128, 3, 3, 64)
    wh = (B.cadnn_pack_q8 if dtype == "s8" else B.cadnn_pack)(B.make_desc(64, 128, 3, 3, 1, 1, 1, 14, 14, 2, dtype), w, gen.random_mask(g, w.shape, 0.03))
    assert B.cadnn_weights_info(wh)["packed_bytes"] < w.size * (1 if dtype == "s8" else 6)


def test_float_network_on_the_nhwc_sparse_kernel(monkeypatch):
    """Float residuals and stride-2 layers of a whole ResNet-50 in sconv_kernel (the planar kernels left out too)."""
    from paper_1905_00571_b200 import binding as B
    from paper_1905_00571_b200.network import PackedModel
    monkeypatch.setenv("CADNN_NO_PLANAR", "1")
    m = models.resnet50(width=0.25, image=72, classes=100)
    x = models.make_input(m, 3)
    pm = PackedModel(m, 3, DEV)
    assert not B.cadnn_net_layout(pm.net)["planar"]
    y = pm.new_output()
    pm.forward(torch.from_numpy(x).to(DEV), y)
    torch.cuda.synchronize()
    want, _ = oracle_forward.forward(m, x)
    assert_close_f32(y.cpu().numpy(), want, "logits", floor=NET_FLOOR)
    assert len({a.tobytes() for a in y.cpu().numpy()}) == 3 and np.isfinite(want).all()
