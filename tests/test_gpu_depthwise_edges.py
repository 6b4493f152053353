"""Depthwise 3x3 at the edges of its tiling (column tiles, images per block, channel slabs, row blocks), against the
oracle: one or two columns, odd sizes at stride 2, a row wider than one column tile, 16 / 48 / 64-channel slabs with
padding channels, one image and a batch that does not fill the last image group.  Tolerance: the float32 rule of the
other forward tests, 1e-3 (1 + |ref|)."""
import numpy as np
import pytest

from aiq_workloads import depthwise_stack, gen_model, gen_images
from oracle import aiq_oracle as O
from gpu_util import binding, to_dev, assert_logits_close, compute_path

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["fp32", "tensor"])
@pytest.mark.parametrize("hw,channels,batch", [(2, 16, 1), (7, 36, 19), (17, 64, 9), (20, 96, 5), (130, 20, 2), (232, 16, 1)])
def test_depthwise_tile_edges(hw, channels, batch, path):
    aiq = binding()
    arch = depthwise_stack(hw, channels)
    params = gen_model(arch, 9500 + hw)
    x = gen_images(batch, 3, hw, hw, 9600 + hw)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8, 16, 32))
    with compute_path(path):
        model = aiq.Model(arch, params)
    for sc in ([8, 8, 8, 4, 8], [8, 16, 8, 32, 8]):
        ref = O.forward_scheme(arch, bank, np.array(sc, np.uint8), x)
        got = model.aiq_forward(np.array(sc, np.uint8), to_dev(x)).cpu().numpy()
        assert_logits_close(got, ref, f"depthwise stack {hw} {channels} {batch} {path} {sc}")
    model.close()


@pytest.mark.parametrize("stride,hw", [(3, 30), (4, 448)])
def test_depthwise_refuses_other_strides_as_a_shape(stride, hw):
    """Also on maps so wide that the input box of such a stride would be no legal tensor map."""
    import torch
    aiq = binding()
    arch = depthwise_stack(hw, 32)
    for l in arch["layers"]:
        if l["kind"] == "dw" and l["stride"] == 2:
            l["stride"] = stride
    model = aiq.Model(arch, gen_model(arch, 3))
    with pytest.raises(aiq.AiqError) as e:
        model.aiq_forward(np.full(len(arch["layers"]), 8, np.uint8), torch.zeros((1, 3, hw, hw), device="cuda"))
    assert e.value.status == aiq.ERR_SHAPE
    model.close()
