"""The pointwise (1x1) tensor-core kernel at the edges of its tiling, against the oracle: channel
counts that are padded (24 -> 40, 136 -> 200), a single 16-channel unit, a channel tile narrower than a store unit,
odd map sizes (border rows inside a warp's 32 pixels), one image and a batch that leaves the last pixel tile partly
empty, all four bit-widths, a shortcut into the layer; and 1,024 input channels, whose weights are
streamed.  Tolerance: the float32 rule of the other forward tests, 1e-3 (1 + |ref|)."""
import numpy as np
import pytest

from aiq_workloads import pointwise_stack, inverted_residual_stack, gen_model, gen_images
from oracle import aiq_oracle as O
from gpu_util import binding, to_dev, assert_logits_close, compute_path

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,hw,batch", [(16, 16, 5, 1), (24, 40, 7, 3), (136, 200, 13, 2), (96, 264, 4, 9),
                                               (320, 48, 9, 30), (1024, 48, 5, 3),
                                               (1032, 320, 3, 5)])
def test_pointwise_tile_edges(cin, cout, hw, batch):
    aiq = binding()
    arch = pointwise_stack(cin, cout, hw)
    params = gen_model(arch, 7500 + cin + cout)
    with compute_path("tensor"):
        model = aiq.Model(arch, params)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8, 16, 32))
    x = gen_images(batch, 3, hw, hw, 7600 + batch)
    for bits in (4, 8, 16, 32):
        scheme = np.array([8, bits, 8], np.uint8)
        got = model.aiq_forward(scheme, to_dev(x)).cpu().numpy()
        assert_logits_close(got, O.forward_scheme(arch, bank, scheme, x), f"pointwise {cin}->{cout} {hw} {batch} {bits}")
    model.close()


@pytest.mark.parametrize("c,hw", [(24, 7), (160, 5)])
def test_pointwise_shortcut(c, hw):
    aiq = binding()
    arch = inverted_residual_stack(c, c, hw, 1)
    params = gen_model(arch, 7700 + c)
    model = aiq.Model(arch, params)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8, 16, 32))
    x = gen_images(3, 3, hw, hw, 7701)
    for scheme in ([8, 16, 8, 4, 8], [8, 8, 8, 32, 8]):
        scheme = np.array(scheme, np.uint8)
        got = model.aiq_forward(scheme, to_dev(x)).cpu().numpy()
        assert_logits_close(got, O.forward_scheme(arch, bank, scheme, x), f"shortcut {c} {hw} {scheme}")
    model.close()


def test_pointwise_on_a_map_of_two_to_the_24_pixels():
    """The launch shape is searched at a nominal batch of 256 images, which here is 2^32 pixels (the search ended in a division
    by zero).  One channel of the input is a ramp down the map, so a wrong tile shows in the averages."""
    import torch
    import torch.nn.functional as F
    aiq = binding()
    H, W = 4094, 4096
    arch = pointwise_stack(24, 40, hw=8, n_classes=5)
    arch = dict(arch, in_h=H, in_w=W)
    params = gen_model(arch, 77)
    model = aiq.Model(arch, params)
    x = torch.zeros((1, 3, H, W), device="cuda")
    x[0, 0] = torch.linspace(-1, 1, H, device="cuda")[:, None]
    x[0, 1] = torch.linspace(1, -1, W, device="cuda")[None, :]
    got = model.aiq_forward(np.full(3, 8, np.uint8), x).double().cpu().numpy()
    v = x.double()
    for i, l in enumerate(arch["layers"]):
        packed, scales = model.layer_packed(i, 8)
        k = l["cin"] * l["k"] ** 2
        w = packed.view(torch.int8)[:, :k].double() * scales.double()[:, None]
        b = model.layer_folded(i)[1].double()
        if l["kind"] == "fc":
            v = v.mean((2, 3)) @ w.T + b
        else:
            v = F.conv2d(v, w.view(l["cout"], l["cin"], l["k"], l["k"]), b, l["stride"], l["pad"])
            v = v.clamp(min=0) if l["act"] == "relu" else v.clamp(0, 6) if l["act"] == "relu6" else v
    want = v.cpu().numpy()
    assert np.all(np.abs(got - want) <= 1e-3 * (1 + np.abs(want)))
    model.close()
