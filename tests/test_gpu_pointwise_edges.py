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
