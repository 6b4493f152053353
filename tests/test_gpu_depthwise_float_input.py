"""The tensor between an expansion and its depthwise layer, stored as floats: hidden channel counts whose last store unit of 32
channels is half empty or partly padding, pixel tiles that end inside an image, one column, both strides, every weight class
of the expansion.  Tolerance: the float32 rule of the other forward tests, 1e-3 (1 + |ref|)."""
import numpy as np
import pytest

from aiq_workloads import inverted_residual_stack, gen_model, gen_images
from oracle import aiq_oracle as O
from gpu_util import binding, to_dev, assert_logits_close

pytestmark = pytest.mark.gpu


# (block input channels, expansion factor, size, stride, batch)
@pytest.mark.parametrize("cin,t,hw,stride,batch", [(16, 1, 8, 1, 1), (16, 3, 9, 2, 5), (24, 6, 7, 1, 19), (40, 2, 13, 2, 3), (24, 5, 33, 1, 2),
                                                   (160, 6, 4, 1, 33)])
def test_expansion_to_depthwise_in_floats(cin, t, hw, stride, batch):
    aiq = binding()
    arch = inverted_residual_stack(cin, 32, hw, stride, t=t)
    params = gen_model(arch, 9700 + cin + hw)
    x = gen_images(batch, 3, hw, hw, 9701)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8, 16, 32))
    model = aiq.Model(arch, params)
    for sc in ([8, 4, 8, 8, 8], [8, 8, 4, 8, 8], [8, 16, 32, 8, 8], [32, 32, 8, 8, 8]):
        scheme = np.array(sc, np.uint8)
        got = model.aiq_forward(scheme, to_dev(x)).cpu().numpy()
        assert_logits_close(got, O.forward_scheme(arch, bank, scheme, x), f"{cin} x {t}, {hw}, stride {stride}, batch {batch}, {sc}")
    model.close()
