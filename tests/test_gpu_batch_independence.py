"""An image's logits do not depend, bit for bit, on the batch around it: the launch shapes of the pointwise layers and of the
classifier may change with the batch, the order of their sums may not."""
import numpy as np
import pytest

from aiq_workloads import gen_model, gen_images, pointwise_stack, mobilenet_v2, mixed_int4_int8_scheme, conv_layer_indices
from gpu_util import binding, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,classes", [(64, 384, 10), (160, 960, 33), (960, 320, 1000), (96, 576, 70)])
def test_logits_do_not_depend_on_the_batch(cin, cout, classes):
    aiq = binding()
    arch = pointwise_stack(cin, cout, hw=8, n_classes=classes)
    model = aiq.Model(arch, gen_model(arch, 9900 + cin))
    x = gen_images(256, 3, 8, 8, 9901)
    for sc in ([8, 8, 8], [16, 4, 16]):
        scheme = np.array(sc, np.uint8)
        full = model.aiq_forward(scheme, to_dev(x)).cpu().numpy()
        for batch in (1, 4, 5, 17, 64):
            part = model.aiq_forward(scheme, to_dev(x[:batch])).cpu().numpy()
            assert np.array_equal(part, full[:batch]), (sc, batch)
    model.close()


def test_mobilenet_v2_logits_and_predictions_do_not_depend_on_the_batch():
    """The whole network, on either side of one wave of 8 x 8 images (128 to one per SM), as a forward pass and as chunks of
    an evaluation."""
    import torch
    aiq = binding()
    arch = mobilenet_v2("cifar")
    model = aiq.Model(arch, gen_model(arch, 9911))
    L = len(arch["layers"])
    schemes = np.stack([np.full(L, 8, np.uint8), mixed_int4_int8_scheme(L, conv_layer_indices(arch), 10, 43)])
    x = to_dev(gen_images(149, 3, 32, 32, 9912))
    for scheme in schemes:
        full = model.aiq_forward(scheme, x).cpu().numpy()
        for batch in (1, 32, 100, 127, 128, 140, 148):
            part = model.aiq_forward(scheme, x[:batch].contiguous()).cpu().numpy()
            assert np.array_equal(part, full[:batch]), batch
        want = full.argmax(1)
        labels = torch.zeros(149, dtype=torch.int32, device="cuda")
        for chunk in (50, 128, 149):
            preds = torch.empty((1, 149), dtype=torch.int32, device="cuda")
            aiq.aiq_set_eval_options(chunk, True)
            try:
                model.aiq_eval_schemes(scheme[None], x, labels, preds=preds, chunk=chunk)
            finally:
                aiq.aiq_set_eval_options(0, True)
            assert np.array_equal(preds[0].cpu().numpy(), want), chunk
    model.close()
