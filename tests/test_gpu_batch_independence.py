"""An image's logits do not depend, bit for bit, on the batch around it: the launch shapes of the pointwise layers and of the
classifier may change with the batch, the order of their sums may not."""
import numpy as np
import pytest

from aiq_workloads import gen_model, gen_images, pointwise_stack
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
