"""The stem convolution at its edges (one and four pixels per thread, rows that are no multiple of four, both strides, one to
four input channels, padded output channels, wide and unaligned rows) against the oracle, behind a depthwise layer, so that a
misplaced pixel shows.  Tolerance: the float32 rule of the other forward tests, 1e-3 (1 + |ref|)."""
import numpy as np
import pytest

from aiq_workloads import gen_model, gen_images
from oracle import aiq_oracle as O
from gpu_util import binding, to_dev, assert_logits_close, compute_path

pytestmark = pytest.mark.gpu


def _layer(name, kind, cin, cout, k, stride, act, inp):
    return dict(name=name, kind=kind, cin=cin, cout=cout, k=k, stride=stride, pad=k // 2, act=act, input=inp, residual=-1,
                has_bn=kind != "fc")


def _net(cin, cout, stride, h, w):
    layers = [_layer("stem", "conv", cin, cout, 3, stride, "relu6", -1), _layer("dw", "dw", cout, cout, 3, 1, "relu", 0),
              _layer("fc", "fc", cout, 5, 1, 1, "none", 1)]
    return dict(name="stem_edges", in_c=cin, in_h=h, in_w=w, n_classes=5, layers=layers)


@pytest.mark.parametrize("path", ["fp32", "tensor"])
@pytest.mark.parametrize("cin,cout,stride,h,w,batch", [(3, 32, 2, 12, 16, 1), (3, 24, 2, 9, 13, 3), (1, 16, 1, 7, 5, 2),
                                                       (4, 64, 1, 6, 8, 5), (3, 32, 1, 16, 16, 150), (3, 32, 2, 31, 33, 160),
                                                       (3, 12, 1, 10, 22, 200), (3, 48, 2, 20, 36, 120)])
def test_stem_edges(cin, cout, stride, h, w, batch, path):
    aiq = binding()
    arch = _net(cin, cout, stride, h, w)
    params = gen_model(arch, 9700 + h + w)
    x = gen_images(batch, cin, h, w, 9800 + batch)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8, 16, 32))
    with compute_path(path):
        model = aiq.Model(arch, params)
    sample = np.unique(np.concatenate([np.arange(min(batch, 4)), [batch - 1]]))
    for bits in (8, 4, 16, 32):
        sc = np.array([bits, 8, 8], np.uint8)
        got = model.aiq_forward(sc, to_dev(x)).cpu().numpy()
        ref = O.forward_scheme(arch, bank, sc, x[sample])
        assert_logits_close(got[sample], ref, f"stem {cin} {cout} {stride} {h}x{w} batch {batch} {path} {bits}")
    model.close()
