"""The one-launch bank kernel at its edges: rows longer than it keeps in registers (1,300 and 1,290 elements, the second
not a multiple of 4), layers above and below the size that is uploaded through the blob, a classifier without a bias,
9-element rows; folded weights, biases, codes and scales against the oracle, bit for bit.  A layer of 2,048-element rows
takes the per-layer kernels beside it."""
import numpy as np
import pytest

from aiq_workloads import gen_model, tiny_net
from aiq_workloads.archs import _conv, _fc
from oracle import aiq_oracle as O
from gpu_util import binding

pytestmark = pytest.mark.gpu


def _net(widths, kinds):
    layers = [_conv("stem", 3, widths[0], 3, 1, "relu6", -1)]
    for i in range(1, len(widths)):
        layers.append(_conv(f"l{i}", widths[i - 1], widths[i], kinds[i - 1], 1, "relu6", i - 1))
    layers.append(_conv("dw", widths[-1], widths[-1], 3, 1, "relu6", len(layers) - 1, kind="dw"))
    layers.append(_fc("fc", widths[-1], 7, len(layers) - 1))
    return dict(name="bank", in_c=3, in_h=8, in_w=8, n_classes=7, layers=layers)


@pytest.mark.parametrize("widths,kinds,bias", [((16, 1300, 24), (1, 1), True), ((20, 1290, 8), (1, 1), False),
                                               ((2048, 600, 12), (1, 3), True)])
def test_bank_bits(widths, kinds, bias):
    aiq = binding()
    arch = _net(widths, kinds)
    params = gen_model(arch, 9900 + widths[1])
    if not bias:
        params[-1].pop("bias")
    model = aiq.Model(arch, params)
    ref = [dict(p) for p in params]
    if not bias:
        ref[-1]["bias"] = np.zeros(7, np.float32)
    folded = O.fold_model(arch, ref)
    for i, (wf, bf) in enumerate(folded):
        got_w, got_b = model.layer_folded(i)
        wf = np.asarray(wf).reshape(got_w.shape)
        assert np.array_equal(got_w.cpu().numpy().view(np.uint32), wf.view(np.uint32)), i
        assert np.array_equal(got_b.cpu().numpy().view(np.uint32), np.asarray(bf, np.float32).view(np.uint32)), i
        for bits in (4, 8, 16, 32):
            packed, scales = model.layer_packed(i, bits)
            v, s = O.quantize_rows(wf, bits)
            assert np.array_equal(packed.cpu().numpy(), O.pack_rows(v, bits)), (i, bits)
            assert np.array_equal(scales.cpu().numpy().view(np.uint32), np.asarray(s, np.float32).view(np.uint32)), (i, bits)
    model.close()


def test_packed_views_follow_the_model_not_the_callers_dict():
    """The shapes of the packed views are the library's: a classifier's K is its input channels whatever kernel size the
    description gives, and a description that is changed after the model was made changes nothing."""
    aiq = binding()
    arch = tiny_net()
    arch["layers"][-1]["k"] = 3                         # not read for a classifier
    params = gen_model(tiny_net(), 5)
    model = aiq.Model(arch, params)
    shapes = [tuple(model.layer_packed(i, 8)[0].shape) for i in range(len(arch["layers"]))]
    fc = arch["layers"][-1]
    assert shapes[-1] == (fc["cout"], aiq.aiq_packed_row_bytes(fc["cin"], 8))
    for i in range(len(arch["layers"])):
        n, k = (t.shape for t in (model.layer_folded(i)[1], model.layer_folded(i)[0]))
        assert shapes[i] == (n[0], aiq.aiq_packed_row_bytes(k[1], 8))
    arch["layers"][1]["cout"] += 1
    assert [tuple(model.layer_packed(i, 8)[0].shape) for i in range(len(arch["layers"]))] == shapes
    model.close()
