"""The tensor between a pointwise layer and its depthwise readers, stored as floats: hidden channel counts whose last store unit
of 32 channels is half empty or partly padding, pixel tiles that end inside an image, maps of one and two columns, both strides,
two and four columns per thread, every launch variant and weight class of the pointwise layer, every activation, a depthwise
layer with a shortcut, two readers.

Two checks.  Against the oracle, with the float32 rule of the other forward tests, 1e-3 (1 + |ref|).  And bit for bit against
the same weights in a network with one more reader of the tensor, a pointwise layer whose own output nothing reads: hi / lo
pairs are stored there, and a float has to be exactly the value of the pair it replaces."""
import numpy as np
import pytest

from aiq_workloads import gen_model, gen_images
from oracle import aiq_oracle as O
from gpu_util import binding, to_dev, assert_logits_close

pytestmark = pytest.mark.gpu


def _layer(kind, cin, cout, k, stride, act, inp, residual=-1):
    return dict(name=f"{kind}{cout}", kind=kind, cin=cin, cout=cout, k=k, stride=stride, pad=k // 2, act=act, input=inp,
                residual=residual, has_bn=kind != "fc")


def _net(cin, hid, hw, depthwise, act="relu6", project=32):
    """Stem, pointwise layer (layer 1), depthwise layers [(input, stride, residual)] from layer 2 on, projection, classifier."""
    layers = [_layer("conv", 3, cin, 3, 1, "relu6", -1), _layer("conv", cin, hid, 1, 1, act, 0)]
    layers += [_layer("dw", hid, hid, 3, stride, "relu6", inp, res) for inp, stride, res in depthwise]
    if project:
        layers.append(_layer("conv", hid, project, 1, 1, "none", len(layers) - 1))
    layers.append(_layer("fc", project or hid, 6, 1, 1, "none", len(layers) - 1))
    return dict(name="float_tensor", in_c=3, in_h=hw, in_w=hw, n_classes=6, layers=layers)


def _with_a_pointwise_reader(arch, params):
    """The same network and weights, and a pointwise layer that reads layer 1 and that nothing reads (before the classifier)."""
    layers = arch["layers"][:-1] + [_layer("conv", arch["layers"][1]["cout"], 16, 1, 1, "none", 1)] + arch["layers"][-1:]
    pairs = dict(arch, layers=layers)
    return pairs, params[:-1] + [gen_model(pairs, 77)[-2]] + params[-1:]


def _check(arch, seed, batch, schemes):
    """schemes: bits of the layers from the first on, 8 for the others."""
    aiq = binding()
    hw, n = arch["in_h"], len(arch["layers"])
    params = gen_model(arch, seed)
    x = gen_images(batch, 3, hw, hw, seed + 1)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8, 16, 32))
    model = aiq.Model(arch, params)
    other = aiq.Model(*_with_a_pointwise_reader(arch, params))
    for sc in schemes:
        scheme = np.array(list(sc) + [8] * (n - len(sc)), np.uint8)
        got = model.aiq_forward(scheme, to_dev(x)).cpu().numpy()
        what = f"{[l['name'] for l in arch['layers']]} {hw} wide, batch {batch}, {scheme.tolist()}"
        assert_logits_close(got, O.forward_scheme(arch, bank, scheme, x), what)
        pairs = other.aiq_forward(np.insert(scheme, n - 1, 8), to_dev(x)).cpu().numpy()
        assert np.array_equal(got.view(np.uint32), pairs.view(np.uint32)), what
    model.close()
    other.close()


# (block input channels, expansion factor, size, stride, batch)
@pytest.mark.parametrize("cin,t,hw,stride,batch", [(24, 1, 8, 1, 1), (16, 3, 9, 2, 5), (24, 6, 7, 1, 19), (40, 2, 13, 2, 3), (24, 5, 33, 1, 2),
                                                   (160, 6, 4, 1, 33), (24, 2, 1, 1, 1), (24, 2, 1, 2, 3), (24, 2, 2, 1, 1), (16, 3, 2, 2, 1),
                                                   (16, 3, 33, 1, 21)])
def test_expansion_to_depthwise_in_floats(cin, t, hw, stride, batch):
    _check(_net(cin, cin * t, hw, [(1, stride, -1)]), 9700 + cin + hw, batch, ([8, 4], [8, 8, 4], [8, 16, 32], [32, 32]))


# streamed weights (one and two pieces), one block per SM with 24 and with 12 epilogue warps
@pytest.mark.parametrize("cin,hid,hw,batch", [(160, 64, 4, 9), (16, 960, 4, 64), (160, 1280, 8, 64)])
def test_pointwise_variants_store_floats(cin, hid, hw, batch):
    _check(_net(cin, hid, hw, [(1, 1, -1)]), 9800 + cin, batch, ([8, 4], [8, 32]))


@pytest.mark.parametrize("act", ["none", "relu"])
def test_pointwise_activations_in_floats(act):
    _check(_net(24, 72, 11, [(1, 1, -1)], act), 9900, 4, ([8, 8], [8, 16]))


@pytest.mark.parametrize("hid,hw,stride,batch", [(48, 9, 1, 3), (48, 9, 2, 3), (96, 16, 1, 48)])
def test_two_depthwise_readers_and_a_shortcut(hid, hw, stride, batch):
    """Both depthwise layers read the floats; the second adds the first one's output, a tensor of pairs."""
    _check(_net(24, hid, hw, [(1, stride, -1), (1, stride, 2)]), 9950, batch, ([8, 8, 4, 8], [8, 4, 8, 32]))


@pytest.mark.parametrize("act,hid,bits", [("relu6", 72, 8), ("none", 48, 4), ("relu", 40, 32)])
def test_stored_floats_are_the_values_of_the_pairs(act, hid, bits):
    """The tensor itself, as the workspace holds it after the pass.  Slots: stem and depthwise output 0, pointwise output 1,
    the other reader's 2; they are the end of the workspace, in this order, each rounded up to 256 bytes."""
    import torch
    aiq = binding()
    cs, hw, batch = (hid + 15) // 16 * 16, 10, 3
    arch = _net(24, hid, hw, [(1, 1, -1)], act, project=0)
    params = gen_model(arch, 9990 + hid)
    pairs_arch, pairs_params = _with_a_pointwise_reader(arch, params)
    x = to_dev(gen_images(batch, 3, hw, hw, 9991))
    slot = lambda channels: (batch * (hw + 2) * hw * 4 * channels + 255) // 256 * 256
    stored = []
    for a, p, after in ((arch, params, 0), (pairs_arch, pairs_params, slot(16))):
        model = aiq.Model(a, p)
        ws = torch.zeros(model.aiq_workspace_bytes(batch, 1), dtype=torch.uint8, device="cuda")
        scheme = np.full(len(a["layers"]), 8, np.uint8)
        scheme[1] = bits
        model.aiq_forward(scheme, x, workspace=ws)
        first = ws.numel() - after - slot(cs)
        stored.append(ws[first:first + batch * (hw + 2) * hw * 4 * cs].clone())
        model.close()
    floats = stored[0].view(torch.float32).view(batch, hw + 2, hw, cs)
    halves = stored[1].view(torch.bfloat16).view(batch, hw + 2, hw, 2, cs).float()
    assert torch.equal(floats, halves[..., 0, :] + halves[..., 1, :])
    assert not torch.equal(stored[0], stored[1])
    inside = floats[:, 1:-1, :, :hid]
    assert (inside != 0).any(dim=3).all() and not floats[:, [0, -1]].any() and not floats[..., hid:].any()
    assert not torch.equal(inside, inside.bfloat16().float())            # the lo half counts
