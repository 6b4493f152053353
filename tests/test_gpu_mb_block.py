"""The fused inverted-residual block kernel (expansion 1x1 -> depthwise 3x3 -> projection 1x1 with
the hidden tensor in shared memory) at the block shapes of MobileNetV2, alone, at the float32-path
tolerance: a dropped hidden chunk, a wrong halo row or a misplaced band would move the logits by
far more.

Shapes: the channel triples and map sizes of the CIFAR variant (32 / 16 / 8 wide maps, stride 1
with and without shortcut, stride 2) and map widths of the ImageNet variant that are not powers
of two (56, 28, 14, 7: bands that do not fill 128 accumulator lanes, a last band with fewer rows).
Every case checks that the fused kernel really ran (two launches fewer than layer by layer)."""
import numpy as np
import pytest

from aiq_workloads import inverted_residual_stack, gen_model, gen_images
from oracle import aiq_oracle as O
from gpu_util import binding, to_dev, assert_logits_close

pytestmark = pytest.mark.gpu

# (cin, cout, hw, stride)
SHAPES = [
    (16, 24, 32, 1), (24, 24, 32, 1), (32, 64, 32, 2), (64, 64, 16, 1), (96, 96, 16, 1), (96, 160, 16, 2),
    (160, 160, 8, 1), (160, 320, 8, 1),
    (24, 32, 56, 2), (32, 32, 28, 1), (64, 64, 14, 1), (96, 160, 14, 2), (160, 160, 7, 1), (16, 16, 4, 1),
]


@pytest.mark.parametrize("cin,cout,hw,stride", SHAPES)
def test_fused_block_tight_tolerance(cin, cout, hw, stride):
    aiq = binding()
    arch = inverted_residual_stack(cin, cout, hw, stride)
    params = gen_model(arch, 8100 + cin + cout + hw)
    model = aiq.Model(arch, params)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8))
    for batch in (1, 3):
        x = gen_images(batch, 3, hw, hw, 8200 + batch)
        xd = to_dev(x)
        for scheme in ([8, 8, 8, 8, 8], [8, 4, 8, 4, 8], [8, 8, 4, 8, 4]):
            scheme = np.array(scheme, np.uint8)
            ref = O.forward_scheme(arch, bank, scheme, x)
            aiq.aiq_set_fusion(True, True, inverted_residual=True)
            try:
                got = model.aiq_forward(scheme, xd).cpu().numpy()
                fused_launches = aiq.aiq_last_call_stats()["kernel_launches"]
            finally:
                aiq.aiq_set_fusion(True, True)
            plain = model.aiq_forward(scheme, xd).cpu().numpy()
            plain_launches = aiq.aiq_last_call_stats()["kernel_launches"]
            what = f"block {cin}->{cout} {hw}x{hw} stride {stride} batch {batch} scheme {scheme.tolist()}"
            assert fused_launches == plain_launches - 2, what
            assert_logits_close(got, ref, what + " fused")
            assert_logits_close(plain, ref, what + " layer by layer")
    model.close()


def test_fused_block_versions_share_one_launch():
    """Several candidates that differ inside the block (expansion, depthwise or projection bits)
    are jobs of one fused launch; predictions and counts follow the oracle."""
    import torch
    from gpu_util import assert_preds_match
    aiq = binding()
    arch = inverted_residual_stack(32, 32, 16, 1)
    params = gen_model(arch, 8301)
    x = gen_images(40, 3, 16, 16, 8302)
    folded = O.fold_model(arch, params)
    mean_logits = O.forward_fp32_unquantized(arch, folded, x).astype(np.float64).mean(axis=0)
    params = [dict(p) for p in params]
    params[-1]["bias"] = (params[-1]["bias"].astype(np.float64) - mean_logits).astype(np.float32)
    folded = O.fold_model(arch, params)
    bank = O.build_weight_bank(folded, (4, 8, 16))
    labels = O.predict(O.forward_fp32_unquantized(arch, folded, x))
    model = aiq.Model(arch, params)
    schemes = np.array([[8, 8, 8, 8, 8], [8, 4, 8, 8, 8], [8, 8, 4, 8, 8], [8, 8, 16, 8, 8], [8, 8, 8, 4, 8], [4, 8, 8, 8, 8]],
                       np.uint8)
    oacc, ocounts, opreds, omargins = O.eval_schemes(arch, bank, schemes, x, labels)
    preds = torch.full((len(schemes), 40), -1, dtype=torch.int32, device="cuda")
    aiq.aiq_set_fusion(True, True, inverted_residual=True)
    try:
        acc, counts = model.aiq_eval_schemes(schemes, to_dev(x), to_dev(labels), preds=preds, chunk=40)
        fused_launches = aiq.aiq_last_call_stats()["kernel_launches"]
    finally:
        aiq.aiq_set_fusion(True, True)
    model.aiq_eval_schemes(schemes, to_dev(x), to_dev(labels), chunk=40)
    assert fused_launches < aiq.aiq_last_call_stats()["kernel_launches"]
    assert_preds_match(preds.cpu().numpy(), opreds, omargins, "fused block, six candidates")
    assert np.all(np.abs(counts - ocounts) <= (omargins <= 1e-2).sum(axis=1))
    model.close()


@pytest.mark.parametrize("variant,hw,batch", [("cifar", 32, 24), ("imagenet", 224, 3)])
def test_mobilenet_v2_with_fused_blocks(variant, hw, batch):
    """The whole MobileNetV2 (16 of its 17 blocks fused, 10 seeded conv layers at 4 bits) against the
    oracle at the tensor-path tolerance, with the classifier balanced so that the labels spread."""
    from aiq_workloads import mobilenet_v2, mixed_int4_int8_scheme, conv_layer_indices
    from gpu_util import assert_preds_match
    from test_gpu_forward import balance_classifier, assert_tensor_path_logits
    aiq = binding()
    arch = mobilenet_v2(variant)
    x = gen_images(batch, 3, hw, hw, 8624)
    params = balance_classifier(arch, gen_model(arch, 2234), x)
    model = aiq.Model(arch, params)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8))
    scheme = mixed_int4_int8_scheme(53, conv_layer_indices(arch), 10, 43)
    ref = O.forward_scheme(arch, bank, scheme, x)
    aiq.aiq_set_fusion(True, True, inverted_residual=True)
    try:
        got = model.aiq_forward(scheme, to_dev(x)).cpu().numpy()
        fused_launches = aiq.aiq_last_call_stats()["kernel_launches"]
    finally:
        aiq.aiq_set_fusion(True, True)
    model.aiq_forward(scheme, to_dev(x))
    assert fused_launches <= aiq.aiq_last_call_stats()["kernel_launches"] - 2 * 15
    assert_tensor_path_logits(got, ref, f"mbv2 {variant} fused blocks")
    assert_preds_match(O.predict(got), O.predict(ref), O.top2_margin(ref), f"mbv2 {variant} fused blocks")
    model.close()


def test_default_policy_does_not_depend_on_the_batch():
    """The default setting runs a block layer by layer whatever the number of images: where the fused kernel is the
    faster one depends on the batch, an image's logits must not.  The pass follows the oracle on sampled images."""
    aiq = binding()
    arch = inverted_residual_stack(160, 160, 8, 1)
    params = gen_model(arch, 8401)
    model = aiq.Model(arch, params)
    bank = O.build_weight_bank(O.fold_model(arch, params), (8,))
    scheme = np.full(5, 8, np.uint8)
    x = gen_images(149, 3, 8, 8, 8402)
    got = model.aiq_forward(scheme, to_dev(x)).cpu().numpy()
    launches = aiq.aiq_last_call_stats()["kernel_launches"]
    for batch in (100, 128, 148):
        part = model.aiq_forward(scheme, to_dev(x[:batch])).cpu().numpy()
        assert aiq.aiq_last_call_stats()["kernel_launches"] == launches
        assert np.array_equal(part, got[:batch]), batch
    sample = np.arange(3, 149, 16)
    assert_logits_close(got[sample], O.forward_scheme(arch, bank, scheme, x[sample]), "default policy")
    model.close()


def _separable_net(hw, shapes):
    """Stem, then 1x1 and depthwise layers in turn without shortcuts; shapes: (kind, channels, stride)."""
    layers = [dict(name="stem", kind="conv", cin=3, cout=24, k=3, stride=1, pad=1, act="relu6", input=-1, residual=-1, has_bn=True)]
    for kind, cout, stride in shapes:
        k = 3 if kind == "dw" else 1
        layers.append(dict(name=f"l{len(layers)}", kind=kind, cin=layers[-1]["cout"], cout=cout, k=k, stride=stride, pad=k // 2,
                           act="relu6", input=len(layers) - 1, residual=-1, has_bn=True))
    layers.append(dict(name="fc", kind="fc", cin=layers[-1]["cout"], cout=6, k=1, stride=1, pad=0, act="none",
                       input=len(layers) - 1, residual=-1, has_bn=False))
    return dict(name="separable", in_c=3, in_h=hw, in_w=hw, n_classes=6, layers=layers)


def _check_separable_net(arch, hw, batch, fused_blocks):
    aiq = binding()
    params = gen_model(arch, 8500 + hw)
    model = aiq.Model(arch, params)
    bank = O.build_weight_bank(O.fold_model(arch, params), (4, 8, 16))
    x = gen_images(batch, 3, hw, hw, 8501)
    L = len(arch["layers"])
    for low, bits in ((0, 8), (1, 4), (2, 16), (3, 4)):
        scheme = np.full(L, 8, np.uint8)
        scheme[low] = bits
        ref = O.forward_scheme(arch, bank, scheme, x)
        launches = []
        for on in (True, False):
            aiq.aiq_set_fusion(True, True, inverted_residual=on)
            try:
                got = model.aiq_forward(scheme, to_dev(x)).cpu().numpy()
                launches.append(aiq.aiq_last_call_stats()["kernel_launches"])
            finally:
                aiq.aiq_set_fusion(True, True)
            assert_logits_close(got, ref, f"{[l['name'] for l in arch['layers']]} fused {on} scheme {scheme.tolist()}")
        assert launches[0] == launches[1] - 2 * fused_blocks
    model.close()


@pytest.mark.parametrize("hw,batch,stride", [(9, 3, 2), (16, 2, 1)])
def test_fused_block_before_a_depthwise_layer(hw, batch, stride):
    """The projection's tensor is read by a depthwise layer alone: floats where the projection runs as a layer, hi / lo pairs
    where the fused kernel writes it, and the depthwise layer has to read what was written."""
    _check_separable_net(_separable_net(hw, [("conv", 96, 1), ("dw", 96, 1), ("conv", 48, 1), ("dw", 48, stride)]), hw, batch, 1)


@pytest.mark.parametrize("hw,batch", [(9, 3), (16, 2)])
def test_blocks_that_share_a_layer(hw, batch):
    """1x1 and depthwise layers in turn: each 1x1 layer between two depthwise ones could end a block and begin the next.  Of
    the three candidates the first and the third are fused."""
    _check_separable_net(_separable_net(hw, [("conv", 96, 1), ("dw", 96, 1), ("conv", 48, 1), ("dw", 48, 2), ("conv", 64, 1),
                                             ("dw", 64, 1), ("conv", 32, 1)]), hw, batch, 2)


@pytest.mark.parametrize("between,hw,batch,fused", [("second stem", 12, 5, 0), ("second reader", 48, 24, 0), ("late stem", 12, 5, 1)])
def test_block_with_other_layers_between_its_own(between, hw, batch, fused):
    """Layers listed between the three of a block run before the fused kernel, which reads the block's input only then.  Where
    one of them, or the block's result, was given the input's memory, the block must run layer by layer; else it is fused."""
    def conv(cin, cout, k, inp, kind="conv", residual=-1):
        return dict(name=f"{kind}{cout}", kind=kind, cin=cin, cout=cout, k=k, stride=1, pad=k // 2, act="relu6", input=inp,
                    residual=residual, has_bn=True)
    layers = [conv(3, 24, 3, -1), conv(24, 96, 1, 0)]
    if between == "second stem":
        layers += [conv(3, 24, 3, -1), conv(96, 96, 3, 1, "dw"), conv(96, 32, 1, 3), conv(24, 32, 1, 2, residual=4)]
    elif between == "late stem":        # after the depthwise layer: gets the expansion's memory, which nothing needs
        layers += [conv(96, 96, 3, 1, "dw"), conv(3, 24, 3, -1), conv(96, 32, 1, 2), conv(24, 32, 1, 3, residual=4)]
    else:
        layers += [conv(96, 96, 3, 1, "dw"), conv(24, 32, 1, 0), conv(96, 32, 1, 2), conv(32, 32, 1, 3, residual=4)]
    layers.append(dict(name="fc", kind="fc", cin=32, cout=6, k=1, stride=1, pad=0, act="none", input=5, residual=-1, has_bn=False))
    _check_separable_net(dict(name="branches", in_c=3, in_h=hw, in_w=hw, n_classes=6, layers=layers), hw, batch, fused)
