"""CPU-side checks of libsurgeon.so: it builds for sm_100a, loads, exports every symbol that
include/surgeon.h declares, and its host-only entry points (ratio rule, size arithmetic, argument
checks) agree with the oracle.  No kernel is launched here."""
import ctypes
import os
import re

import numpy as np
import pytest

import oracle
from paper_2503_20354_b200 import binding as B
from paper_2503_20354_b200 import build as lib_build
from paper_2503_20354_b200 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_build.build()


def test_exports_every_declared_symbol():
    text = open(os.path.join(ROOT, "include", "surgeon.h")).read()
    names = set(re.findall(r"\b(surgeon_[a-z_0-9]+)\s*\(", text))
    assert {"surgeon_layer_ratios", "surgeon_compact_sizes", "surgeon_prune_compact",
            "surgeon_weight_grad", "surgeon_weight_grad_workspace", "surgeon_decompress",
            "surgeon_status_string", "surgeon_layer_ratios_rule",
            "surgeon_gradient_importance"} <= names
    l = ctypes.CDLL(B.LIB_PATH)
    for n in names:
        assert hasattr(l, n), n


def test_struct_layouts_match_header():
    assert ctypes.sizeof(B.Header) == 32
    assert ctypes.sizeof(B.Compressed) == 48
    assert ctypes.sizeof(B.LayerDesc) == 48


@pytest.mark.parametrize("layer", [
    W.conv("shortcut", 200, 16, 32, 160, 1, 1, 0), W.conv("3x3", 200, 160, 32, 160, 3), W.conv("expand", 64, 64, 56, 256, 1, 1, 0),
    W.conv("stem", 64, 3, 224, 64, 7, 2, 3), W.conv("head", 16, 64, 512, 19, 1, 1, 0), W.linear("fc1", 12608, 768, 3072),
    W.linear("few columns", 1_000_000, 64, 10)], ids=lambda l: l.name)
def test_scratch_of_the_fp32_path_is_bounded(layer):
    """The bf16 parts of the gradient: 128 MB, or half the fp32 gradient where that is more; and the partial sums, one per
    20 K-tiles of 64 (the number of weights each), or 64 MB of them."""
    grad = 4 * int(np.prod(layer.grad_shape))
    positions = grad // 4 // layer.c_out
    partial = 4 * layer.n_weight * (positions // (20 * 64) + 2)
    assert B.surgeon_weight_grad_workspace(B.layer_desc(layer, B.PATH_FP32)) <= max(128 << 20, grad // 2) + max(64 << 20, partial) + (1 << 20)


def test_strides_of_7_and_8_with_few_outputs_stay_on_cuda_cores():
    """Their scratch is partial sums alone; layers of the other kernel have the gradient's parts in it too."""
    for k, outputs, alone in ((8, 64, True), (7, 16, True), (8, 96, False), (6, 64, False)):
        l = W.conv("k", 16, 64, 64, outputs, k, k, 0)
        assert (B.surgeon_weight_grad_workspace(B.layer_desc(l, B.PATH_FP32)) % (4 * l.n_weight) == 0) == alone, (k, outputs)
    assert B.surgeon_weight_grad_workspace(B.layer_desc(W.conv("k", 16, 32, 64, 64, 8, 8, 0), B.PATH_FP32)) % (4 * 64 * 32 * 64)


def test_linear_layers_of_up_to_16_rows_stay_on_cuda_cores():
    for rows in (1, 2, 16, 17):
        for c, o in ((320, 16), (2048, 1000)):
            l = W.linear("few", rows, c, o)
            alone = B.surgeon_weight_grad_workspace(B.layer_desc(l, B.PATH_FP32)) % (4 * l.n_weight) == 0
            assert alone == (rows <= 16), (rows, c, o)


def test_ratios_match_oracle_and_fixture():
    st, p = oracle.layer_ratios([2, 1, 4], [4, 2, 2])
    got = B.surgeon_layer_ratios([2, 1, 4], [4, 2, 2])
    assert got.tolist() == [0.75, 0.75, 0.0] == p.tolist()
    rng = np.random.default_rng(4)
    for layers in (W.wrn28_10(), W.resnet50(), W.vit_b16()):
        gi = W.gradient_importance(len(layers), seed=0)
        lam = np.array([l.act_bytes for l in layers], dtype=np.float64)
        _, ref = oracle.layer_ratios(gi, lam)
        np.testing.assert_allclose(B.surgeon_layer_ratios(gi, lam), ref, rtol=0, atol=1e-14)


def test_ratios_errors():
    with pytest.raises(B.SurgeonError) as e:
        B.surgeon_layer_ratios([1.0], [5.0])
    assert e.value.status == B.SURGEON_ERR_DEGENERATE
    assert B.surgeon_layer_ratios([1.0], [5.0], allow_degenerate=True).tolist() == [0.0]
    for gi, lam in (([1.0, -1.0], [1.0, 1.0]), ([1.0, np.nan], [1.0, 1.0]), ([1.0, 1.0], [0.0, 1.0]),
                    ([1.0, 1.0], [np.inf, 1.0])):
        with pytest.raises(B.SurgeonError) as e:
            B.surgeon_layer_ratios(gi, lam)
        assert e.value.status == B.SURGEON_ERR_INVALID_ARG


def test_ratio_rule_variants_match_oracle():
    for layers in (W.wrn28_10(), W.resnet50(), W.vit_b16()):
        gi = W.gradient_importance(len(layers), seed=1)
        lam = np.array([l.act_bytes for l in layers], dtype=np.float64)
        for rule in (oracle.RULE_BOTH, oracle.RULE_NO_GRADIENT, oracle.RULE_NO_MEMORY):
            _, ref = oracle.layer_ratios_rule(gi, lam, rule)
            np.testing.assert_allclose(B.surgeon_layer_ratios_rule(gi, lam, rule), ref, rtol=0, atol=1e-14)
        _, ref = oracle.layer_ratios_rule(gi, lam, oracle.RULE_STATIC, 0.9)
        assert np.array_equal(B.surgeon_layer_ratios_rule(gi, lam, B.SURGEON_RULE_STATIC, 0.9), ref)
    # the factor that is left out need not be passed
    np.testing.assert_allclose(B.surgeon_layer_ratios_rule(None, [8, 4, 2, 2], B.SURGEON_RULE_NO_GRADIENT),
                               [2 / 3, 1 / 3, 0, 0], rtol=0, atol=1e-12)
    np.testing.assert_allclose(B.surgeon_layer_ratios_rule([3, 3, 1, 2], None, B.SURGEON_RULE_NO_MEMORY),
                               [0, 0, 2 / 3, 1 / 3], rtol=0, atol=1e-15)
    for args in (([1.0, 2.0], [1.0, 1.0], 7, 0.0), ([1.0, 2.0], [1.0, 1.0], B.SURGEON_RULE_STATIC, 1.5),
                 (None, [1.0, 1.0], B.SURGEON_RULE_NO_MEMORY, 0.0), ([1.0, -2.0], None, B.SURGEON_RULE_NO_MEMORY, 0.0)):
        with pytest.raises(B.SurgeonError) as e:
            B.surgeon_layer_ratios_rule(*args)
        assert e.value.status == B.SURGEON_ERR_INVALID_ARG
    with pytest.raises(B.SurgeonError) as e:
        B.surgeon_layer_ratios_rule([0.0, 0.0], None, B.SURGEON_RULE_NO_MEMORY)
    assert e.value.status == B.SURGEON_ERR_DEGENERATE


def test_compact_sizes_match_oracle_kept_count():
    for n in (0, 1, 31, 32, 33, 1023, 1024, 1025, 1 << 20, 12345677, (1 << 31) - 1):
        for ratio in (0.0, 0.1, 0.3, 0.5, 0.6, 0.9, 0.99, 1.0):
            for dt, es in ((B.SURGEON_F32, 4), (B.SURGEON_BF16, 2)):
                s = B.surgeon_compact_sizes(n, dt, ratio)
                assert s.n_keep == oracle.n_keep(n, ratio)
                assert s.bitmap_bytes == 4 * ((n + 31) // 32)
                assert s.values_bytes == s.n_keep * es
                assert s.offsets_bytes == 4 * ((n + 127) // 128 + 1)
                assert s.workspace_bytes > 0 and s.workspace_bytes % 256 == 0
    for bad in ((-1, 0, 0.5), (10, 0, 1.5), (10, 0, -0.1), (10, 2, 0.5), (10, 0, float("nan"))):
        with pytest.raises(B.SurgeonError) as e:
            B.surgeon_compact_sizes(*bad)
        assert e.value.status == B.SURGEON_ERR_INVALID_ARG
    with pytest.raises(B.SurgeonError) as e:
        B.surgeon_compact_sizes(1 << 31, 0, 0.5)
    assert e.value.status == B.SURGEON_ERR_UNSUPPORTED


def test_argument_checks_need_no_device():
    l = B.lib()
    comp = B.Compressed(16, 0, 0, 0, 0, 0, 0)
    assert l.surgeon_prune_compact(0, 16, 0, 0.5, ctypes.byref(comp), 0, 0, 0) == B.SURGEON_ERR_INVALID_ARG
    assert l.surgeon_prune_compact(0, 16, 0, 2.0, ctypes.byref(comp), 0, 0, 0) == B.SURGEON_ERR_INVALID_ARG
    d = B.LayerDesc(1, 2, 3, 8, 8, 4, 3, 3, 1, 1, 1)
    assert B.surgeon_weight_grad_workspace(d) > 0
    bad = B.LayerDesc(0, 2, 3, 8, 8, 4, 3, 3, 1, 1, 1)     # linear with a spatial extent
    assert B.surgeon_weight_grad_workspace(bad) == 0
    assert l.surgeon_weight_grad(ctypes.byref(comp), ctypes.byref(bad), 16, 16, 0, 0, 0, 0) == B.SURGEON_ERR_INVALID_ARG
    assert B.status_string(B.SURGEON_ERR_TIMEOUT).startswith("device-side")


def test_grouped_layers_that_have_a_plan():
    """Groups of many odd channel counts, and depthwise layers on wide maps: what a tile of 110 KB holds is not refused."""
    for layer in (W.conv("wide_groups", 4, 254, 40, 2, 3, groups=2), W.conv("out51", 1, 4, 256, 204, 3, groups=4),
                  W.conv("c15", 1, 30, 240, 30, 3, groups=2), W.conv("dw4096", 1, 2, 4096, 2, 3, groups=2),
                  W.conv("dw6144_s2", 1, 2, 6144, 2, 3, 2, groups=2)):
        assert B.surgeon_weight_grad_workspace(B.layer_desc(layer, B.PATH_TENSOR_CORE)) > 0, layer.name
