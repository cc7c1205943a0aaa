"""Layers of stride 2 and more on the tensor-core path: the edges of their row slots, pieces and patches.

Tolerance 5e-3 (relative Frobenius error against the fp64 oracle): bf16 operands, as for every layer of this path."""
import pytest
from dataclasses import replace

import oracle
from paper_2503_20354_b200 import binding as B
from paper_2503_20354_b200 import workloads as W
from gpu_util import oracle_dw, rel_frobenius

pytestmark = pytest.mark.gpu

SHAPES = [
    # 1x1: slots of 8, 16, 32 and 64 positions, full and not; odd maps; the last, partial block of the bitmap
    W.conv("w16", 3, 40, 16, 48, 1, 2, 0), W.conv("w15", 3, 33, 15, 56, 1, 2, 0), W.conv("w17", 2, 24, 17, 64, 1, 2, 0),
    W.conv("w32", 2, 130, 32, 72, 1, 2, 0), W.conv("w33", 1, 19, 33, 48, 1, 2, 0), W.conv("w64", 1, 16, 64, 264, 1, 2, 0),
    W.conv("w65", 1, 9, 65, 48, 1, 2, 0), W.conv("w128", 1, 8, 128, 48, 1, 2, 0), W.conv("w1", 70, 32, 1, 48, 1, 2, 0),
    W.Layer("h3w56", 1, 2, 20, 3, 56, 48, 1, 1, 2, 0), W.Layer("h56w3", 1, 2, 20, 56, 3, 48, 1, 1, 2, 0),
    # slots that are a third empty, with more than 64 channels: shared from 45 or 55 % kept on
    W.conv("w17c72", 2, 72, 17, 64, 1, 2, 0), W.conv("w33c130", 1, 130, 33, 48, 1, 2, 0), W.conv("w65c72", 1, 72, 65, 48, 1, 2, 0),
    # what keeps the other kernel: wider maps, few output channels, channels no multiple of 8
    W.conv("w130", 1, 4, 130, 48, 1, 2, 0), W.conv("o40", 2, 24, 14, 40, 1, 2, 0), W.conv("o50", 2, 24, 14, 50, 1, 2, 0),
    # k x k: rows of whole pieces and not, macros that begin inside a row (20 and 12 positions), images shorter than a macro
    W.conv("k3w32", 2, 40, 32, 48, 3, 2), W.conv("k3w40", 2, 24, 40, 32, 3, 2), W.conv("k3w23", 3, 20, 23, 72, 3, 2),
    W.conv("k3w28", 2, 24, 28, 48, 3, 2), W.conv("k3w14s1", 2, 12, 14, 24, 3),
    W.conv("k3w6", 9, 40, 6, 48, 3, 2), W.conv("k5w48", 1, 20, 48, 32, 5, 2, 2), W.conv("k7w50", 1, 3, 50, 64, 7, 2, 3),
    W.conv("k4s4", 2, 24, 32, 64, 4, 4, 0), W.conv("k3s3w31", 2, 24, 31, 40, 3, 3, 1), W.conv("k3s1c12", 2, 12, 24, 40, 3),
    # rows of the patch with and without padding between them
    W.conv("k3w56", 1, 24, 56, 48, 3, 2), W.conv("k3w112", 1, 16, 112, 64, 3, 2), W.conv("k5w72", 1, 20, 72, 40, 5, 2, 2),
    W.Layer("k3h5w80", 1, 2, 20, 5, 80, 24, 3, 3, 2, 1),
]


@pytest.mark.parametrize("ratio", [0.0, 0.45, 0.55, 0.8])       # 0: fully kept pieces; both sides of the share rules
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", SHAPES, ids=lambda l: l.name)
def test_against_the_oracle(layer, bf16, ratio):
    layer = replace(layer, dt=W.BF16 if bf16 else W.F32)
    a, g = W.activation(layer, 11), W.grad_out(layer, 11)
    dw = B.surgeon_weight_grad(B.surgeon_prune_compact(a.cuda(), ratio), B.layer_desc(layer, B.PATH_TENSOR_CORE), g.cuda())
    bits = W.as_numpy_bits(a).reshape(-1)
    r = oracle.prune_compact(bits, ratio)
    ref = oracle_dw(layer, oracle.decompress(r["bitmap"], r["values"], bits.size), g.numpy())
    assert rel_frobenius(dw.cpu().numpy(), ref) <= 5e-3


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", [W.conv("147 rows", 25, 3, 224, 8, 7, 2, 3), W.conv("245 rows", 112, 5, 97, 24, 7, 2, 3),
                                   W.conv("144 rows", 80, 16, 64, 16, 3)], ids=lambda l: l.name)
def test_two_row_tiles_in_a_cta(layer, bf16):
    """129 to 256 operand rows and at least 32 K-tiles of 64 positions an SM: one CTA takes all rows."""
    test_against_the_oracle(layer, bf16, 0.7)
