"""The fp32 path on the tensor cores, against the fp64 oracle: edges of its tiles, and operands that the three bf16
parts of a number cannot hold.

Tolerance 1e-6 (relative Frobenius error).  A K-tile's sum of the large products is cut off four times, by a unit in the
last place (2^-23) at most each: 4.8e-7.  At most 32 of them are added in fp32, errors of 2^-24 and random sign:
3.4e-7.  What is left out of a product, and what is cut off the small ones, is below 1e-7."""
import numpy as np
import pytest
import torch
from dataclasses import replace

import oracle
from paper_2503_20354_b200 import binding as B
from paper_2503_20354_b200 import workloads as W
from gpu_util import oracle_dw, rel_frobenius

pytestmark = pytest.mark.gpu

SHAPES = [
    # K-tiles of 64 positions over the images: one short of a tile, one more; maps whose rows are split
    W.conv("k63", 1, 24, 7, 40, 1, 1, 0), W.conv("k65_chunks", 13, 130, 5, 17, 1, 1, 0),
    W.conv("w14_c136_o161", 5, 136, 14, 161, 1, 1, 0), W.conv("w7_o159", 3, 15, 7, 159, 3),
    W.conv("w4", 9, 9, 4, 33, 3), W.conv("w33_5x5", 1, 5, 33, 16, 5, 1, 2), W.conv("w16_o320", 2, 43, 16, 320, 3),
    W.Layer("h3w50_2x3", 1, 2, 7, 3, 50, 20, 2, 3, 1, 1),
    # strides: pieces of 16, 11, 7 and 4 positions
    W.conv("s2", 6, 40, 30, 96, 3, 2), W.conv("s3", 8, 24, 40, 64, 5, 3, 1), W.conv("s5", 8, 16, 64, 96, 7, 5, 3),
    W.conv("s8", 12, 64, 64, 32, 8, 8, 0),
    # (of these two the CUDA cores are the faster; the same kinds where the tensor cores are: even and odd maps with padding on the left)
    W.conv("s2_b8", 8, 40, 30, 96, 3, 2), W.conv("s2_w31", 8, 40, 31, 96, 3, 2), W.conv("stem_w65", 12, 3, 65, 64, 7, 2, 3),
    W.conv("s8_o96", 12, 24, 64, 96, 8, 8, 0),
    # linear: columns and channels around the tiles, channels that are no multiple of 4 or 16
    W.linear("t64", 64, 128, 64, dist="normal"), W.linear("t65", 65, 129, 65, dist="normal"),
    W.linear("t1000", 1000, 31, 127, dist="normal"), W.linear("t2049", 2049, 17, 130, dist="normal"),
    W.linear("t1", 1, 300, 10, dist="normal"),
    # the fewest rows of the tensor cores, and one less
    W.linear("t17", 17, 300, 70, dist="normal"), W.linear("t16", 16, 300, 70, dist="normal"),
]
ON_CUDA_CORES = ("s2", "s8", "t1", "t16")


def weight_grad(layer, store, g, **kw):
    """The call, and how many kernels it launched: two on CUDA cores; with the tensor cores two more per slab."""
    before = B.surgeon_launch_count()
    dw = B.surgeon_weight_grad(store, B.layer_desc(layer, B.PATH_FP32), g, **kw)
    return dw, B.surgeon_launch_count() - before


@pytest.mark.parametrize("ratio", [0.0, 0.8])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", SHAPES, ids=lambda l: l.name)
def test_tile_edges(layer, bf16, ratio):
    layer = replace(layer, dt=W.BF16 if bf16 else W.F32)
    a, g = W.activation(layer, 5), W.grad_out(layer, 5)
    store = B.surgeon_prune_compact(a.cuda(), ratio)
    dw, launches = weight_grad(layer, store, g.cuda())
    assert launches == (2 if layer.name in ON_CUDA_CORES else 4)
    bits = W.as_numpy_bits(a).reshape(-1)
    r = oracle.prune_compact(bits, ratio)
    ref = oracle_dw(layer, oracle.decompress(r["bitmap"], r["values"], bits.size), g.numpy())
    assert rel_frobenius(dw.cpu().numpy(), ref) <= 1e-6
    # added to what is there
    twice = B.surgeon_weight_grad(store, B.layer_desc(layer, B.PATH_FP32), g.cuda(), dw=dw.clone(), accumulate=True)
    assert rel_frobenius(twice.cpu().numpy(), 2 * ref) <= 1e-6


LINEAR = W.linear("tokens", 700, 160, 96, dist="normal", dt=W.F32)


@pytest.mark.parametrize("scale_a,scale_g", [(1e-32, 1.0), (1.0, 1e-36), (1e-18, 1e-17), (1e18, 1e17), (3e37, 1e-30)])
def test_magnitudes_at_the_ends_of_the_range(scale_a, scale_g):
    a, g = W.activation(LINEAR, 7) * scale_a, W.grad_out(LINEAR, 7) * scale_g
    store = B.surgeon_prune_compact(a.cuda(), 0.0)
    dw = B.surgeon_weight_grad(store, B.layer_desc(LINEAR, B.PATH_FP32), g.cuda()).cpu().numpy().astype(np.float64)
    ref = g.numpy().astype(np.float64).T @ a.numpy().astype(np.float64).reshape(700, -1)
    # (fp32 ends at 2^-149: half of it for each of the 700 terms where the products lie there)
    assert np.linalg.norm(dw - ref) <= 1e-5 * np.linalg.norm(ref) + 2.0 ** -150 * 700 * np.sqrt(ref.size)


ROWS = [replace(LINEAR, name="linear"), W.conv("k3", 2, 24, 12, 40, 3, dt=W.F32), W.conv("k3s2", 8, 40, 31, 96, 3, 2, dt=W.F32)]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", ROWS, ids=lambda l: l.name)
def test_small_channels_beside_large_ones(layer, bf16):
    """Output channels from 1e-30 down to the smallest subnormal numbers beside ordinary ones, and an input channel of each
    size: every row of dW is as near to its own sum as an ordinary one (1e-6, and half of fp32's last bit, 2^-149)."""
    layer = replace(layer, dt=W.BF16 if bf16 else W.F32)
    a, g = W.activation(layer, 11), W.grad_out(layer, 11)
    a, g = a.reshape(layer.act_shape), g.reshape(layer.grad_shape)
    sizes = [1e-30, 1e-32, 1e-34, 1e-36, 1e-38, 1e-40, 1e-42, 1e-44]
    for i, size in enumerate(sizes):
        g[:, 3 + i] *= size / layer_scale(g)
        a[:, 4 + i] = (a[:, 4 + i].float() * size).to(a.dtype)
    a[:, 12:] = (a[:, 12:].float() * 1e6).to(a.dtype)          # (so that small rows are not all below fp32's range)
    store = B.surgeon_prune_compact(a.cuda(), 0.0)
    dw = B.surgeon_weight_grad(store, B.layer_desc(layer, B.PATH_FP32), g.cuda()).cpu().numpy().astype(np.float64)
    ref = oracle_dw(layer, W.as_numpy_bits(a).reshape(-1), g.numpy()).astype(np.float64).reshape(dw.shape)
    for rows, want in ((dw, ref), (dw.swapaxes(0, 1), ref.swapaxes(0, 1))):        # by output channel, by input channel
        rows, want = rows.reshape(rows.shape[0], -1), want.reshape(rows.shape[0], -1)
        far = np.linalg.norm(rows - want, axis=1) / (1e-6 * np.linalg.norm(want, axis=1) + 2.0 ** -150 * np.sqrt(want.shape[1]))
        assert far.max() <= 1, (np.argmax(far), far.max())


def layer_scale(g):
    return float(g.abs().max())


@pytest.mark.parametrize("small", ["activation", "gradient"])
def test_subnormal_times_large(small):
    """Every product is an ordinary number, one operand rounds to no bf16 number but zero."""
    a, g = W.activation(LINEAR, 12), W.grad_out(LINEAR, 12)
    a, g = (a * 4e-43, g * 1e30) if small == "activation" else (a * 1e30, g * 4e-43)
    store = B.surgeon_prune_compact(a.cuda(), 0.0)
    dw = B.surgeon_weight_grad(store, B.layer_desc(LINEAR, B.PATH_FP32), g.cuda()).cpu().numpy()
    ref = g.numpy().astype(np.float64).T @ a.numpy().astype(np.float64).reshape(700, -1)
    assert np.linalg.norm(ref) > 0 and rel_frobenius(dw, ref) <= 1e-6


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("where", ["activation", "gradient"])
def test_infinities_and_nan(where, value):
    a, g = W.activation(LINEAR, 8), W.grad_out(LINEAR, 8)
    (a.view(700, -1) if where == "activation" else g)[123, 45] = value
    store = B.surgeon_prune_compact(a.cuda(), 0.0)
    dw = B.surgeon_weight_grad(store, B.layer_desc(LINEAR, B.PATH_FP32), g.cuda()).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = g.numpy().astype(np.float64).T @ a.numpy().astype(np.float64).reshape(700, -1)
    assert np.array_equal(np.isnan(dw), np.isnan(ref))
    assert np.array_equal(np.where(np.isinf(dw), dw, 0), np.where(np.isinf(ref), ref, 0))
    ok = np.isfinite(ref)
    assert ok.any() and rel_frobenius(dw[ok], ref[ok]) <= 1e-5


# 22, 313, 100, 64 and 210 partial sums on CUDA cores, 11, 105, 49, 32 and 69 before them on the tensor cores
AGAIN = [LINEAR, W.linear("t20000", 20_000, 16, 16, dist="normal", dt=W.F32), W.conv("k3", 4, 24, 28, 40, 3, dt=W.F32),
         W.conv("k3s2", 8, 40, 31, 96, 3, 2, dt=W.F32), W.conv("stem", 12, 3, 65, 64, 7, 2, 3, dt=W.F32)]


@pytest.mark.parametrize("why", ["activation", "gradient", "large"])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", AGAIN, ids=lambda l: l.name)
def test_calls_that_are_computed_again(layer, bf16, why):
    """What the parts cannot hold: one infinity, or operands whose product the factor would make infinite.  The CUDA cores' sums take
    the place of the others, in another number, also where dW is added to what is there."""
    layer = replace(layer, dt=W.BF16 if bf16 else W.F32)
    a, g = W.activation(layer, 14), W.grad_out(layer, 14)
    if why == "large":
        a, g = a * 2.0 ** 50, g * 2.0 ** 50
    store = B.surgeon_prune_compact(a.cuda(), 0.0)
    ref = oracle_dw(layer, W.as_numpy_bits(a).reshape(-1), g.numpy())
    if why != "large":                             # the element in the middle of what dW's first or last channel is made of
        t = (a if why == "activation" else g).view(layer.batch, -1)
        t[layer.batch // 2, t.shape[1] // 2] = np.inf
        store = B.surgeon_prune_compact(a.cuda(), 0.0)
    dw, launches = weight_grad(layer, store, g.cuda())
    assert launches == 4
    dw = dw.cpu().numpy()
    ok = np.isfinite(dw)
    assert ok.all() == (why == "large") and ok.mean() >= 0.5
    assert rel_frobenius(dw[ok], ref.reshape(dw.shape)[ok]) <= 1e-5
    base = torch.full(dw.shape, 1.0, device="cuda")
    added, _ = weight_grad(layer, store, g.cuda(), dw=base, accumulate=True)
    added = added.cpu().numpy()
    assert np.array_equal(np.isfinite(added), ok)
    assert rel_frobenius(added[ok], 1.0 + ref.reshape(dw.shape)[ok]) <= 1e-5


# gradients whose planes are done in two or three slabs (154, 151 and 164 MB), the last one shorter
SLABS = [W.linear("tokens", 400_003, 24, 40, dist="normal"), W.conv("k3", 48, 4, 128, 20, 3), W.conv("k3s2", 13, 3, 512, 24, 3, 2)]


@pytest.mark.parametrize("layer", SLABS, ids=lambda l: l.name)
def test_slabs(layer):
    a, g = W.activation(layer, 13), W.grad_out(layer, 13)
    store = B.surgeon_prune_compact(a.cuda(), 0.5)
    dw, launches = weight_grad(layer, store, g.cuda())
    assert launches in (6, 8)
    dw = dw.cpu().numpy()
    bits = W.as_numpy_bits(a).reshape(-1)
    r = oracle.prune_compact(bits, 0.5)
    ref = oracle_dw(layer, oracle.decompress(r["bitmap"], r["values"], bits.size), g.numpy())
    assert rel_frobenius(dw, ref) <= 1e-6
    # seen by the last slab alone
    g.view(-1)[-1] = np.inf
    again = B.surgeon_weight_grad(store, B.layer_desc(layer, B.PATH_FP32), g.cuda()).cpu().numpy().reshape(layer.c_out, -1)
    assert not np.isfinite(again[-1]).all() and rel_frobenius(again[:-1], ref.reshape(layer.c_out, -1)[:-1]) <= 1e-5


def test_an_exact_product_stays_exact():
    """One row of the gradient is one value: dW is that row of the activation, to the last bit."""
    a, g = W.activation(LINEAR, 9), torch.zeros(700, 96)
    g[77, 5] = 1.0
    dw = B.surgeon_weight_grad(B.surgeon_prune_compact(a.cuda(), 0.0), B.layer_desc(LINEAR, B.PATH_FP32), g.cuda()).cpu()
    assert torch.equal(dw.view(96, -1)[5], a.view(700, -1)[77]) and not dw.view(96, -1)[6].any()
