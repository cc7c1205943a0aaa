"""Sizes at which the variants that a dispatch chooses between can go wrong: edges of tiles and remainders,
the smallest and the largest of each range, against the oracle."""
import numpy as np
import pytest
import torch
from dataclasses import replace

import oracle
from paper_2503_20354_b200 import binding as B
from paper_2503_20354_b200 import workloads as W
from gpu_util import assert_store_equals_oracle, oracle_dw, rel_frobenius

pytestmark = pytest.mark.gpu


def _dw(layer, ratio, path, seed=5):
    a, g = W.activation(layer, seed), W.grad_out(layer, seed)
    comp, ref = assert_store_equals_oracle(a, ratio)
    dw = B.surgeon_weight_grad(comp, B.layer_desc(layer, path), g.cuda()).cpu().numpy()
    dense = oracle.decompress(ref["bitmap"], ref["values"], a.numel())
    if layer.dt == W.BF16:
        dense = dense.view(np.uint16)
    assert comp.read_header().status == B.SURGEON_OK
    return dw, oracle_dw(layer, dense, g.numpy())


TRANSPOSED = [
    # slabs (maps 16, 32, 64 wide): partial last K-tile, channels past a row tile, columns past a unit
    W.conv("slab16", 3, 40, 16, 72, 3),
    W.Layer("slab16_h5", 1, 5, 24, 5, 16, 48, 3, 3, 1, 1),
    W.Layer("slab32_h3", 1, 7, 144, 3, 32, 176, 3, 3, 1, 1),
    W.Layer("slab64_h1", 1, 9, 20, 1, 64, 64, 3, 3, 1, 1),
    W.conv("slab64", 1, 20, 64, 328, 3),
    # boxes with halo rows (rows a multiple of 8 wide)
    W.conv("halo8", 9, 72, 8, 168, 3),
    W.Layer("halo8_h3", 1, 4, 20, 3, 8, 56, 3, 3, 1, 1),
    W.conv("halo24", 2, 20, 24, 64, 3),
    W.conv("halo56", 1, 40, 56, 48, 3),
    W.conv("halo16_nopad", 2, 20, 16, 64, 3, 1, 0),
    W.Layer("halo16_2x3", 1, 2, 20, 9, 16, 48, 2, 3, 1, 1),
    # one kernel row: its single accumulator is as wide as an MMA allows, not as the 512 columns would
    W.Layer("halo8_1x3", 1, 3, 20, 9, 8, 264, 1, 3, 1, 0),
    W.Layer("halo16_1x5", 1, 2, 40, 5, 16, 320, 1, 5, 1, 0),
    W.Layer("halo32_1x3", 1, 1, 20, 3, 32, 512, 1, 3, 1, 0),
    W.Layer("halo56_1x2", 1, 1, 24, 2, 56, 768, 1, 2, 1, 0),
    # a box per tap (other widths, other kernels)
    W.conv("tap7", 9, 40, 7, 136, 3),
    W.conv("tap14", 3, 24, 14, 264, 3),
    W.conv("tap30_5x5", 2, 20, 30, 48, 5, 1, 2),
    W.conv("tap3_7x7", 11, 24, 3, 64, 7, 1, 3),
    W.conv("tap1", 70, 24, 1, 56, 3),
    # just outside: wider than a K-tile, too few or unaligned output channels
    W.conv("copies65", 1, 20, 65, 64, 3),
    W.conv("copies72", 1, 20, 72, 56, 3),
    W.conv("copies_o52", 2, 20, 16, 52, 3),
]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", TRANSPOSED, ids=lambda l: l.name)
def test_stride_one_taps(layer, bf16):
    dw, ref = _dw(replace(layer, dt=W.BF16 if bf16 else W.F32), 0.6, B.PATH_TENSOR_CORE)
    assert rel_frobenius(dw, ref) <= 5e-3


DEPTHWISE = [
    # one band and several, one strip a thread and none, one image and more than a tile holds
    W.conv("dw8", 3, 3, 8, 3, 3, groups=3),
    W.conv("dw64", 1, 5, 64, 5, 3, groups=5),
    W.conv("dw56_b9", 9, 4, 56, 4, 3, groups=4),
    W.conv("dw128_bands", 1, 2, 128, 2, 3, groups=2),
    W.conv("dw112_s2", 2, 3, 112, 3, 3, 2, groups=3),
]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", DEPTHWISE, ids=lambda l: l.name)
def test_depthwise_sums_shared_by_lanes(layer, bf16):
    layer = replace(layer, dt=W.BF16 if bf16 else W.F32)
    a, g = W.activation(layer, 6), W.grad_out(layer, 6)
    comp, ref = assert_store_equals_oracle(a, 0.5)
    dw = B.surgeon_weight_grad(comp, B.layer_desc(layer, B.PATH_TENSOR_CORE), g.cuda()).cpu().numpy()
    dense = oracle.decompress(ref["bitmap"], ref["values"], a.numel()).reshape(layer.act_shape)
    exp = oracle.dw_conv2d_grouped(dense.view(np.uint16) if bf16 else dense, g.numpy(), 3, 3, layer.stride, 1, layer.groups)
    assert rel_frobenius(dw, exp) <= 1e-5      # fp32 sums of at most 4096 terms (3e-6), doubles after


STRIDED = [
    W.conv("s2_w17", 3, 20, 17, 40, 3, 2),
    W.conv("s2_w112_many_macros", 1, 3, 112, 16, 7, 2, 3),
    W.conv("s2_two_units", 2, 30, 14, 520, 3, 2),
    W.conv("s3_5x5", 2, 9, 23, 24, 5, 3, 2),
    W.conv("s8", 2, 20, 64, 64, 8, 8, 0),
    W.conv("s2_2x2_c70", 1, 70, 30, 24, 2, 2, 0),
    W.conv("s1_c8", 3, 8, 33, 24, 3),
    W.conv("s1_c16_w40", 2, 16, 40, 160, 3),
    W.conv("s2_long_reduction", 40, 8, 20, 8, 3, 2),
]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", STRIDED, ids=lambda l: l.name)
def test_expanded_operand(layer, bf16):
    dw, ref = _dw(replace(layer, dt=W.BF16 if bf16 else W.F32), 0.4, B.PATH_TENSOR_CORE)
    assert rel_frobenius(dw, ref) <= 5e-3


@pytest.mark.parametrize("layer", [
    W.conv("c_stride2", 3, 9, 33, 70, 3, 2), W.conv("c_wide", 1, 5, 70, 9, 3), W.conv("c_stride5", 2, 30, 41, 65, 5, 5, 2),
    W.conv("c_w3", 9, 20, 3, 129, 3), W.linear("l", 77, 129, 65, dt=W.F32), W.linear("l1", 1, 128, 64, dt=W.F32)],
    ids=lambda l: l.name)
def test_fp32_tiles(layer):
    dw, ref = _dw(layer, 0.5, B.PATH_FP32)
    assert rel_frobenius(dw, ref) <= 1e-5


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("layer", [
    W.conv("map1", 70, 40, 1, 65, 1, 1, 0), W.conv("map2", 37, 33, 2, 20, 1, 1, 0), W.conv("map2_2x2", 75, 20, 2, 24, 2, 1, 0),
    W.conv("map3", 15, 20, 3, 66, 3), W.Layer("rows_of_3", 1, 5, 9, 8, 3, 130, 3, 3, 1, 1), W.conv("map7", 5, 20, 7, 24, 3),
    W.Layer("rows_of_4", 1, 7, 9, 5, 4, 20, 3, 3, 1, 1), W.conv("map9", 3, 10, 9, 70, 3, 2), W.conv("one_output", 45, 12, 5, 24, 5, 1, 0),
    W.conv("stride21", 2, 6, 90, 9, 3, 21), W.conv("stride22", 2, 6, 90, 9, 3, 22), W.conv("stride64", 3, 4, 130, 9, 2, 64, 1),
    W.conv("stride70", 2, 3, 211, 8, 70, 70, 0), W.linear("ragged", 61, 77, 70, dt=W.F32), W.linear("rows8", 8, 200, 9, dt=W.F32)],
    ids=lambda l: l.name)
def test_fp32_tiles_over_images(layer, bf16):
    """K-tiles that end inside an image, hold several, or are partly used; columns by rows of the map and by elements."""
    dw, ref = _dw(replace(layer, dt=W.BF16 if bf16 else W.F32), 0.5, B.PATH_FP32)
    assert rel_frobenius(dw, ref) <= 1e-5


@pytest.mark.parametrize("batch,c_in,c_out,k", [(256, 16, 20, 1), (300, 64, 64, 1), (64, 7, 9, 1), (64, 20, 20, 3)])
def test_reductions_of_small_weights(batch, c_in, c_out, k):
    layer = W.conv("r", batch, c_in, 8, c_out, k)
    dw, ref = _dw(layer, 0.5, B.PATH_TENSOR_CORE)
    assert rel_frobenius(dw, ref) <= 5e-3
    a, g = W.activation(layer, 5).cuda(), W.grad_out(layer, 5).cuda()
    comp, d = B.surgeon_prune_compact(a, 0.5), B.layer_desc(layer, B.PATH_TENSOR_CORE)
    acc = torch.ones(layer.dw_shape, device="cuda")
    B.surgeon_weight_grad(comp, d, g, dw=acc, accumulate=True)
    torch.testing.assert_close(acc, 1 + torch.from_numpy(dw).cuda(), rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("layer", [
    W.Layer("7x5", 1, 47, 4, 11, 35, 624, 7, 5, 1, 2), W.conv("5x5", 51, 4, 28, 605, 5)], ids=lambda l: l.name)
def test_tap_reduction_of_few_channels_and_many_outputs(layer):
    """A block of the tap reduction has fewer channels than it could take and several threads per element: its
    shared memory is that of the channels that exist (a buffer for 256 would exceed 48 KB)."""
    dw, ref = _dw(layer, 0.5, B.PATH_TENSOR_CORE)
    assert rel_frobenius(dw, ref) <= 5e-3


@pytest.mark.parametrize("layer", [
    W.linear("few_rows", 200, 320, 320), W.linear("ragged", 333, 136, 200), W.linear("wide", 260, 64, 1288),
    W.conv("one_image", 1, 40, 14, 72, 1, 1, 0), W.conv("one_image_3x3", 1, 24, 13, 56, 3), W.conv("taps_part", 2, 20, 8, 48, 3),
    W.conv("one_map", 1, 132, 16, 500, 1, 1, 0)], ids=lambda l: l.name)
@pytest.mark.parametrize("ratio", [0.5, 0.9])
def test_small_reductions_on_narrow_column_tiles(layer, ratio):
    """Fewer tiles than SMs: narrower column tiles, splits of four K-tiles, partial tiles of every width; and runs
    with few kept elements."""
    for dt in (W.BF16, W.F32):
        dw, ref = _dw(replace(layer, dt=dt), ratio, B.PATH_TENSOR_CORE)
        assert rel_frobenius(dw, ref) <= 5e-3


@pytest.mark.parametrize("layer", [
    W.linear("few_rows", 200, 320, 320), W.linear("ragged", 1333, 136, 200), W.conv("one_map", 1, 132, 16, 500, 1, 1, 0),
    W.conv("taps_part", 2, 20, 8, 48, 3), W.conv("s2", 2, 20, 14, 24, 3, 2)], ids=lambda l: l.name)
def test_layers_cut_into_fewer_parts(layer):
    """SURGEON_SHARE_GPU: other splits than the default's, in the scratch that the query asks for."""
    a, g = W.activation(layer, 5), W.grad_out(layer, 5)
    comp, ref = assert_store_equals_oracle(a, 0.5)
    d = B.layer_desc(layer, B.PATH_TENSOR_CORE)
    ws = torch.empty(B.surgeon_weight_grad_workspace(d), dtype=torch.uint8, device="cuda")
    dense = oracle.decompress(ref["bitmap"], ref["values"], a.numel())
    exp = oracle_dw(layer, dense.view(np.uint16) if layer.dt == W.BF16 else dense, g.numpy())
    for flags in (B.SURGEON_SHARE_GPU, 0):
        dw = B.surgeon_weight_grad(comp, d, g.cuda(), workspace=ws, flags=flags).cpu().numpy()
        assert rel_frobenius(dw, exp) <= 5e-3
    with pytest.raises(B.SurgeonError) as e:
        B.surgeon_weight_grad(comp, d, g.cuda(), workspace=ws, flags=B.SURGEON_STORE_DROP_ZEROS)
    assert e.value.status == B.SURGEON_ERR_INVALID_ARG


# prune: whole chunks and one element around them, resident and streamed ranges (a CTA's range is resident up to 48
# chunks of 4 KB), counts in global memory (beyond 512 chunks per CTA on 148 SMs)
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("chunks,extra", [(1, 0), (16, 1), (17, -1), (48 * 148, 0), (48 * 148, 1), (512 * 148 + 1, 3)])
def test_prune_ranges(chunks, extra, bf16):
    n = chunks * (2048 if bf16 else 1024) + extra
    x = W.draw("relu_normal", n, seed=4, device="cuda").cpu()
    x = x.to(torch.bfloat16) if bf16 else x
    for ratio in (0.3, 0.85):
        assert_store_equals_oracle(x, ratio)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("share", [0, B.SURGEON_SHARE_GPU])
@pytest.mark.parametrize("chunks,extra", [(48 * 148 + 600, 5), (48 * 148 + 601, 700), (512 * 148 + 33, 30)])
def test_partial_last_row_of_a_streamed_tensor(chunks, extra, share, bf16):
    """The emitting pass runs backwards: the place of the tensor's last chunk, whose partial row is put there by
    ordinary stores, is the first that another chunk's load fills.  Little or nothing of it is kept."""
    n = chunks * (2048 if bf16 else 1024) + extra
    x = W.draw("normal", n, seed=6, device="cuda").cpu()
    x = x.to(torch.bfloat16) if bf16 else x
    for tail, ratio in ((1.0, 0.95), (0.0, 0.7)):
        x[-(extra + 1500):] *= tail
        comp = B.surgeon_prune_compact(x.cuda(), ratio, flags=share)
        assert_store_equals_oracle(x, ratio, comp=comp)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("chunks,extra", [(1, -1), (49, 0), (48 * 37, 0), (48 * 37, 1), (1024 * 37, 0), (1024 * 37 + 1, 3)])
def test_prune_on_a_part_of_the_gpu(chunks, extra, bf16):
    """SURGEON_SHARE_GPU, asked for or implied by a stream that is not the current one: at most a quarter of the
    SMs, resident up to 48 chunks a CTA, counts in global memory beyond 1024."""
    n = chunks * (2048 if bf16 else 1024) + extra
    x = W.draw("relu_normal", n, seed=4, device="cuda").cpu()
    x = x.to(torch.bfloat16) if bf16 else x
    side = torch.cuda.Stream()
    for ratio in (0.3, 0.85):
        assert_store_equals_oracle(x, ratio, comp=B.surgeon_prune_compact(x.cuda(), ratio, flags=B.SURGEON_SHARE_GPU))
    xd = x.cuda()
    out = B.CompressedActivation(n, B.dtype_code(x.dtype), 0.0, "cuda")
    side.wait_stream(torch.cuda.current_stream())
    assert_store_equals_oracle(x, 0.85, comp=B.surgeon_prune_compact(xd, 0.85, out=out, stream=side))


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("chunks", [300 * 37, 385 * 37, 900 * 37 + 1])
def test_calls_in_a_row_on_a_part_of_the_gpu(chunks, bf16):
    """Lists of which a part, or most, is in global memory, read by eight lanes per chunk or by one, and
    chunks that have no tie; thirty calls with nothing to wait for in between."""
    n = chunks * (2048 if bf16 else 1024)
    for dist, ratio in (("normal", 0.95), ("relu_normal", 0.6)):
        x = W.draw(dist, n, seed=12, device="cuda")
        x = x.to(torch.bfloat16) if bf16 else x
        out = B.CompressedActivation(n, B.dtype_code(x.dtype), ratio, "cuda")
        ws = torch.zeros(out.sizes.workspace_bytes, dtype=torch.uint8, device="cuda")
        headers = []
        for _ in range(30):
            B.surgeon_prune_compact(x, ratio, out=out, workspace=ws, flags=B.SURGEON_SHARE_GPU)
            headers.append(out.header.clone())
        assert_store_equals_oracle(x.cpu(), ratio, comp=out)
        assert all(torch.equal(h, headers[-1]) for h in headers)


@pytest.mark.parametrize("bf16", [False, True])
def test_sample_that_misleads(bf16):
    """A short stretch holds all the large values: the strided sample sees few of them or none, so the bracket can
    miss and the select has to start over with what its counts prove."""
    n = 1 << 23
    for where in (0, n // 2 + 13, n - 5000):
        x = W.draw("normal", n, seed=9) * 1e-3
        x[where:where + 5000] = W.draw("normal", 5000, seed=10) * 100.0
        x = x.to(torch.bfloat16) if bf16 else x
        for ratio in (1 - 2500 / n, 1 - 5000 / n, 1 - 5200 / n):
            assert_store_equals_oracle(x, ratio)


@pytest.mark.parametrize("dist, n, bf16", [("normal", 9_000_001, False), ("relu_normal", 15_500_001, True),
                                           ("ties16", 8_000_000, False), ("normal", 40_000_003, False)])
def test_streamed_tensor_at_extreme_ratios(dist, n, bf16):
    """Thresholds of which a CTA's own sample holds few elements, or none, above or below; and more chunks per
    CTA than one trip to the lists takes."""
    x = W.draw(dist, n, seed=31, device="cuda")
    x = x.to(torch.bfloat16) if bf16 else x
    ratios = (0.9,) if n > 1 << 24 else (1 - 3 / n, 0.9995, 0.996, 0.5, 0.004, 0.0005, 2 / n)
    for ratio in ratios:
        assert_store_equals_oracle(x.cpu(), ratio)


def _awkward(kind, n, seed=0):
    """Values that lead the select off its usual way: brackets of many keys (bf16: more than the list's bytes can
    tell apart), all keys near the threshold in one place (lists and the keys of one CTA overflow), many more
    of them in a bin than CTA 0 takes at once, or a bin of few distinct keys with many copies each."""
    g = torch.Generator().manual_seed(n + seed)
    if kind == "log_uniform":
        return torch.exp2(240.0 * torch.rand(n, generator=g) - 120.0)
    if kind == "sorted":
        return torch.linspace(-1.0, 1.0, n)
    x = torch.randn(n, generator=g)
    if kind == "clustered":                      # a tenth of the tensor, in one place, has two in three of its keys in 1e-3 of the range
        x[n // 2:n // 2 + n // 10] = 1.0 + 1e-3 * torch.rand(n // 10, generator=g)
    if kind == "few_keys":                       # neighbouring fp32 numbers around the threshold, ten thousand copies each
        at = torch.randint(0, n, (n // 4,), generator=g)
        x[at] = (torch.tensor(1.0).view(torch.int32) + torch.randint(0, max(2, n // 40000), (n // 4,), generator=g)).int().view(torch.float32)
    return x


# two or three CTAs, resident, streamed; claimed (on a part of the GPU, where that begins at the fewest chunks)
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("n", [40000, 3_000_001, 18_000_003, "claimed"])
@pytest.mark.parametrize("kind", ["log_uniform", "sorted", "clustered", "few_keys"])
def test_select_off_its_usual_way(kind, n, bf16):
    flags = B.SURGEON_SHARE_GPU if n == "claimed" else 0
    n = (1024 * 37 + 1) * (2048 if bf16 else 1024) + 5 if flags else n
    xs = [_awkward(kind, n), 1.25 * _awkward(kind, n, 1).flip(0), torch.randn(n, generator=torch.Generator().manual_seed(n))]
    ratio = 1.0 - float((xs[0].abs() > 1.0005).double().mean()) if kind == "clustered" else 0.7
    refs = []
    for i, x in enumerate(xs):
        xs[i] = x = (x.to(torch.bfloat16) if bf16 else x).cuda()
        comp = B.surgeon_prune_compact(x, ratio)       # (claimed: the same tensor streamed on the whole GPU is the reference)
        if not flags:
            assert_store_equals_oracle(x.cpu(), ratio, comp=comp)
        refs.append([v.clone() for v in (comp.bitmap, comp.values, comp.block_offsets, comp.header)])
    x, out = xs[0].clone(), B.CompressedActivation(n, B.dtype_code(xs[0].dtype), ratio, "cuda")
    ws = torch.zeros(out.sizes.workspace_bytes, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.surgeon_prune_compact(x, ratio, out=out, workspace=ws, flags=flags)
    for i in (0, 1, 2, 1, 0, 0):                 # replays carry the same token, and find the scratch as another tensor's left it
        x.copy_(xs[i])
        for part in (out.bitmap, out.values, out.block_offsets):
            part.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert out.read_header().status == B.SURGEON_OK
        for got, ref in zip((out.bitmap, out.values, out.block_offsets, out.header), refs[i]):
            assert torch.equal(got.view(torch.uint8), ref.view(torch.uint8))


@pytest.mark.parametrize("n", [5000, (1 << 23) + 77])
def test_captured_call_replays_and_alternating_streams(n):
    xs = [W.draw("normal", n, seed=20 + i).cuda() for i in range(3)]
    ref = [B.surgeon_prune_compact(x, 0.8).to_numpy()[:3] for x in xs]
    x, out = xs[0].clone(), B.CompressedActivation(n, B.SURGEON_F32, 0.0, "cuda")
    ws = torch.empty(out.sizes.workspace_bytes, dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        B.surgeon_prune_compact(x, 0.8, out=out, workspace=ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.surgeon_prune_compact(x, 0.8, out=out, workspace=ws)
    for i in (1, 2, 0, 1):                      # the replays of one graph carry the same call
        x.copy_(xs[i])
        graph.replay()
        torch.cuda.synchronize()
        assert out.read_header().status == B.SURGEON_OK
        assert all(np.array_equal(u, v) for u, v in zip(out.to_numpy()[:3], ref[i]))
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = [B.CompressedActivation(n, B.SURGEON_F32, 0.0, "cuda") for _ in range(3)]
    wss = [torch.empty_like(ws) for _ in range(3)]
    torch.cuda.synchronize()
    for _ in range(4):
        for i in range(3):
            B.surgeon_prune_compact(xs[i], 0.8, out=outs[i], workspace=wss[i], stream=streams[i])
    torch.cuda.synchronize()
    for i in range(3):
        assert all(np.array_equal(u, v) for u, v in zip(outs[i].to_numpy()[:3], ref[i]))


@pytest.mark.parametrize("n", [5000, 1 << 20, 10_000_000])
def test_call_that_timed_out_leaves_no_words_behind(n):
    """Replays of a captured call carry one token, so the words {token, 8 bytes} that the CTAs exchange (the first
    12 x 256 + 12 x 258 pairs of the scratch) have to be gone after a call that gave up."""
    x = W.draw("normal", n, seed=8, device="cuda")
    out = B.CompressedActivation(n, B.SURGEON_F32, 0.0, "cuda")
    out.header.fill_(0x7777)                     # a header made by the call may hold anything
    ws = torch.zeros(out.sizes.workspace_bytes, dtype=torch.uint8, device="cuda")
    B.surgeon_prune_compact(x, 0.5, out=out, workspace=ws, flags=B.SURGEON_DEBUG_STALL_BARRIER)
    torch.cuda.synchronize()
    assert out.read_header().status == B.SURGEON_ERR_TIMEOUT and out.read_header().n_keep == 0
    tokens = ws[:16 * 12 * (256 + 258)].view(torch.int64).view(-1, 2)[:, 0]
    assert int(tokens.count_nonzero()) == 0
    assert_store_equals_oracle(x.cpu(), 0.5, comp=B.surgeon_prune_compact(x, 0.5, out=out, workspace=ws))


@pytest.mark.parametrize("n, flags", [(2_000_001, 0), (18_000_003, 0), (1024 * (1024 * 37 + 1), B.SURGEON_SHARE_GPU)])
def test_keys_reported_more_than_once(n, flags):
    """Two hundred copies of the threshold in one CTA: more keys than it can report, so the bin is narrowed and keys go
    into the same words again.  Each replay of one captured call has other values, and ordinary ones in between."""
    k = B.surgeon_compact_sizes(n, B.SURGEON_F32, 0.7).n_keep
    xs, refs = [], []
    for i in range(3):
        x = W.draw("normal", n, seed=60 + i, device="cuda") * (1.0 + 0.3 * i)
        if i != 1:
            at = n // 2 + 37 * torch.arange(200, device="cuda")
            x[at] = x.abs().kthvalue(n - k + 1).values * torch.tensor([1.0, -1.0], device="cuda").repeat(100)
        comp = B.surgeon_prune_compact(x, 0.7, flags=flags)
        assert_store_equals_oracle(x.cpu(), 0.7, comp=comp)
        xs.append(x)
        refs.append([v.copy() for v in comp.to_numpy()[:3]])
    x, out = xs[0].clone(), B.CompressedActivation(n, B.SURGEON_F32, 0.7, "cuda")
    ws = torch.zeros(out.sizes.workspace_bytes, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.surgeon_prune_compact(x, 0.7, out=out, workspace=ws, flags=flags)
    for i in (0, 2, 1, 2, 0, 0):
        x.copy_(xs[i])
        graph.replay()
        torch.cuda.synchronize()
        assert out.read_header().status == B.SURGEON_OK
        assert all(np.array_equal(u.view(np.uint8), v.view(np.uint8)) for u, v in zip(out.to_numpy()[:3], refs[i]))
        answered = ws[16 * 12 * 256:16 * 12 * (256 + 258)].view(torch.int64).view(12, 258, 2)[:, 0, 0].count_nonzero()
        assert flags or int(answered) >= 4       # two rounds and two last exchanges


KEY_WORDS = slice(16 * 12 * (256 + 258), 16 * 12 * (256 + 258) + 256 * 64 * 4)      # of the scratch: the keys that CTAs report


@pytest.mark.parametrize("n, flags", [(40000, 0), (3_000_001, 0), (18_000_003, 0), (1024 * (1024 * 37 + 1), B.SURGEON_SHARE_GPU)])
def test_scratch_that_holds_what_looks_like_keys(n, flags):
    """The scratch may hold anything, words with the very tag of the call among them (a replay carries the token of the
    one before): keys inside and outside the bin, in every place that a CTA reports keys in."""
    xs = [W.draw("normal", n, seed=40 + i, device="cuda") for i in range(2)]
    refs = []
    for x in xs:
        comp = B.surgeon_prune_compact(x, 0.7, flags=flags)
        assert_store_equals_oracle(x.cpu(), 0.7, comp=comp)
        refs.append([v.copy() for v in comp.to_numpy()[:3]] + [comp.read_header().threshold_key])
    x, out = xs[0].clone(), B.CompressedActivation(n, B.SURGEON_F32, 0.7, "cuda")
    ws = torch.zeros(out.sizes.workspace_bytes, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.surgeon_prune_compact(x, 0.7, out=out, workspace=ws, flags=flags)
    rng = np.random.default_rng(n)
    for turn in range(6):
        ref = refs[turn % 2]
        x.copy_(xs[turn % 2])
        if turn:
            low = token & 0xFFFFFFFF
            tags = np.array([low, low | 1] + [(low << 4 | p) & 0xFFFFFFFF for p in range(12)], dtype=np.uint64)
            near = (ref[3] + rng.integers(-300, 300, 8192)).astype(np.uint64)
            far = rng.integers(0, 1 << 32, 8192, dtype=np.uint64)
            words = tags[rng.integers(0, len(tags), 8192)] << np.uint64(32) | np.where(rng.random(8192) < 0.5, near, far)
            ws[KEY_WORDS].copy_(torch.from_numpy(words.view(np.uint8)))
        graph.replay()
        torch.cuda.synchronize()
        assert out.read_header().status == B.SURGEON_OK
        assert all(np.array_equal(u.view(np.uint8), v.view(np.uint8)) for u, v in zip(out.to_numpy()[:3], ref))
        answers = ws[16 * 12 * 256:KEY_WORDS.start].view(torch.int64).view(-1, 2)[:, 0].cpu()
        token = int(answers[answers != 0][0])


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("n", [1, 31, 1023, 1025, 4 * 8192 + 5])
def test_rebuild(n, bf16):
    x = W.draw("normal", n, seed=30)
    x = x.to(torch.bfloat16) if bf16 else x
    for ratio in (0.0, 0.5, 0.97):
        comp, ref = assert_store_equals_oracle(x, ratio)
        got = B.surgeon_decompress(comp).cpu()
        got = got.view(torch.int16).numpy() if bf16 else got.numpy()
        exp = oracle.decompress(ref["bitmap"], ref["values"], n)
        assert np.array_equal(got.view(np.uint8), exp.view(np.uint8))
