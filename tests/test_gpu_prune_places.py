"""Places that every CTA adds up from what the others show (thresholds known after one exchange): narrow and wide brackets,
thresholds of zero, one key everywhere, and replays of a captured call, whose words of the replay before are still there."""
import numpy as np
import pytest
import torch

from paper_2503_20354_b200 import binding as B
from paper_2503_20354_b200 import workloads as W
from gpu_util import assert_store_equals_oracle

pytestmark = pytest.mark.gpu


# a bf16 bracket near 0 spans many octaves (more than 256 keys), one in the body of the distribution some dozens
@pytest.mark.parametrize("ratio", [0.004, 0.03, 0.1, 0.5, 0.97])
@pytest.mark.parametrize("dist", ["normal", "relu_normal", "ties16"])
@pytest.mark.parametrize("n", [700, 40000, 1_200_011, (15 << 20) + 3])
def test_bf16_against_the_oracle(n, dist, ratio):
    x = W.draw(dist, n, seed=n % 97).to(torch.bfloat16)
    assert_store_equals_oracle(x, ratio)
    if dist == "relu_normal":
        assert_store_equals_oracle(x, ratio, drop_zeros=True)


@pytest.mark.parametrize("n, bf16", [(60_000, True), (1_500_001, True), ((15 << 20) + 3, True), (1_500_001, False), ((9 << 20) + 3, False)])
def test_replays_with_other_values(n, bf16):
    """Every tensor keeps its large values in another part, so that places left by an earlier replay are wrong."""
    xs, refs = [], []
    for i in range(3):
        x = W.draw("relu_normal", n, seed=i, device="cuda")
        x[i * n // 3:(i + 1) * n // 3] *= 3.0 + i
        x = x.to(torch.bfloat16) if bf16 else x
        xs.append(x)
        refs.append([v.copy() for v in B.surgeon_prune_compact(x, 0.6 if bf16 else 0.3).to_numpy()[:3]])
        assert_store_equals_oracle(x.cpu(), 0.6 if bf16 else 0.3)
    x, out = xs[0].clone(), B.CompressedActivation(n, B.dtype_code(xs[0].dtype), 0.6 if bf16 else 0.3, "cuda")
    ws = torch.zeros(out.sizes.workspace_bytes, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.surgeon_prune_compact(x, 0.6 if bf16 else 0.3, out=out, workspace=ws)
    for i in (1, 0, 2, 2, 1, 0, 2):
        x.copy_(xs[i])
        graph.replay()
        torch.cuda.synchronize()
        assert out.read_header().status == B.SURGEON_OK
        assert all(np.array_equal(u.view(np.uint8), v.view(np.uint8)) for u, v in zip(out.to_numpy()[:3], refs[i]))


@pytest.mark.parametrize("n, bf16", [(1_500_001, False), (9 << 20, False), (1_500_001, True)])
def test_every_execution_has_its_own_tag(n, bf16):
    """What the CTAs show is told from an earlier replay's by a count of executions: words of the scratch that grow by one
    from each replay to the next, at least one for each of dozens of CTAs."""
    x = W.draw("relu_normal", n, seed=1, device="cuda")
    x = x.to(torch.bfloat16) if bf16 else x
    out = B.CompressedActivation(n, B.dtype_code(x.dtype), 0.6, "cuda")
    ws = torch.zeros((out.sizes.workspace_bytes + 7) // 8, dtype=torch.int64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.surgeon_prune_compact(x, 0.6, out=out, workspace=ws.view(torch.uint8))
    seen = []
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        seen.append(ws.clone())
    grown = ((seen[1] - seen[0] == 1) & (seen[2] - seen[1] == 1)).sum().item()
    assert grown >= 32, grown
