"""How many kernels a step launches depends on its sizes; the benchmark line counts them."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H_q,H_kv,want", [
    (256, 1, 1, 3),         # statistics in clusters: no fold
    (16384, 32, 8, 4),      # statistics in slices with V's tiles, fold, Q and K tiles, attention
    (65536, 40, 8, 5),      # V in a launch of its own
])
def test_launches_of_a_step(N, H_q, H_kv, want):
    import bench
    from paper_2609_33135_b200 import binding
    q, k, v = (torch.zeros(1, N, h, 128, dtype=torch.bfloat16, device="cuda") for h in (H_q, H_kv, H_kv))
    ws = binding.quantize_workspace(1, H_q, H_kv)
    s1 = binding.stage1(q, k, v, workspace=ws)
    out, status = torch.empty_like(q), torch.zeros(1, dtype=torch.int32, device="cuda")

    def step():
        binding.stage1(q, k, v, workspace=ws, out=s1)
        binding.prefill(s1, True, 0.088, out=out, status=status)

    step()
    torch.cuda.synchronize()
    assert bench.kernels_launched(step) == want
