"""Device memory of an environment against its budget.

Beside the operators, an environment holds the intermediates of one term chunk
(T and the partial tiles of K2), which t_budget_bytes bounds, and its plan.  The
plan of this window is 127,059 tasks of 24 bytes, its task lists (one entry per
left block and output block, at most one per task and block) and tiles, a few MB;
allocations are rounded up to 2 MB pieces.  16 MB are allowed for both.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MB = 1 << 20


@pytest.mark.parametrize("budget_mb", [32, 64, 200])
def test_fp64_intermediates_fit_the_budget(budget_mb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    ctx = P.Context(0, stream=torch.cuda.current_stream())
    cfg = synth.CONFIGS["qc16"]
    workload.build(ctx, cfg, t_budget_bytes=budget_mb * MB)[1].close()  # (loads what a first build loads)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    _, env = workload.build(ctx, cfg, t_budget_bytes=budget_mb * MB)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    assert env.info["t_chunk_bytes"] <= budget_mb * MB
    assert used <= env.info["env_bytes"] + budget_mb * MB + 16 * MB, used / MB
    env.close()
