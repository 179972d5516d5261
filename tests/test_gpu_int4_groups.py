"""The block-int4 expert kernel with many units per CTA: runs of whole row blocks and cut ones, every group and stage used
many times over, token counts on both sides of where the groups (three or two), the accumulators' width and the number of
chains in them change.  Tolerance: the library's own for block-int4 weights; the second projection's sums by themselves have a
bound of their own."""
import pytest
import torch

from gpu_util import check_outputs, run_case
from paper_2608_15018_b200 import binding, workloads
from paper_2608_15018_b200.workloads import CONFIGS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,f", [(2048, 3584), (512, 7168)])
@pytest.mark.parametrize("B", [1, 8, 9, 16, 17, 32, 33, 64])
def test_many_units(d, f, B):
    wl = CONFIGS["cfg4"].with_(d_model=d, d_ff=f, d_ff_shared=768, n_shared=1, shared_gate=True, sigma=1.0, seed=B)
    rep, _ = run_case(wl, n_tokens=B, plan=3, tok_list=sorted({0, B // 2, B - 1}))
    assert rep.plan == 3


# Error of a token's output (relative 2-norm, the largest of the batch) where nearly all of it comes from the second
# projection: the block scales are powers of two (every weight exact in binary16) and four columns of the hidden states differ
# from zero.  The tensor core truncates at every accumulation, so the error grows with the length of a chain of them: with
# two chains to a run of k-pieces measured 2.0 to 2.5e-7 (d_ff 1536) and 3.2 to 4.2e-7 (3072), with one chain 3.4 to 4.5e-7 and
# 6.6 to 8.6e-7; the bounds lie half way between them.
@pytest.mark.parametrize("f,bound", [(1536, 2.9e-7), (3072, 5.2e-7)])
@pytest.mark.parametrize("B", [8, 17, 24, 32])
@pytest.mark.parametrize("shared", [False, True])
def test_sums_of_the_second_projection(f, bound, B, shared):
    wl = CONFIGS["cfg4"].with_(d_model=4096, d_ff=256 if shared else f, d_ff_shared=f if shared else 0, n_shared=4 if shared else 0,
                               n_experts=4, top_k=1 if shared else 4, cap=4, seed=B)
    T = workloads.layer_weights(wl, 0, "cuda")
    for name, t in T.items():
        if t.dtype == torch.float16:
            T[name] = torch.exp2(torch.round(torch.log2(t.float().clamp_min(2.0 ** -14)))).half()
    H = workloads.hidden_states(wl, 0, B, device="cuda")
    H[:, 4:] = 0
    H[:, :4] = 16 + 8 * H[:, :4].clamp(-1, 1)
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=1, kernel_plan=3), [T]) as m:
        o = m.verify_layer(0, H)
        torch.cuda.synchronize()
        assert m.device_status() == 0
    assert check_outputs(wl, T, H, None, o).rms_rel_err <= bound
