"""The bf16 expert kernel that cuts the first projection by rows (kernel plan 3) at the sizes where it can
go wrong: widths that are no multiple of a task, row block or k-tile, one k-tile, a last row block of 64
rows, token counts around the padding steps, few and many experts, and the layouts of W_gate and W_up in
memory (ascending, descending, the same matrix twice).  Tolerance: the library's own for bf16 weights."""
import pytest
import torch

from gpu_util import check_outputs, run_case
from paper_2608_15018_b200 import binding, workloads
from paper_2608_15018_b200.workloads import CONFIGS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,f,f_sh", [(64, 32, 32), (128, 96, 160), (192, 1056, 0), (576, 224, 2080), (1152, 544, 64)])
@pytest.mark.parametrize("B", [1, 8, 9, 17, 33, 64])
def test_ragged_sizes(d, f, f_sh, B):
    wl = CONFIGS["cfg3"].with_(d_model=d, d_ff=f, d_ff_shared=f_sh, n_shared=2 if f_sh else 0, shared_gate=bool(f_sh),
                               n_experts=24, top_k=3, cap=6, seed=B)
    rep, _ = run_case(wl, n_tokens=B, plan=3)
    assert rep.plan == 3 and rep.tokens_checked == B


@pytest.mark.parametrize("E,k,B", [(1, 1, 1), (2, 1, 64), (256, 16, 5), (200, 2, 40)])
def test_few_and_many_experts(E, k, B):
    wl = CONFIGS["cfg2"].with_(d_model=256, d_ff=320, n_experts=E, top_k=k, cap=min(E, 2 * k), sigma=1.0, seed=E)
    rep, _ = run_case(wl, n_tokens=B, plan=3)
    assert rep.plan == 3 and rep.tokens_checked == B


@pytest.mark.parametrize("shared_gate", [False, True])
@pytest.mark.parametrize("E,B", [(72, 48), (73, 64), (74, 64), (74, 47), (100, 48)])
def test_both_forms_of_the_logit_pass(E, B, shared_gate):
    """Two sets of row blocks fit beside each other up to 73 router rows (148 SMs); with more rows, batches of
    48 tokens and more take the logit pass by warp tasks."""
    wl = CONFIGS["cfg3"].with_(d_model=512, d_ff=96, d_ff_shared=64 if shared_gate else 0, n_shared=int(shared_gate),
                               shared_gate=shared_gate, n_experts=E, top_k=4, cap=20, sigma=1.0, seed=E)
    rep, _ = run_case(wl, n_tokens=B, plan=3)
    assert rep.plan == 3 and rep.tokens_checked == B


@pytest.mark.parametrize("layout", ["up_first", "tied"])
def test_layouts_of_gate_and_up(layout):
    wl = CONFIGS["cfg3"].with_(d_model=320, d_ff=352, d_ff_shared=416, n_experts=10, top_k=2, cap=4, n_layers=1)
    T = workloads.layer_weights(wl, 0, "cuda")
    for g, u in (("w_gate", "w_up"), ("sh_gate", "sh_up")):
        if layout == "tied":
            T[u] = T[g]
        else:
            both = torch.stack([T[u], T[g]])
            T[u], T[g] = both[0], both[1]
            assert T[u].data_ptr() < T[g].data_ptr()
    H = workloads.hidden_states(wl, 0, 11, device="cuda")
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=1, kernel_plan=3), [T]) as m:
        o = m.verify_layer(0, H)
        assert m.device_status() == 0
    check_outputs(wl, T, H, None, o)


def test_large_expert_count_and_width_still_run():
    """256 experts of a wide layer: the task table of a CTA is at its largest."""
    wl = CONFIGS["cfg2"].with_(d_model=64, d_ff=14336, n_experts=256, top_k=16, cap=256, sigma=1.0, n_layers=1)
    rep, _ = run_case(wl, n_tokens=64, plan=3, tok_list=list(range(0, 64, 9)))
    assert rep.plan == 3


def test_early_start_that_does_not_fit():
    """One token of one wide expert: the plan fits for the expert that is selected, but not for one more that the
    early start would read beside it, so the batch runs without the early start."""
    wl = CONFIGS["cfg2"].with_(d_model=64, d_ff=400000, n_experts=2, top_k=1, cap=2, n_layers=1)
    rep, _ = run_case(wl, n_tokens=1, plan=3)
    assert rep.plan == 3 and rep.tokens_checked == 1


@pytest.mark.parametrize("E,k,f,B", [(2, 1, 400000, 2), (256, 16, 40000, 16)])
def test_very_wide_experts(E, k, f, B):
    """More units of the first projection than a 32-bit product with the units of an expert holds, and more tasks per
    CTA than 1024: both are bounded by the shared memory of the table only."""
    wl = CONFIGS["cfg2"].with_(d_model=64, d_ff=f, n_experts=E, top_k=k, cap=E, sigma=1.0, n_layers=1)
    rep, _ = run_case(wl, n_tokens=B, plan=3, tok_list=[0, B - 1])
    assert rep.plan == 3 and rep.tokens_checked == 2


# Relative 2-norm of a token's error, the largest over the batch.  The bf16 hi + lo parts of the activations give about
# 2.4e-6; what the tensor core truncates at every accumulation adds to it in proportion to the length L of a chain:
# the sum of squares of 2.4e-6 and c * L fits two, four and eight chains with c = 3.7e-8 (OLMoE width, L = 64, 32, 16).
# The bounds lie half way between the measured errors (2.5, 3.0, 3.1, 3.2, 3.6, 2.7, 2.7 and 3.6e-6) and those of
# chains of twice and four times the length (3.2, 4.5, 4.8, 4.8, 4.8, 3.7, 4.6 and 5.5e-6).
@pytest.mark.parametrize("cfg,B,bound", [("cfg2", 1, 2.9e-6), ("cfg2", 8, 3.7e-6), ("cfg2", 20, 3.9e-6), ("cfg2", 48, 4.0e-6),
                                         ("cfg2", 64, 4.2e-6), ("cfg3", 16, 3.2e-6), ("e128b", 8, 3.6e-6), ("e128b", 64, 4.5e-6)])
def test_error_against_float64(cfg, B, bound):
    wl = CONFIGS[cfg].with_(n_experts=16, cap=2 * CONFIGS[cfg].top_k)
    rep, _ = run_case(wl, n_tokens=B, plan=3)
    assert rep.plan == 3 and rep.rms_rel_err <= bound


def test_ctas_without_tasks():
    """Narrow experts of a wide model: most CTAs get no task, copy the hidden states into shared memory all the same
    and make room for the next layer's CTA."""
    wl = CONFIGS["cfg2"].with_(d_model=2048, d_ff=32, n_experts=2, top_k=1, cap=2, n_layers=6, n_tokens=8)
    W = [workloads.layer_weights(wl, l, "cuda") for l in range(6)]
    H = torch.stack([workloads.hidden_states(wl, l, 8, device="cuda") for l in range(6)])
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=6, kernel_plan=3), W) as m:
        o = m.alloc_outputs(8, stack=True)
        for _ in range(20):
            m.verify_stack(H, None, o)
        torch.cuda.synchronize()
        assert m.device_status() == 0
    for l in range(6):
        check_outputs(wl, W[l], H[l], None, binding.LayerOutput(o.out[l], o.sel_idx[l], o.sel_w[l], o.n_unique[l:l + 1]))
