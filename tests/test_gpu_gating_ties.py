"""Selection where logits or importances are equal, or equal in the upper half of their 64 bits (the gating
compares 32 bits at a time and takes an exact path then).  All numbers are dyadic, so logits, importances
and biases are exact in float64 whatever the order of the sums, and the selection has to be the oracle's,
order included.  Also: experts of large importance that no token selects (the expert kernel may have
started on them), and a single row of confidences equal to zero."""
import numpy as np
import pytest
import torch

from gpu_util import check_outputs
from oracle import layer as oracle_layer
from oracle import parity
from paper_2608_15018_b200 import binding, workloads
from paper_2608_15018_b200.workloads import BF16, CONFIGS, F32

pytestmark = pytest.mark.gpu


def _run(wl, T, H, conf):
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=1, kernel_plan=3), [T]) as m:
        o = m.verify_layer(0, H, conf)
        torch.cuda.synchronize()
        assert m.device_status() == 0
        lists = m.debug_lists()
    parity.check_bucketing(lists, o.sel_idx.cpu().numpy(), o.sel_w.cpu().numpy(), wl.n_experts, wl.n_shared)
    ocfg, ow = parity.from_workload(wl, T)
    ref = oracle_layer(ocfg, ow, workloads.raw_numpy(H), None if conf is None else conf.cpu().numpy().astype(np.float64), tok_list=[0])
    assert np.array_equal(o.sel_idx.cpu().numpy(), ref.sel)
    check_outputs(wl, T, H, conf, o)
    return ref.sel


@pytest.mark.parametrize("fine", [0.0, 2.0 ** -24, 2.0 ** -3], ids=["equal", "equal upper halves", "plain"])
@pytest.mark.parametrize("E,k,cap,B", [(16, 2, 4, 1), (64, 8, 18, 8), (64, 6, 12, 64), (128, 4, 6, 16), (200, 3, 5, 9), (256, 8, 8, 5)])
def test_ties(E, k, cap, B, fine):
    wl = CONFIGS["cfg2"].with_(d_model=64, d_ff=32, n_experts=E, top_k=k, cap=cap, alpha=0.5, n_layers=1, router_dtype=F32, act_dtype=BF16)
    T = workloads.layer_weights(wl, 0, "cuda")
    g = torch.Generator().manual_seed(E + B)
    r = torch.zeros(E, 64)
    r[:, 0] = torch.randint(0, 3, (E,), generator=g) / 2.0          # few distinct values
    r[:, 1] = torch.randint(-4, 5, (E,), generator=g).float()       # told apart by the second column only
    T["router"] = r.cuda()
    H = torch.zeros(B, 64)
    H[:, 0] = 2.0 ** torch.randint(-1, 2, (B,), generator=g).float()
    H[:, 1] = fine
    conf = (2.0 ** -torch.randint(0, 4, (B,), generator=g).float()).cuda()
    _run(wl, T, H.to(torch.bfloat16).cuda(), conf)
    _run(wl, T, H.to(torch.bfloat16).cuda(), torch.zeros(B, device="cuda"))   # every importance is 0


@pytest.mark.parametrize("weight_dtype", [BF16, workloads.Q4B32])
@pytest.mark.parametrize("k,B", [(1, 8), (2, 8), (8, 8), (8, 2)])
def test_experts_of_large_importance_that_no_token_selects(k, B, weight_dtype):
    """Expert 0 is nearly as good as the best for every token (largest importance), but token b prefers
    experts of its own; the bias is off."""
    wl = CONFIGS["cfg2"].with_(d_model=256, d_ff=256, n_experts=64, top_k=k, cap=64, n_layers=1, weight_dtype=weight_dtype, router_dtype=F32)
    T = workloads.layer_weights(wl, 0, "cuda")
    r = torch.full((64, 256), -1.0)
    r[:8] = 0.5
    H = torch.zeros(B, 256)
    for b in range(B):
        H[b, b] = 1.0
        for j in range(k):
            r[8 + (k * b + j) % 56, b] = 1.0 + j / 8.0
    T["router"] = r.cuda()
    sel = _run(wl, T, H.to(torch.bfloat16).cuda(), None)
    assert sel.min() >= 8
