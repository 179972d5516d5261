"""Infinite and NaN hidden states: router logits are float64 sums of products of the stored values, so a token
that holds one gets infinite or NaN logits and NaN mixing weights, and no other token's logits change.
Both forms of the logit pass, both activation types, elements in the first and last columns."""
import pytest
import torch

from paper_2608_15018_b200 import binding, workloads
from paper_2608_15018_b200.workloads import CONFIGS

pytestmark = pytest.mark.gpu

INF, NAN = float("inf"), float("nan")


def _batch(wl, B, bad):
    H = workloads.hidden_states(wl, 0, B, device="cuda")
    for b, col, value in bad:
        H[b, col] = value
    return H


def _want(H, router):
    """float64 logits: the products of the non-finite elements decide, whatever the order of the sum."""
    return H.double() @ router.double().T


# (74 rows and 64 tokens: the logit pass by warp tasks; the others by row blocks, 1 to 4 passes)
@pytest.mark.parametrize("E,B,plan", [(24, 1, 0), (24, 4, 0), (24, 7, 0), (64, 40, 0), (74, 64, 0), (74, 64, 4), (24, 7, 4)])
@pytest.mark.parametrize("act", [workloads.BF16, workloads.F32])
def test_logits_of_a_layer(E, B, plan, act):
    if act == workloads.F32 and plan == 4:
        pytest.skip("the one-launch plan takes bf16 activations")
    wl = CONFIGS["cfg2"].with_(d_model=2624, d_ff=64, n_experts=E, top_k=4, cap=8, alpha=0.0, n_layers=1, act_dtype=act)
    T = workloads.layer_weights(wl, 0, "cuda")
    bad = [(B - 1, 2623, -INF)] if B == 1 else [(0, 0, INF), (B // 2, 1311, NAN), (B - 1, 2623, -INF)]
    H = _batch(wl, B, bad)
    rows = sorted({b for b, _, _ in bad})
    good = [b for b in range(B) if b not in rows]
    clean = H.clone()
    for b, col, _ in bad:
        clean[b, col] = 0.0
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=1, kernel_plan=plan), [T]) as m:
        ref = m.verify_layer(0, clean)
        torch.cuda.synchronize()
        ref_logits = m.debug_lists()["logits"].clone()
        o = m.verify_layer(0, H)
        torch.cuda.synchronize()
        assert m.device_status() == 0
        logits = m.debug_lists()["logits"]
    want = _want(H, T["router"]).cpu()
    for b in rows:
        assert torch.equal(torch.isnan(logits[b]), torch.isnan(want[b])), b
        keep = ~torch.isnan(want[b])
        assert torch.isinf(want[b][keep]).all() and torch.equal(logits[b][keep], want[b][keep]), b
        assert torch.isnan(o.sel_w[b]).all() and torch.isnan(o.out[b]).any(), b
    assert torch.equal(logits[good], ref_logits[good])
    assert torch.equal(o.sel_idx[good], ref.sel_idx[good]) and torch.equal(o.sel_w[good], ref.sel_w[good])
    assert torch.isfinite(o.out[good]).all()


@pytest.mark.parametrize("alpha", [0.0, 0.5])
def test_routing_without_a_context(alpha):
    wl = CONFIGS["cfg2"].with_(d_model=512, n_experts=64, top_k=8, cap=16, alpha=alpha)
    T = workloads.layer_weights(wl, 0, "cuda")
    H = _batch(wl, 6, [(2, 100, INF), (5, 511, NAN)])
    sel, w, n, _ = binding.route_noalloc(binding.Config.from_workload(wl, n_layers=1), H, T["router"])
    assert binding.route_noalloc_status() == 0
    assert torch.isnan(w[[2, 5]]).all()
    assert int(sel.min()) >= 0 and int(sel.max()) < 64 and 8 <= int(n) <= 48
    for b in range(6):
        assert len(set(sel[b].tolist())) == 8
    if alpha == 0.0:
        clean = H.clone()
        clean[2, 100] = clean[5, 511] = 0.0
        sel0, w0, _, _ = binding.route_noalloc(binding.Config.from_workload(wl, n_layers=1), clean, T["router"])
        good = [0, 1, 3, 4]
        assert torch.equal(sel[good], sel0[good]) and torch.equal(w[good], w0[good])
