"""Kernel plan 3 keeps state between the calls of a context (activation maps of a batch size, importances that must be
zero again, words and counters between its two kernels): one context, batches of changing size back to back with
nothing waited for in between, every call against the oracle, eagerly and from captured graphs."""
import pytest
import torch

from gpu_util import check_outputs
from paper_2608_15018_b200 import binding, workloads
from paper_2608_15018_b200.workloads import CONFIGS

pytestmark = pytest.mark.gpu

SIZES = (8, 64, 1, 17, 48, 2, 33, 8)
LAYERS = 3


def _workload(cfg):
    shared = dict(n_shared=1, d_ff_shared=512, shared_gate=True)
    return CONFIGS[cfg].with_(d_model=512, d_ff=256, n_experts=24, top_k=4, cap=8, sigma=0.6, n_layers=LAYERS,
                              **(shared if cfg in ("cfg3", "cfg4") else {}))


def _layer(o, l):
    return binding.LayerOutput(o.out[l], o.sel_idx[l], o.sel_w[l], o.n_unique[l:l + 1])


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("cfg", ["cfg2", "cfg3", "cfg4"])
def test_batches_of_changing_size_in_one_context(cfg, graph):
    wl = _workload(cfg)
    W = [workloads.layer_weights(wl, l, "cuda") for l in range(LAYERS)]
    calls = []
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=LAYERS, kernel_plan=3), W) as m:
        for i, B in enumerate(SIZES):
            w = wl.with_(seed=100 + i)
            H = torch.stack([workloads.hidden_states(w, l, B, device="cuda") for l in range(LAYERS)])
            C = torch.stack([workloads.confidences(w, l, B) for l in range(LAYERS)]).cuda()
            calls.append((H, C, m.alloc_outputs(B, stack=True)))
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            for H, C, o in calls:
                m.verify_stack(H, C, o)
            if graph:
                graphs = []
                for H, C, o in calls:
                    graphs.append(torch.cuda.CUDAGraph())
                    with torch.cuda.graph(graphs[-1], stream=side):
                        m.verify_stack(H, C, o, stream=side)
                for _, _, o in calls:
                    o.out.zero_()
                for k in (0, 1, 2, 3, 4, 5, 6, 7, 1, 0, 5, 3):
                    graphs[k].replay()
        torch.cuda.synchronize()
        assert m.device_status() == 0
    for H, C, o in calls:
        for l in range(LAYERS):
            check_outputs(wl, W[l], H[l], C[l], _layer(o, l))


@pytest.mark.parametrize("B", [1, 8, 24, 64])
def test_int4_weights_that_are_exact_in_binary16(B):
    """Block scales that are powers of two: every weight is exact in binary16, so what is left of the error is that of
    the activations' two binary16 parts (2^-23 of a value at most) and of the fp32 sums, measured 1.5 to 2.2e-7.  Without
    the second part it would be up to 2^-12 of a value, 1.4e-4 over a layer."""
    wl = _workload("cfg4")
    T = workloads.layer_weights(wl, 0, "cuda")
    for name, t in T.items():
        if t.dtype == torch.float16:
            T[name] = torch.exp2(torch.round(torch.log2(t.float().clamp_min(2.0 ** -14)))).half()
    H = workloads.hidden_states(wl, 0, B, device="cuda")
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=1, kernel_plan=3), [T]) as m:
        o = m.verify_layer(0, H)
        torch.cuda.synchronize()
        assert m.device_status() == 0
    rep = check_outputs(wl, T, H, None, o)
    assert rep.rms_rel_err <= 1e-6
