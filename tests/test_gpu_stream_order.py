"""Weights that the work in front of a call on its stream writes are the ones that the call uses, also where
that work is a kernel which lets its successor start before it has written them (programmatic launch)."""
import pytest
import torch

from gpu_util import check_outputs
from paper_2608_15018_b200 import binding, workloads
from paper_2608_15018_b200.workloads import CONFIGS

pytestmark = pytest.mark.gpu

# waits at most `cycles` of its own clock, a fraction of a millisecond, then copies n 16-byte units
WRITER = r"""
extern "C" __global__ void late_copy(uint4 *dst, const uint4 *src, int n, int cycles)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long t0 = clock64();
    while (clock64() - t0 < cycles) {}
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i];
}
"""


def _write(how, kernel, dst, src):
    if how == "copy":
        dst.copy_(src)
    else:
        n = dst.numel() * dst.element_size() // 16
        kernel(grid=(8, 1, 1), block=(256, 1, 1), args=[dst.view(-1), src.view(-1), n, 400000])


@pytest.mark.parametrize("how", ["copy", "early trigger"])
@pytest.mark.parametrize("call", ["layer", "stack", "graph"])
@pytest.mark.parametrize("cfg,B", [("cfg3", 8), ("cfg3", 16), ("cfg5", 4), ("cfg5", 33)])
@pytest.mark.parametrize("early", [True, False])
def test_weights_written_just_before_the_call(cfg, B, early, call, how, monkeypatch):
    if not early:
        monkeypatch.setenv("S2MOE_NO_EARLY", "1")
    wl = CONFIGS[cfg].with_(d_model=512, d_ff=256, n_experts=16, cap=8, d_ff_shared=1024, n_layers=2)
    kernel = torch.cuda._compile_kernel(WRITER, "late_copy") if how != "copy" else None
    names = ("sh_gate", "sh_up", "sh_down", "w_gate", "w_up", "w_down", "router")
    old = [workloads.layer_weights(wl.with_(seed=91), l, "cuda") for l in range(2)]
    new = [workloads.layer_weights(wl, l, "cuda") for l in range(2)]
    H = torch.stack([workloads.hidden_states(wl, l, B, device="cuda") for l in range(2)])
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=2, kernel_plan=3), old) as m:
        o = m.alloc_outputs(B, stack=True)
        views = [binding.LayerOutput(o.out[l], o.sel_idx[l], o.sel_w[l], o.n_unique[l:l + 1]) for l in range(2)]
        m.verify_stack(H, None, o)
        torch.cuda.synchronize()
        if "sh_scale" in new[0]:
            for l in range(2):
                old[l]["sh_scale"].copy_(new[l]["sh_scale"])
        # the shared experts' weights last: the writer directly in front of the call
        def refresh():
            for name in reversed(names):
                for l in (1, 0):
                    if call != "layer" or l == 0 or not name.startswith("sh_"):
                        _write(how, kernel, old[l][name], new[l][name])

        if call == "graph":
            side = torch.cuda.Stream()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                refresh()
                m.verify_stack(H, None, o, stream=side)
            graph.replay()
        elif call == "stack":
            refresh()
            m.verify_stack(H, None, o)
        else:
            refresh()
            m.verify_layer(0, H[0], None, views[0])
            for name in ("sh_down", "sh_up", "sh_gate"):
                _write(how, kernel, old[1][name], new[1][name])
            m.verify_layer(1, H[1], None, views[1])
        torch.cuda.synchronize()
        assert m.device_status() == 0
    for l in range(2):
        check_outputs(wl, new[l], H[l], None, views[l])


@pytest.mark.parametrize("how", ["copy", "early trigger"])
@pytest.mark.parametrize("call", ["layer", "stack", "graph"])
@pytest.mark.parametrize("cfg,B", [("cfg1", 1), ("cfg1", 9), ("cfg2", 4), ("cfg4", 4)])
def test_weights_written_just_before_the_call_of_the_cuda_core_kernels(cfg, B, call, how):
    """The second kernel of kernel plan 1 reads the routing kernel's tables and weights before it waits for the first: both
    layers' weights written in front of the call, the second layer's again between the two calls of single layers."""
    wl = CONFIGS[cfg].with_(d_model=256, d_ff=512, n_experts=12, top_k=3, cap=6, n_layers=2, n_shared=1, d_ff_shared=256,
                            shared_gate=True)
    kernel = torch.cuda._compile_kernel(WRITER, "late_copy") if how != "copy" else None
    old = [workloads.layer_weights(wl.with_(seed=91), l, "cuda") for l in range(2)]
    new = [workloads.layer_weights(wl, l, "cuda") for l in range(2)]
    H = torch.stack([workloads.hidden_states(wl, l, B, device="cuda") for l in range(2)])
    with binding.S2MoE(binding.Config.from_workload(wl, n_layers=2, kernel_plan=1), old) as m:
        o = m.alloc_outputs(B, stack=True)
        views = [binding.LayerOutput(o.out[l], o.sel_idx[l], o.sel_w[l], o.n_unique[l:l + 1]) for l in range(2)]
        m.verify_stack(H, None, o)
        torch.cuda.synchronize()
        side = torch.cuda.Stream()

        def refresh(l):
            for name in sorted(new[l], key=lambda n: "down" in n):       # W_down last
                if new[l][name].numel() * new[l][name].element_size() % 16:
                    old[l][name].copy_(new[l][name])
                else:
                    _write(how, kernel, old[l][name], new[l][name])

        def calls(stream=None):
            if call == "layer":
                for l in range(2):
                    refresh(l)
                    m.verify_layer(l, H[l], None, views[l], stream=stream)
            else:
                for l in (1, 0):
                    refresh(l)
                m.verify_stack(H, None, o, stream=stream)

        if call == "graph":
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                calls(side)
            graph.replay()
        else:
            calls()
        torch.cuda.synchronize()
        assert m.device_status() == 0
    for l in range(2):
        check_outputs(wl, new[l], H[l], None, views[l])
