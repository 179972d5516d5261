"""The block-int4 expert kernel (kernel plan 3) at the sizes where it can go wrong: the smallest widths (one
stage per row block, one unit per run), token counts around the padding steps and where three groups of
dequantising warps give way to two, shared experts, few and many experts, more units per CTA than its table holds, with the
early start and without.  Tolerance: the library's own for block-int4 weights."""
import pytest

from gpu_util import run_case
from paper_2608_15018_b200.workloads import CONFIGS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("early", [True, False])
@pytest.mark.parametrize("d,f,f_sh", [(256, 256, 0), (512, 768, 256), (1280, 256, 1024)])
@pytest.mark.parametrize("B", [1, 8, 9, 16, 17, 32, 33, 64])
def test_token_counts_and_widths(d, f, f_sh, B, early, monkeypatch):
    if not early:
        monkeypatch.setenv("S2MOE_NO_EARLY", "1")
    wl = CONFIGS["cfg4"].with_(d_model=d, d_ff=f, d_ff_shared=f_sh, n_shared=2 if f_sh else 0, shared_gate=bool(f_sh),
                               n_experts=12, top_k=3, cap=5, sigma=1.0, seed=B)
    rep, _ = run_case(wl, n_tokens=B, plan=3)
    assert rep.plan == 3 and rep.tokens_checked == B


@pytest.mark.parametrize("E,k,B", [(1, 1, 1), (2, 1, 64), (256, 16, 5), (200, 2, 40)])
def test_few_and_many_experts(E, k, B):
    wl = CONFIGS["cfg4"].with_(d_model=256, d_ff=256, n_experts=E, top_k=k, cap=min(E, 2 * k), sigma=1.0, seed=E)
    rep, _ = run_case(wl, n_tokens=B, plan=3)
    assert rep.plan == 3 and rep.tokens_checked == B


def test_more_units_than_the_table_of_a_cta_holds():
    wl = CONFIGS["cfg4"].with_(d_model=256, d_ff=14336, n_experts=256, top_k=16, cap=256, sigma=1.0, n_layers=1)
    rep, _ = run_case(wl, n_tokens=64, plan=3, tok_list=list(range(0, 64, 9)))
    assert rep.plan == 3


@pytest.mark.parametrize("B", [57, 64])
def test_row_blocks_without_tokens(B):
    """12 router rows and a wide model: a third of the row blocks gets no tokens, and some of them still write a
    part of the binary16 copy of the hidden states that the expert kernel reads behind their arrival."""
    wl = CONFIGS["cfg4"].with_(d_model=8192, d_ff=256, n_experts=12, top_k=3, cap=5, sigma=1.0, seed=B)
    for _ in range(4):
        rep, _ = run_case(wl, n_tokens=B, plan=3)
        assert rep.plan == 3 and rep.tokens_checked == B


def test_largest_tables():
    """All limits at once: the tables leave two stages of the ring, one per group of dequantising warps."""
    wl = CONFIGS["cfg4"].with_(d_model=512, d_ff=256, d_ff_shared=512, n_shared=4, shared_gate=True, n_experts=256, top_k=16,
                               cap=256, sigma=1.0, n_layers=1)
    rep, _ = run_case(wl, n_tokens=64, plan=3, tok_list=list(range(0, 64, 7)))
    assert rep.plan == 3
