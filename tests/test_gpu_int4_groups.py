"""The block-int4 expert kernel with many units per CTA: runs of whole row blocks and cut ones, every group and stage used
many times over, token counts on both sides of where the groups (three or two), the accumulators' width and the number of
chains in them change.  Tolerance: the library's own for block-int4 weights."""
import pytest

from gpu_util import run_case
from paper_2608_15018_b200.workloads import CONFIGS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,f", [(2048, 3584), (512, 7168)])
@pytest.mark.parametrize("B", [1, 8, 9, 16, 17, 32, 33, 64])
def test_many_units(d, f, B):
    wl = CONFIGS["cfg4"].with_(d_model=d, d_ff=f, d_ff_shared=768, n_shared=1, shared_gate=True, sigma=1.0, seed=B)
    rep, _ = run_case(wl, n_tokens=B, plan=3, tok_list=sorted({0, B // 2, B - 1}))
    assert rep.plan == 3
