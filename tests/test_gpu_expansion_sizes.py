"""The admission kernels at the edges of their layouts (words in registers, rows in shared memory, rows too large for
it; test_gpu_expansion_close has the layouts in registers one by one):
bit-exact against the oracle, through the check of test_gpu_expansion."""
import pytest

from test_gpu_expansion import test_expand_matches_oracle as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_layers,n_experts,k", [(2, 1, 64, 2), (31, 33, 64, 2), (65, 100, 256, 3), (256, 101, 64, 2),
                                                  (200, 128, 256, 2)])
def test_expand_sizes(n, n_layers, n_experts, k):
    check(n, n_layers, n_experts, k)
