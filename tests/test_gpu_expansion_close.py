"""The admission kernel where an approximate utility cannot decide: utilities that differ in the last places of float32
or float64, that are equal, that lie at 1, and operands outside the ranges of the approximation (zero, negative, tiny,
huge, not a number), in every layout of the words in registers (1 to 32 threads a candidate, two and four pairs of words each,
blocks on both sides of 512 threads) and beyond them.  Decisions exactly those of the oracle."""
import random

import numpy as np
import pytest
import torch

from oracle import expansion as ox
from test_gpu_expansion import _masks_tensor

pytestmark = pytest.mark.gpu


def _f32(x):
    return float(np.float32(x))


def _operands(kind, n, rng):
    """(p_tok, c_draft, t_ar, t_exp)"""
    ulps = [_f32(np.nextafter(np.float32(0.75), np.float32(2), dtype=np.float32)), 0.75,
            _f32(np.nextafter(np.float32(0.75), np.float32(0), dtype=np.float32))]
    near = [rng.choice(ulps) for _ in range(n)]
    if kind == "last places":
        return near, [0.5] * n, 64.0, 0.125
    if kind == "at one":          # benefit and cost of a candidate with four new experts agree to the last place of p
        return near, [0.25] * n, 1.0, 0.125
    if kind == "products":        # prefix products that differ in the last places of float64 only
        return [rng.choice([_f32(1 / 3), _f32(0.1), _f32(0.7)]) for _ in range(n)], [0.0625] * n, 8.0, _f32(0.01)
    if kind == "zero costs":
        return near, [rng.choice([0.0, 0.5]) for _ in range(n)], 4.0, rng.choice([0.0, 0.25])
    if kind == "signs":
        return ([rng.choice([0.0, -0.0, 0.5, 0.75]) for _ in range(n)], [rng.choice([-0.0, -0.5, 0.25]) for _ in range(n)],
                2.0, 0.125)
    if kind == "tiny":
        return [x * 2.0 ** -80 for x in near], [2.0 ** -82] * n, 1.0, 2.0 ** -84
    if kind == "equal":
        return [1.0] * n, [0.5] * n, 64.0, 0.125
    if kind == "no draft cost":   # c_draft NULL: a candidate that brings nothing new costs nothing, whatever its confidence
        return [rng.choice([0.0, 1e-30, 0.5, 0.75, 0.75]) for _ in range(n)], None, 16.0, 0.125
    if kind == "not a number":
        return [rng.choice([float("nan"), 0.5, 0.75, 0.875]) for _ in range(n)], [0.25] * n, 16.0, 0.125
    if kind == "huge benefit":
        return [rng.choice([2.0 ** 90, 0.5]) for _ in range(n)], [0.25] * n, 4.0, 0.125
    if kind == "huge":
        return near, [2.0 ** 100] * n, 2.0 ** 102, 2.0 ** 98
    return near, [rng.choice([0.5, float("inf")]) for _ in range(n)], 16.0, 0.125


@pytest.mark.parametrize("kind", ["last places", "at one", "products", "zero costs", "signs", "tiny", "huge", "infinite", "equal",
                                  "no draft cost", "not a number", "huge benefit"])
@pytest.mark.parametrize("n,n_layers,n_experts", [(5, 1, 64), (64, 16, 64), (33, 9, 128), (64, 48, 128), (65, 3, 64),
                                                  (96, 24, 128), (160, 48, 128), (256, 20, 128), (1, 48, 128), (32, 48, 128),
                                                  (32, 128, 128), (8, 128, 128), (64, 32, 64), (33, 16, 64), (128, 16, 64),
                                                  (129, 16, 64), (256, 8, 64)])
def test_close_and_extreme_utilities(n, n_layers, n_experts, kind):
    from paper_2608_15018_b200 import binding

    dev = torch.device("cuda", 0)
    rng = random.Random(n + 7 * n_layers)
    p_tok, c_draft, t_ar, t_exp = _operands(kind, n, rng)
    parent = [-1 if i < 3 or rng.random() < 0.5 else rng.randrange(i) for i in range(n)]
    # few different sets, four experts each, spread over the layers
    sets = [[0] * n_layers for _ in range(8)]
    for s in sets:
        for _ in range(4):
            s[rng.randrange(n_layers)] |= 1 << rng.randrange(n_experts)
    masks = [list(rng.choice(sets)) for _ in range(n)]
    want_adm, want_order, want_union = ox.adaptive_expand(parent, p_tok, masks, c_draft or [0.0] * n, t_ar, t_exp)
    words = (n_experts + 63) // 64
    adm, order, n_adm, union = binding.adaptive_expand(
        torch.tensor(parent, dtype=torch.int32, device=dev), torch.tensor(p_tok, dtype=torch.float32, device=dev),
        _masks_tensor(masks, words, dev), n_experts, None if c_draft is None else torch.tensor(c_draft, dtype=torch.float32, device=dev),
        t_ar, t_exp)
    torch.cuda.synchronize()
    assert order.cpu().tolist() == want_order + [-1] * (n - len(want_order))
    assert adm.cpu().tolist() == want_adm and n_adm.item() == len(want_order)
    got = union.cpu().numpy().view(np.uint64)
    assert [sum(int(got[l, w]) << (64 * w) for w in range(words)) for l in range(n_layers)] == want_union
