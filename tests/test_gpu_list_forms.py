"""Candidate lists and matches of the form the library picks for them, just
where it changes over (few and many candidates, tiles and references, one pair
and several, each kind of rows, tolerances per keypoint): the form picked is
the documented one and everything equals the plain form's, bit by bit.  (Not
calls that mix float rows with others: their plain kernel adds a float row's
squares in another order.)"""
import numpy as np
import pytest

import synth
from test_gpu_parity import mt  # noqa: F401

pytestmark = pytest.mark.gpu

U8, F32, BIN = synth.DESC_U8_L2, synth.DESC_F32_L2, synth.DESC_BIN256
KEYS = ("best", "second", "best_d", "second_d", "flags", "cand_offsets", "cand_idx")


def scene(m, n, row, kind, seed, per_keypoint=False):
    """About `row` candidates a query."""
    rng = np.random.default_rng(seed)
    K = synth.intrinsics(4800.0, 6048, 4032)
    F = synth.fundamental(K, K, synth.rotation([0, 1, 0], 5.0), [1.0, 0.2, 0.01])
    eps = row / n * 6048 * 4032 / (2 * 0.8 * np.hypot(6048, 4032))
    sc = synth.uniform_pair(rng, m, n, F, w=6048, h=4032, eps=eps, kind=kind, dim=256 if kind == BIN else 128)
    if per_keypoint:
        sc.eps = np.full(n, eps) * rng.uniform(0.5, 1.5, n)
    return sc


def both_forms(mt, scenes, cap):
    items, got = [mt.to_device(s) for s in scenes], []
    for form in (0, 1):
        mt.set_params(form=form)
        mt.set_timing(True)
        try:
            o = mt.match_batch(items, csr=True, cand_capacity=cap)
            banded = mt.timing()["banded_calls"]
        finally:
            mt.set_timing(False)
            mt.set_params(form=0)
        got.append(({k: o[k].cpu().numpy() for k in KEYS}, banded))
    (a, banded), (b, plain) = got
    assert plain == 0
    for k in KEYS:
        assert np.array_equal(a[k], b[k]), k
    return banded


@pytest.mark.parametrize("m,n,row,kind,banded", [
    (3000, 3000, 60, U8, 1), (3000, 3000, 20, U8, 0), (3000, 6100, 60, U8, 0), (9000, 19000, 900, U8, 1), (20000, 3000, 320, U8, 1),
    (45000, 45000, 4, U8, 0), (45000, 30000, 200, U8, 1), (40000, 150000, 30, U8, 0),
    (45000, 45000, 10, BIN, 0), (45000, 45000, 400, BIN, 1), (45000, 45000, 10, F32, 0), (45000, 20000, 250, F32, 1)])
def test_one_pair(mt, m, n, row, kind, banded):
    assert both_forms(mt, [scene(m, n, row, kind, m + row)], int(m * row * 2.5)) == banded


@pytest.mark.parametrize("kinds,pairs,m,row,banded", [([U8], 8, 2000, 10, 0), ([U8], 20, 6000, 80, 1), ([BIN], 20, 6000, 200, 1),
                                                      ([F32], 20, 6000, 100, 1), ([F32], 6, 3000, 20, 0),
                                                      ([U8, BIN], 6, 4000, 60, 1), ([U8, BIN], 6, 1500, 12, 0)])
def test_several_pairs(mt, kinds, pairs, m, row, banded):
    scs = [scene(m - 37 * k, m + 11 * k, row, kinds[k % len(kinds)], k) for k in range(min(pairs, 4))]
    assert both_forms(mt, [scs[k % len(scs)] for k in range(pairs)], int(pairs * m * row * 2.5)) == banded


@pytest.mark.parametrize("m,banded", [(5000, 0), (100_000, 1)])
def test_tolerances_per_keypoint(mt, m, banded):
    assert both_forms(mt, [scene(m, 4000, 30, U8, m, per_keypoint=True)], m * 100) == banded
