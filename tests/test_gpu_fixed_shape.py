"""Banded calls whose tile shape no timing decides: the sizes on both sides of
the rule's lines (tiles per SM and estimated candidates a query), where the
shape and the items of a tile change, of one pair and of several, matches and
candidate counts.  All equal the plain form's."""
import numpy as np
import pytest

import synth
from test_gpu_parity import check_candidates, check_matches, mt  # noqa: F401
from test_gpu_tile_split import KEYS, scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [synth.DESC_U8_L2, synth.DESC_BIN256])
@pytest.mark.parametrize("tiles", [152, 182, 183, 405, 406, 608, 609])
@pytest.mark.parametrize("eps", [0.02, 20.0, 120.0])
def test_matches(mt, kind, tiles, eps):
    d = mt.to_device(scene(128 * tiles - 1, 1200, eps, tiles, kind))
    args = (d["xy1"], d["xy2"], d["F"], d["eps"], d["desc1"], d["desc2"], d["kind"], d["dim"], d["width"], d["height"])
    try:
        mt.set_params(form=1, tune=0)
        ref = {k: v.cpu().numpy() for k, v in mt.match(*args).items()}
        mt.set_params(form=2, tune=0)
        got = {k: v.cpu().numpy() for k, v in mt.match(*args).items()}
    finally:
        mt.set_params(form=0, tune=1)
    for k in KEYS:
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("m", [23000, 24000])
@pytest.mark.parametrize("eps", [8.0, 120.0])
def test_counts(mt, m, eps):
    sc = scene(m, 1200, eps, m)
    d = mt.to_device(sc)
    o = mt.match(d["xy1"], d["xy2"], d["F"], d["eps"], d["desc1"], d["desc2"], d["kind"], d["dim"], d["width"],
                 d["height"], csr=True, cand_capacity=m * 1200)
    check_candidates({k: v.cpu().numpy() for k, v in o.items()}, sc)


def test_several_pairs(mt):
    items = [mt.to_device(scene(5000 + k, 1100, 90.0, k)) for k in range(5)]
    try:
        mt.set_params(form=1, tune=0)
        ref = {k: v.cpu().numpy() for k, v in mt.match_batch(items).items()}
        mt.set_params(form=2, tune=0)
        got = {k: v.cpu().numpy() for k, v in mt.match_batch(items).items()}
    finally:
        mt.set_params(form=0, tune=1)
    for k in KEYS:
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("tiles", [1, 152, 304, 305])
@pytest.mark.parametrize("eps", [0.05, 30.0, 300.0])
def test_floats(mt, tiles, eps):
    """Float rows on both sides of two tiles per SM; matches and counts."""
    sc = synth.uniform_pair(np.random.default_rng(tiles), 128 * tiles - 3, 230,
                            synth.fundamental(*2 * [synth.intrinsics(500.0, 640, 480)],
                                              synth.rotation([0, 1, 0], 5.0), [1.0, 0.1, 0.02]),
                            eps=eps, kind=synth.DESC_F32_L2, dim=128)
    d = mt.to_device(sc)
    args = (d["xy1"], d["xy2"], d["F"], d["eps"], d["desc1"], d["desc2"], d["kind"], d["dim"], d["width"], d["height"])
    try:
        mt.set_params(form=2, tune=0)
        got = {k: v.cpu().numpy() for k, v in mt.match(*args).items()}
    finally:
        mt.set_params(form=0, tune=1)
    ref = check_matches(got, sc)
    out = {k: v.cpu().numpy() for k, v in mt.match(*args, csr=True, cand_capacity=sc.m * 230).items()}
    check_candidates(out, sc)
    check_matches(out, sc, ref)
