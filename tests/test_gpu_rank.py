"""Fundamental matrices off rank 2, as estimates are whose rank was not
enforced: the lines then miss the computed epipole, most of all those of
queries near image 1's epipole.  Matches equal the oracle's, for one pair and
several, integer and float rows; and such a query widens its own window, not
those of the whole pair (counted by the references visited)."""
import numpy as np
import pytest

import synth
from test_gpu_parity import check_matches, mt  # noqa: F401

pytestmark = pytest.mark.gpu

U8, F32, BIN = synth.DESC_U8_L2, synth.DESC_F32_L2, synth.DESC_BIN256
KEYS = ("best", "second", "best_d", "second_d", "flags")


def scene(m, n, t, off, kind, seed, per_keypoint=False):
    """Smallest singular value `off` times the second (in coordinates of about unit size); a few queries close to
    image 1's epipole where that is finite."""
    rng = np.random.default_rng(seed)
    K = synth.intrinsics(500.0, 640, 480)
    N = np.diag([1 / 500.0, 1 / 500.0, 1.0])
    F = synth.fundamental(K, K, synth.rotation([0, 1, 0], 4.0), t)
    U, S, V = np.linalg.svd(np.linalg.inv(N).T @ F @ np.linalg.inv(N))
    e1 = np.linalg.inv(N) @ V[2]
    S[2] = off * S[1]
    F = N.T @ (U * S) @ V @ N
    eps = np.exp(rng.uniform(-2.0, 1.0, n)) if per_keypoint else 0.5
    sc = synth.uniform_pair(rng, m, n, F, eps=eps, kind=kind, dim=256 if kind == BIN else 128)
    if abs(e1[2]) > 1e-6:
        sc.xy1[:6] = e1[:2] / e1[2] + np.array([[0.01, 0], [0, 0.3], [1, 1], [-5, 2], [20, 0], [0, -40]])
    return sc


def run(mt, scenes):
    items = [mt.to_device(s) for s in scenes]
    mt.set_params(form=1)
    try:
        o = {k: v.cpu().numpy() for k, v in mt.match_batch(items).items()}
    finally:
        mt.set_params(form=0)
    out, at = [], 0
    for s in scenes:
        out.append({k: o[k][at:at + s.m] for k in KEYS})
        at += s.m
    return out


POSES = [[0.05, 0.02, 1.0], [1.0, 0.2, 0.05], [1.0, 0.3, 0.0]]


@pytest.mark.parametrize("off", [1e-7, 1e-4, 1e-2, 0.3])
@pytest.mark.parametrize("t", POSES)
@pytest.mark.parametrize("kind", [U8, F32, BIN])
def test_matches(mt, off, t, kind):
    one = scene(700, 650, t, off, kind, 1)
    check_matches(run(mt, [one])[0], one)
    several = [scene(300 + 57 * k, 500 - 31 * k, t, off, kind, 2 + k, per_keypoint=k == 1) for k in range(3)]
    for sc, o in zip(several, run(mt, several)):
        check_matches(o, sc)


@pytest.mark.parametrize("kind", [U8, F32, BIN])
@pytest.mark.parametrize("pairs", [1, 3])
def test_references_visited(mt, kind, pairs):
    """A line misses the epipole by about 1e-4 of the image's size, 0.06 px, and by more only near image 1's epipole:
    a window of 0.5 px then holds a few per cent of the references, that of the pair's worst query all of them."""
    scs = [scene(2000, 2000, POSES[0], 1e-4, kind, 5 + k) for k in range(pairs)]
    mt.set_counters(True)
    try:
        run(mt, scs)
        visited = mt.stats()["window_refs"]
    finally:
        mt.set_counters(False)
    assert visited < 0.1 * 2000 * 2000 * pairs
