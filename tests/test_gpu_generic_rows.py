"""The matching kernel of rows that no warp-per-query instance covers: blocks
whose windows take no, one and several rounds of 1,024 elements, one pair and
several, and calls without descriptors; candidate counts and lists against the
brute force, matches against the oracle."""
import numpy as np
import pytest

import synth
from test_gpu_parity import check_candidates, check_matches, mt  # noqa: F401

pytestmark = pytest.mark.gpu

U8, F32, BIN = synth.DESC_U8_L2, synth.DESC_F32_L2, synth.DESC_BIN256


def scene(m, n, eps, kind, dim, seed):
    rng = np.random.default_rng(seed)
    K = synth.intrinsics(500.0, 640, 480)
    F = synth.fundamental(K, K, synth.rotation([0, 1, 0], 5.0), [1.0, 0.1, 0.02])
    return synth.uniform_pair(rng, m, n, F, eps=eps, kind=kind, dim=dim)


@pytest.mark.parametrize("kind,dim", [(U8, 48), (U8, 512), (BIN, 384), (F32, 96), (F32, 256)])
@pytest.mark.parametrize("n,eps", [(40, 0.01), (700, 1.0), (3000, 6.0)])
@pytest.mark.parametrize("pairs", [1, 3])
def test_counts_lists_and_matches(mt, kind, dim, n, eps, pairs):
    scs = [scene(70 + 33 * k, n + 5 * k, eps, kind, dim, 10 * k + n) for k in range(pairs)]
    mt.set_params(form=1)
    mt.set_counters(True)
    try:
        o = mt.match_batch([mt.to_device(s) for s in scs], csr=True, cand_capacity=sum(s.m * s.n for s in scs))
        found = mt.stats()["candidates"]
    finally:
        mt.set_counters(False)
        mt.set_params(form=0)
    o = {k: v.cpu().numpy() for k, v in o.items()}
    assert found == o["cand_offsets"][-1]
    at = 0
    for sc in scs:
        off = o["cand_offsets"][at:at + sc.m + 1]
        check_candidates({"cand_offsets": off - off[0], "cand_idx": o["cand_idx"][off[0]:off[-1]]}, sc)
        check_matches({k: o[k][at:at + sc.m] for k in ("best", "second", "best_d", "second_d", "flags")}, sc)
        at += sc.m


@pytest.mark.parametrize("n,eps", [(40, 0.01), (3000, 6.0)])
def test_without_descriptors(mt, n, eps):
    sc = scene(100, n, eps, U8, 32, n)
    d = mt.to_device(sc)
    o = mt.match(d["xy1"], d["xy2"], d["F"], d["eps"], None, None, 0, 32, sc.width, sc.height, csr=True,
                 cand_capacity=100 * n)
    check_candidates({k: v.cpu().numpy() for k, v in o.items()}, sc)
    assert bool((o["best"] == -1).all())
