"""Candidate rows of images beyond one bitmap's range: rows sorted in registers
(128 to 1024 keys) and rows walked range by range, at the lengths and
image sizes where the ways change, and several pairs of which one is large.
Every row equals the oracle's (brute force)."""
import numpy as np
import pytest

from test_gpu_parity import check_candidates
from test_gpu_rows import mt, rows_scene, run  # noqa: F401

pytestmark = pytest.mark.gpu

LENS = [0, 1, 33, 64, 65, 96, 127, 128, 129, 200, 255, 256, 257, 383, 384, 385, 511, 512, 513, 700, 1023, 1024, 1025, 2000]


@pytest.mark.parametrize("n", [65535, 65536, 65537, 131072, 131073, 196609, 262144, 262145, 520001])
@pytest.mark.parametrize("contiguous", [False, True])
def test_lengths(mt, n, contiguous):
    sc = rows_scene(LENS, n, 1.0, n, contiguous)
    out = run(mt, sc, sum(LENS))
    assert np.array_equal(np.diff(out["cand_offsets"]), LENS)
    check_candidates(out, sc)


def test_large_and_small_pairs_in_one_call(mt):
    scs = [rows_scene(LENS, n, 1.0, k) for k, n in enumerate((12000, 140_000, 70_000, 10_500))]
    o = mt.match_batch([mt.to_device(s) for s in scs], csr=True, cand_capacity=4 * sum(LENS))
    off, idx = o["cand_offsets"].cpu().numpy(), o["cand_idx"].cpu().numpy()
    for k, sc in enumerate(scs):
        a, b = k * len(LENS), (k + 1) * len(LENS)
        part = {"cand_offsets": off[a:b + 1] - off[a], "cand_idx": idx[off[a]:off[b]]}
        check_candidates(part, sc)
