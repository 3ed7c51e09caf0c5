"""The GMS filter's sorted form, which many pairs and fine grids take: pairs of
uneven sizes (one empty), cells of one match and of thousands, ties and
matches on cell boundaries, just below and above the sizes where the forms
change over; flag by flag against the oracle."""
import numpy as np
import pytest

from oracle import gms as ogms
from test_gpu_gms_cells import boundary_coords
from test_gpu_match import mt  # noqa: F401

pytestmark = pytest.mark.gpu


def pair(rng, m, n, grid, crowd):
    (w1, h1), (w2, h2) = (1023, 767), (6048, 4031)
    xy1 = np.c_[boundary_coords(rng, m, grid, w1), boundary_coords(rng, m, grid, h1)]
    xy2 = np.c_[boundary_coords(rng, n, grid, w2), boundary_coords(rng, n, grid, h2)]
    best = rng.integers(-1, n, m)
    k = int(crowd * m)  # a coherent part, so that some cells pass and lists are long
    if k:
        best[:k] = rng.integers(0, 40, k)
        xy1[:k] = xy1[rng.integers(0, 30, k)]
    return xy1, xy2, best, (rng.random(m) < 0.9).astype(np.uint8) * 3, (w1, h1), (w2, h2)


@pytest.mark.parametrize("grid,pairs,m", [(1, 200, 300), (2, 64, 700), (20, 200, 400), (25, 64, 900), (48, 3, 500),
                                          (48, 4, 500), (48, 12, 1300), (36, 9, 2500), (31, 40, 513), (48, 1, 200_000)])
def test_batches(mt, grid, pairs, m):
    import torch

    rng = np.random.default_rng(100 * grid + pairs)
    ps = [pair(rng, 0 if pairs > 1 and k == 1 else m + 37 * (k % 5), m, grid, (0.0, 0.5, 1.0)[k % 3] if pairs > 1 else 0.5)
          for k in range(min(pairs, 8))]
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a)).to(mt.device)
    items = []
    for k in range(pairs):
        x1, x2, b, f, s1, s2 = ps[k % len(ps)]
        items.append((dev(x1), dev(x2), dev(b.astype(np.int32)), dev(f), s1, s2))
    mt.gms_batch(items, require=2, grid=grid, alpha=3.0)
    want = [ogms.gms(x1, x2, b, f, s1, s2, require=2, grid=grid, alpha=3.0) for x1, x2, b, f, s1, s2 in ps]
    kept = 0
    for k, it in enumerate(items):
        got = it[3].cpu().numpy()
        assert np.array_equal(got, want[k % len(ps)]), k
        kept += np.count_nonzero(got & 32)
    assert kept > 0 or m < 1000  # (few matches on many cells: none may pass)
