"""The compact list of matches around the number of tiles from which their
counts are scanned, and around the scan's rounds: indices, values and count
against a plain selection."""
import pytest

from test_gpu_match import mt  # noqa: F401

pytestmark = pytest.mark.gpu

TILE = 2048


@pytest.mark.parametrize("m", [1, TILE, 6143 * TILE, 6144 * TILE, 6144 * TILE + 1, 8192 * TILE - 1, 8192 * TILE + 1,
                               20480 * TILE + 77])
@pytest.mark.parametrize("share", [0.0, 0.01, 1.0])
def test_counts_of_many_tiles(mt, m, share):
    import torch

    g = torch.Generator(device="cuda").manual_seed(m)
    fl = (torch.rand(m, device="cuda", generator=g) < share).to(torch.uint8) * 2 + 1
    best = torch.randint(-1, 1 << 20, (m,), dtype=torch.int32, device="cuda", generator=g)
    qi, rj = mt.compact_matches(fl, best, 2)
    want = torch.nonzero(fl & 2).flatten()
    assert torch.equal(qi, want.to(torch.int32)) and torch.equal(rj, best[want])
