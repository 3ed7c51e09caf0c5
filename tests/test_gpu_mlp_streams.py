"""The tolerance network on a non-blocking stream, used as soon as it is made
or loaded: its weights, moments and cleared sums are in place before the first
call's kernels (the legacy default stream, which such a stream is not ordered
after, is kept busy meanwhile)."""
import numpy as np
import pytest

from test_gpu_mlp import bf16, feats, mt, oracle_u, params  # noqa: F401
from test_gpu_train import data, reference

pytestmark = pytest.mark.gpu


def test_first_calls_after_create_and_load(mt):
    import torch
    from paper_2603_18401_gb300 import Matcher

    th, other = params(11), params(12)
    f, r = data(th, 300, 1)
    gref, _ = reference(th, f, r, 0.9)
    F, R = torch.as_tensor(f).cuda().contiguous(), torch.as_tensor(r).cuda().contiguous()
    busy = torch.empty(1 << 26, device="cuda")
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    own = Matcher(0, stream=s)
    for _ in range(20):
        for _ in range(4):
            busy.fill_(1.0)  # on the legacy default stream
        net = own.tolnet(th)
        with torch.cuda.stream(s):
            g, _ = net.grad(F, R, 0.9)
        s.synchronize()
        # the bound of test_gpu_train.py for a batch of this size
        d = np.abs(g.cpu().numpy().astype(np.float64) - gref)
        assert np.all(d <= 2e-5 * np.abs(gref).max() + 2e-5 * np.abs(gref))
        z = np.zeros_like(th)
        for _ in range(4):
            busy.fill_(1.0)
        net.load_state({"params": other, "adam_m": z, "adam_v": z, "step": 0})
        with torch.cuda.stream(s):
            e = net.infer(F)
        net.load_state({"params": th, "adam_m": z, "adam_v": z, "step": 0})
        want = mt.tolnet(other).infer(F)
        s.synchronize()
        assert torch.equal(e, want)
        net.close()
    own.close()
