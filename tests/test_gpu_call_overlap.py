"""Banded calls of one pair and different sizes, one after another without
waiting: a call's first kernel runs beside the previous call's last one, on
the same scratch with other offsets.  Every call's results equal those of the
same call waited for, with falling and rising sizes, u8 and float rows, and
from host memory."""
import numpy as np
import pytest

import synth
from test_gpu_parity import mt  # noqa: F401

pytestmark = pytest.mark.gpu

KEYS = ("best", "second", "best_d", "second_d", "flags")
SIZES = [50000, 10000, 65000, 8000, 30000, 45000, 1500, 20000]


def scene(m, kind):
    rng = np.random.default_rng(m)
    K = synth.intrinsics(4800.0, 6048, 4032)
    F = synth.fundamental(K, K, synth.rotation([0, 1, 0], 5.0), [1.0, 0.2, 0.01])
    return synth.uniform_pair(rng, m, m - 3, F, eps=12.0, kind=kind, dim=128, w=6048, h=4032)


def match(mt, d):
    return mt.match(d["xy1"], d["xy2"], d["F"], d["eps"], d["desc1"], d["desc2"], d["kind"], d["dim"], d["width"],
                    d["height"])


@pytest.mark.parametrize("kinds", ["u8", "f32", "both"])
def test_sizes_in_turn(mt, kinds):
    U8, F32 = synth.DESC_U8_L2, synth.DESC_F32_L2
    pick = {"u8": [U8] * 8, "f32": [F32] * 8, "both": [U8, F32, F32, U8, U8, F32, U8, F32]}[kinds]
    ds = [mt.to_device(scene(m, k)) for m, k in zip(SIZES, pick)]
    mt.reserve(70000, 70000)
    mt.set_params(form=2, tune=0)
    try:
        want = [{k: v.clone() for k, v in match(mt, d).items()} for d in ds]
        mt.set_params(sync=False)
        for order in (list(range(8)), list(range(7, -1, -1))):
            outs = [(k, match(mt, ds[k])) for _ in range(4) for k in order]
            assert mt.sync() == 0
            for k, o in outs:
                for key in KEYS:
                    assert bool((o[key] == want[k][key]).all()), (SIZES[k], key)
    finally:
        mt.set_params(form=0, tune=1, sync=True)


def test_uneven_pairs_from_host_memory(mt):
    import torch

    scs = [scene(m, synth.DESC_U8_L2) for m in SIZES]
    mt.set_params(form=2, tune=0)
    try:
        want = [match(mt, mt.to_device(sc)) for sc in scs]
        pairs, outs, res, keep = [], [], [], []
        for sc in scs:
            h = {k: torch.as_tensor(np.ascontiguousarray(getattr(sc, k))).pin_memory()
                 for k in ("xy1", "xy2", "F", "desc1", "desc2")}
            pairs.append(mt.make_pair(h["xy1"], h["xy2"], h["F"], float(sc.eps), h["desc1"], h["desc2"], sc.kind,
                                      sc.dim, sc.width, sc.height))
            o = {k: torch.empty(sc.m, dtype=t, pin_memory=True)
                 for k, t in zip(KEYS, (torch.int32, torch.int32, torch.float32, torch.float32, torch.uint8))}
            outs.append(mt._out_struct(o, 0))
            res.append(o)
            keep.append(h)
        for _ in range(4):
            assert mt.egm_match_batch_host(pairs, outs) == 0
            for k, o in enumerate(res):
                for key in KEYS:
                    assert torch.equal(o[key], want[k][key].cpu()), (SIZES[k], key)
                    o[key].zero_()
    finally:
        mt.set_params(form=0, tune=1)
