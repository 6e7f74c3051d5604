"""The one-sequence recurrence of wide layers at the edges of its slices and of its projection prologue (needs a B200)."""
import pytest

import lstm_workloads as wl
from gpu_util import assert_close, run_gpu

pytestmark = pytest.mark.gpu

# (layers, bidir, H, T): a last CTA with one, two and all units, both slice widths, the widest layer, two directions side by
# side and one after the other, T on both sides of the longest projection computed in the prologue
SHAPES = [(1, False, 1201, 3), (2, False, 1500, 40), (1, False, 1776, 41), (1, False, 1777, 5), (1, False, 2048, 4),
          (1, True, 1026, 4), (1, True, 1186, 3)]


@pytest.mark.parametrize("s", SHAPES, ids=lambda s: f"L{s[0]}D{1 + s[1]}_H{s[2]}_T{s[3]}")
def test_one_sequence_wide_layers(oracle, s):
    L, bidir, H, T = s
    w = wl.Workload("one", L, bidir, 40, H, T, 1, "bf16", 0.03, seed=H + T)
    weights, x = wl.make(w)
    h0, c0 = wl.make_states(w)
    ref = oracle.forward(weights, x, h0, c0, layers=L, bidir=bidir, hidden=H)
    assert_close(run_gpu(w, weights, x, h0, c0), ref, "bf16", "one")


def test_probe_measures_the_kernel_that_serves_the_call(oracle):
    import torch
    import paper_1901_10997_b200 as pkg
    w = wl.Workload("one_probe", 1, False, 40, 1201, 7, 1, "bf16", 0.03, seed=3)
    weights, x = wl.make(w)
    ref = oracle.forward(weights, x, layers=1, bidir=False, hidden=w.hidden)
    m = pkg.LSTM(weights, layers=1, in_dim=40, hidden=w.hidden, dtype="bf16", max_T=7, max_B=1)
    try:
        xd = torch.from_numpy(x).cuda()
        for mask in (1, 2, 4, 1 | 2, 4 | 2, pkg.LSTM_PROBE_WHOLE_STEP, 0):
            m.probe(mask)
            got = m.forward(xd)
            m.check()
            assert m.info()["kernel"] == pkg.LSTM_RAN_ONE
            if mask in (0, pkg.LSTM_PROBE_WHOLE_STEP):
                assert_close([t.cpu().numpy() for t in got], ref, "bf16", f"one/probe {mask}")
    finally:
        m.close()
