"""A NaN in one unit of one batch row's state reaches what it reaches in the oracle, whichever kernel carries h (needs a B200)."""
import numpy as np
import pytest

import lstm_workloads as wl
from gpu_util import csr_weights, run_gpu

pytestmark = pytest.mark.gpu

# (dtype, bidir, H, B): fp32 with one, two, three and four tiles of eight batch rows; bf16 with one row and several
CASES = [("fp32", False, 100, 1), ("fp32", True, 74, 9), ("fp32", False, 296, 20), ("fp32", False, 33, 32), ("fp32", False, 400, 3),
         ("bf16", False, 300, 1), ("bf16", False, 1201, 1), ("bf16", True, 150, 3), ("bf16", False, 700, 17)]


@pytest.mark.parametrize("c", CASES, ids=lambda c: f"{c[0]}_D{1 + c[1]}_H{c[2]}_B{c[3]}")
def test_nan_in_one_unit(oracle, c):
    dtype, bidir, H, B = c
    w = wl.Workload("nan", 1, bidir, 24, H, 6, B, dtype, min(0.3, 1 / H ** 0.5), seed=H + B)
    weights, x = wl.make(w)
    h0, c0 = wl.make_states(w)
    c0[0, B - 1, H // 3] = np.nan
    ref = oracle.forward(weights, x, h0, c0, layers=1, bidir=bidir, hidden=H)
    assert np.isnan(ref[0][0]).sum() == 1 and np.isnan(ref[0][1:, B - 1, :H]).all()      # one unit, then its whole row
    for name, got, want in zip(("y", "hT", "cT"), run_gpu(w, weights, x, h0, c0), ref):
        assert np.array_equal(np.isnan(got), np.isnan(want)), name
        ok = ~np.isnan(want)
        assert np.abs(got - want)[ok].max(initial=0) <= wl.TOLERANCE[dtype], name


@pytest.mark.parametrize("H,B", [(300, 5), (600, 3), (600, 20)])
def test_nan_in_one_unit_of_a_pruned_batch(oracle, H, B):
    # (all 24 bits of h in a word; the removed weights are multiplied, so the NaN reaches the whole row one step later)
    w = wl.Workload("nan", 1, False, 24, H, 6, B, "bf16", min(0.3, 1 / H ** 0.5), density=0.3, seed=H + B)
    weights, x = wl.make(w)
    h0, c0 = wl.make_states(w)
    ref = oracle.forward(weights, x, h0, c0, layers=1, bidir=False, hidden=H)
    c0[0, B - 1, H // 3] = np.nan
    y, hT, cT = run_gpu(w, csr_weights(oracle, weights), x, h0, c0, exec_mode="csr")
    assert np.isnan(y[0]).sum() == 1 and np.isnan(y[0, B - 1, H // 3])
    assert np.isnan(y[2:, B - 1]).all() and np.isnan(hT[0, B - 1]).all() and np.isnan(cT[0, B - 1]).all()
    for got, want in ((y[:, :-1], ref[0][:, :-1]), (hT[:, :-1], ref[1][:, :-1]), (cT[:, :-1], ref[2][:, :-1])):
        assert np.abs(got - want).max() <= wl.TOLERANCE["bf16"]
