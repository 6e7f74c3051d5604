"""The batched recurrence at the edges of its row groups, passes and K groups, against the oracle (needs a B200)."""
import pytest

import lstm_workloads as wl
from gpu_util import assert_close, csr_weights, run_gpu

pytestmark = pytest.mark.gpu

# (layers, bidir, H, T, B, density): 8 / 9 / 24 / 33 / 56 rows, two passes of unequal size, K halves that end inside a
# 16-column piece, a group of one piece, pruned weights
SHAPES = [
    (1, False, 390, 4, 8, 1.0), (1, True, 401, 3, 9, 1.0), (1, False, 66, 3, 24, 1.0), (2, False, 513, 3, 33, 1.0),
    (1, False, 1500, 2, 56, 1.0), (1, False, 300, 3, 101, 1.0), (2, False, 200, 4, 7, 0.2), (1, True, 700, 3, 16, 0.1),
]


@pytest.mark.parametrize("s", SHAPES, ids=lambda s: f"L{s[0]}D{1 + s[1]}_H{s[2]}_T{s[3]}_B{s[4]}_d{s[5]}")
def test_batched_recurrence_row_groups(oracle, s):
    L, bidir, H, T, B, density = s
    w = wl.Workload("rows", L, bidir, 40, H, T, B, "bf16", 0.04 if H > 300 else 0.1, density=density, seed=H + B)
    weights, x = wl.make(w)
    h0, c0 = wl.make_states(w)
    ref = oracle.forward(weights, x, h0, c0, layers=L, bidir=bidir, hidden=H)
    mode = "csr" if density < 1 else "dense"
    got = run_gpu(w, csr_weights(oracle, weights) if density < 1 else weights, x, h0, c0, exec_mode=mode)
    assert_close(got, ref, "bf16", f"rows/{mode}")


# one row group and several, two accumulators and one, N padded to a multiple of 16, two passes, without pairs
@pytest.mark.parametrize("s", [(False, 600, 2, 16, ""), (True, 300, 3, 5, ""), (False, 1500, 2, 30, ""), (False, 390, 3, 40, ""), (False, 700, 2, 64, ""),
                               (False, 1500, 2, 100, ""), (False, 200, 3, 21, "tc1"), (True, 150, 2, 48, "tc1")],
                         ids=lambda s: f"D{1 + s[0]}_H{s[1]}_T{s[2]}_B{s[3]}{s[4]}")
def test_pruned_batches_multiply_all_bits_of_h(oracle, s, monkeypatch):
    """With x = 0 only the recurrent products count.  A sum of n products of fp32 h and bf16 weights is off by at most n 2^-24 of
    its size, a gate by 2^-21 (the fast exponential) and less than a quarter of the sum's error, two steps of both: below 5e-7
    here.  h rounded to sixteen bits reaches 8e-7 and more at these shapes."""
    import numpy as np
    bidir, H, T, B, env = s
    monkeypatch.setenv("LSTM_B200_RECUR", env)
    w = wl.Workload("bits", 1, bidir, 24, H, T, B, "bf16", 1 / (0.1 * H) ** 0.5, density=0.1, seed=H + B)
    weights, x = wl.make(w)
    h0, c0 = wl.make_states(w)
    ref = oracle.forward(weights, np.zeros_like(x), h0, c0, layers=1, bidir=bidir, hidden=H)
    got = run_gpu(w, csr_weights(oracle, weights), np.zeros_like(x), h0, c0, exec_mode="csr")
    for name, g, r in zip(("y", "hT", "cT"), got, ref):
        assert np.abs(g - r).max() <= 5e-7, name
