"""The fp32 kernel for narrow layers at the edges of its tiles (units per CTA, tiles of eight batch rows, K ranges) and just
outside its range, against the oracle (needs a B200)."""
import pytest

import lstm_workloads as wl
from gpu_util import assert_close, run_gpu

pytestmark = pytest.mark.gpu

# (layers, bidir, in_dim, H, T, B)
SHAPES = [(2, False, 9, 1, 4, 8), (1, True, 30, 74, 5, 9), (2, False, 64, 149, 4, 1), (1, False, 33, 295, 4, 17), (1, False, 20, 296, 3, 32),
          (1, False, 20, 297, 3, 4), (1, True, 16, 148, 4, 24), (1, False, 24, 60, 3, 33)]


@pytest.mark.parametrize("s", SHAPES, ids=lambda s: f"L{s[0]}D{1 + s[1]}_H{s[3]}_T{s[4]}_B{s[5]}")
def test_fp32_narrow(oracle, s):
    L, bidir, in_dim, H, T, B = s
    w = wl.Workload("f32", L, bidir, in_dim, H, T, B, "fp32", min(0.3, 2 / (H + in_dim) ** 0.5), seed=H + B)
    weights, x = wl.make(w)
    h0, c0 = wl.make_states(w)
    ref = oracle.forward(weights, x, h0, c0, layers=L, bidir=bidir, hidden=H)
    assert_close(run_gpu(w, weights, x, h0, c0), ref, "fp32", "fp32 narrow")
    if not bidir:
        assert_close(run_gpu(w, weights, x, h0, c0, chunks=[1, T - 1]), ref, "fp32", "fp32 narrow, chunked")
