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


@pytest.mark.parametrize("size", [1e-6, 1e-12, 1e-30])
def test_fp32_narrow_keeps_the_digits_of_small_values(oracle, size):
    """Gate pre-activations of this size: tanh z = z and logistic = 1/2 to all digits, every value keeps its fp32 precision."""
    import numpy as np
    w = wl.Workload("small", 1, False, 24, 100, 3, 12, "fp32", 0.1, seed=3)
    weights, x = wl.make(w)
    for q in weights:
        q["wx"], q["b"] = np.float32(q["wx"] * size), np.float32(q["b"] * size)
    ref = oracle.forward(weights, x, layers=1, bidir=False, hidden=100)
    assert_close(run_gpu(w, weights, x), ref, "fp32", f"small values {size}")


def test_fp32_projection_of_more_rows_than_a_grid_has_in_y():
    """T x B = 2 100 000 rows, more than 65535 tiles of 32; every row against the product in float64."""
    import torch
    import paper_1901_10997_b200 as pkg
    T, K, H = 2_100_000, 3, 9
    g = torch.Generator(device="cuda").manual_seed(5)
    wx = torch.rand((4 * H, K), generator=g, device="cuda") - 0.5
    m = pkg.LSTM([{"wx": wx, "wh": torch.zeros((4 * H, H), device="cuda")}], layers=1, in_dim=K, hidden=H, dtype="fp32", max_T=T, max_B=1)
    try:
        x = torch.randn((T, 1, K), generator=g, device="cuda")
        got = m.input_projection(x).reshape(T, 4 * H)
        ref = x.reshape(T, K).double() @ wx.double().T
        assert float((got.double() - ref).abs().max()) <= 2.0 ** -24 * float(ref.abs().max())      # one rounding to fp32
    finally:
        m.close()
