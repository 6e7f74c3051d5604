"""The H-LSTM tile kernel at the edges of its tiles and modes, against the oracle (needs a B200)."""
import pytest

import lstm_workloads as wl
from gpu_util import assert_close
from test_gpu_hlstm import run

pytestmark = pytest.mark.gpu

# (layers, bidir, in_dim, H, Hh, T, B, scale): four, eight, nine, sixteen rows and more than one launch; several hidden tiles
# per CTA with five and six column tiles per warp (row groups in turn), exact and ragged tiles, a step count of one
SHAPES = [
    (1, False, 20, 64, 48, 3, 4, 0.3),
    (2, True, 24, 130, 100, 4, 9, 0.2),
    (1, True, 40, 800, 800, 3, 16, 0.05),
    (1, False, 32, 1500, 1500, 3, 13, 0.03),
    (1, False, 16, 1040, 320, 1, 8, 0.05),
    (2, False, 24, 96, 16, 5, 37, 0.2),
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"L{s[0]}D{1 + s[1]}_H{s[3]}_Hh{s[4]}_T{s[5]}_B{s[6]}")
@pytest.mark.parametrize("kernel", ["", "mma"])
def test_tile_kernel_and_row_kernel_match_the_oracle(oracle, shape, kernel, monkeypatch):
    L, bidir, in_dim, H, Hh, T, B, scale = shape
    if kernel and B > 16:
        pytest.skip("the row kernel at this batch adds nothing")
    monkeypatch.setenv("LSTM_B200_RECUR", kernel)
    w = wl.Workload("hlstm_tiles", L, bidir, in_dim, H, T, B, "bf16", scale, seed=sum(shape[2:7]))
    weights, x = wl.make_hlstm(w, Hh)
    h0, c0 = wl.make_states(w)
    ref = oracle.forward_hlstm(weights, x, h0, c0, layers=L, bidir=bidir, hidden=H, gate_hidden=Hh)
    assert_close(run(w, Hh, weights, x, h0, c0), ref, "bf16", f"hlstm tiles/{kernel or 'default'}")


# (layers, bidir, in_dim, H, Hh, T, scale): five column tiles per warp, one to three hidden tiles per CTA, ragged tiles on both sides
FIVE = [(1, False, 24, 1200, 320, 5, 0.03), (1, False, 16, 1025, 600, 5, 0.03), (1, False, 16, 1271, 1300, 5, 0.03), (2, True, 16, 1100, 610, 5, 0.03)]


@pytest.mark.parametrize("B", [3, 8, 16])
@pytest.mark.parametrize("shape", FIVE, ids=lambda s: f"L{s[0]}D{1 + s[1]}_H{s[3]}_Hh{s[4]}")
def test_tile_kernel_with_five_column_tiles(oracle, shape, B):
    L, bidir, in_dim, H, Hh, T, scale = shape
    w = wl.Workload("hlstm_tiles", L, bidir, in_dim, H, T, B, "bf16", scale, seed=H + Hh + B)
    weights, x = wl.make_hlstm(w, Hh)
    h0, c0 = wl.make_states(w)
    ref = oracle.forward_hlstm(weights, x, h0, c0, layers=L, bidir=bidir, hidden=H, gate_hidden=Hh)
    assert_close(run(w, Hh, weights, x, h0, c0), ref, "bf16", "hlstm, five column tiles")
