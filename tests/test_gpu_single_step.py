"""Single timesteps (T = 1) on the streaming kernel against the oracle: each number of row tiles, every operand layout of
the batch rows, one and two directions, state given or not, and a chain of steps that carries the state (needs a B200)."""
import pytest

import lstm_workloads as wl
from gpu_util import assert_close, run_gpu

pytestmark = pytest.mark.gpu

# (layers, bidir, in_dim, H, B)
SHAPES = [(2, False, 33, 97, 1), (2, True, 40, 300, 4), (1, False, 515, 600, 2), (2, False, 1501, 1500, 8), (3, False, 64, 2000, 5), (1, True, 7, 1, 3)]


@pytest.mark.parametrize("s", SHAPES, ids=lambda s: f"L{s[0]}D{1 + s[1]}_in{s[2]}_H{s[3]}_B{s[4]}")
@pytest.mark.parametrize("state", [True, False])
def test_single_step(oracle, s, state):
    L, bidir, in_dim, H, B = s
    w = wl.Workload("step", L, bidir, in_dim, H, 1, B, "bf16", min(0.3, 2 / (H + in_dim) ** 0.5), seed=H)
    weights, x = wl.make(w)
    h0, c0 = wl.make_states(w) if state else (None, None)
    ref = oracle.forward(weights, x, h0, c0, layers=L, bidir=bidir, hidden=H)
    assert_close(run_gpu(w, weights, x, h0, c0, max_T=5), ref, "bf16", "single step")


def test_steps_in_a_row_carry_the_state(oracle):
    w = wl.Workload("steps", 2, False, 50, 700, 6, 3, "bf16", 0.05, seed=3)
    weights, x = wl.make(w)
    ref = oracle.forward(weights, x, layers=2, bidir=False, hidden=700)
    assert_close(run_gpu(w, weights, x, chunks=[1, 1, 2, 1, 1]), ref, "bf16", "steps in a row")
