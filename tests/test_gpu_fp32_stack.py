"""fp32 stacks whose layers run in one launch: edges of the tiles (units per CTA, row tiles, groups of four columns), widths of the
input that are staged by 16 and by 4 bytes, the calls it hands to the other kernels, a NaN, a recorded call and a wait that runs
out, against the oracle (needs a B200)."""
import numpy as np
import pytest

import lstm_workloads as wl
from gpu_util import assert_close, run_gpu

pytestmark = pytest.mark.gpu

# (layers, in_dim, H, T, B): two and four units per CTA (148 columns are the widest with two), one to four row tiles; the last
# three run layer by layer: too wide an input, too many rows, too many steps
SHAPES = [(2, 1, 1, 3, 1), (2, 3, 2, 5, 8), (2, 64, 64, 1, 9), (2, 147, 148, 3, 16), (2, 66, 149, 4, 17), (2, 296, 296, 3, 32), (2, 295, 293, 2, 25),
          (3, 40, 98, 5, 3), (3, 21, 196, 3, 24), (4, 16, 148, 4, 20), (2, 297, 60, 3, 4), (2, 24, 60, 3, 33), (2, 5, 9, 257, 2)]


def make(s, seed=0):
    L, in_dim, H, T, B = s
    w = wl.Workload("f32stack", L, False, in_dim, H, T, B, "fp32", min(0.3, 2 / (H + in_dim) ** 0.5), seed=H + B + seed)
    return (w, *wl.make(w), *wl.make_states(w))


@pytest.mark.parametrize("s", SHAPES, ids=lambda s: "L{}_in{}_H{}_T{}_B{}".format(*s))
def test_fp32_narrow_stack(oracle, s):
    w, weights, x, h0, c0 = make(s)
    ref = oracle.forward(weights, x, h0, c0, layers=w.layers, bidir=False, hidden=w.hidden)
    assert_close(run_gpu(w, weights, x, h0, c0), ref, "fp32", "fp32 stack")
    if 1 < w.T < 100:
        assert_close(run_gpu(w, weights, x, h0, c0, chunks=[1, w.T - 1]), ref, "fp32", "fp32 stack, chunked")


def test_fp32_narrow_stack_nan_in_one_unit(oracle):
    w, weights, x, h0, c0 = make((2, 24, 200, 5, 20), 3)
    c0[0, 11, 66] = np.nan
    ref = oracle.forward(weights, x, h0, c0, layers=2, bidir=False, hidden=200)
    for name, got, want in zip(("y", "hT", "cT"), run_gpu(w, weights, x, h0, c0), ref):
        assert np.array_equal(np.isnan(got), np.isnan(want)), name
        ok = ~np.isnan(want)
        assert np.abs(got - want)[ok].max() <= wl.TOLERANCE["fp32"], name


def test_fp32_narrow_stack_recorded_timed_out_and_shorter_calls(oracle):
    """Calls of different lengths and rows on one handle, a recorded one replayed between them, and one whose words are withheld:
    every call meets cleared words, whatever the calls before it wrote."""
    import torch
    import paper_1901_10997_b200 as pkg
    w, weights, x, _, _ = make((2, 40, 150, 9, 20), 5)
    m = pkg.LSTM(weights, layers=2, in_dim=40, hidden=150, dtype="fp32", max_T=9, max_B=20)
    try:
        xd = torch.from_numpy(x).cuda()
        xs = [xd[:T, :B].contiguous() for T, B in ((9, 20), (2, 3), (1, 20), (9, 20), (5, 9))]
        refs = [oracle.forward(weights, v.cpu().numpy(), layers=2, bidir=False, hidden=150) for v in xs]

        def ordinary():
            for v, ref in zip(xs, refs):
                got = m.forward(v)
                m.check()
                assert m.info()["launches_per_forward"] == 1
                assert_close([t.cpu().numpy() for t in got], ref, "fp32", "fp32 stack, mixed calls")

        ordinary()
        out = tuple(torch.empty_like(t) for t in m.forward(xs[4]))
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            m.forward(xs[4], out=out)
        for _ in range(3):
            for t in out:
                t.zero_()
            graph.replay()
            m.check()
            assert_close([t.cpu().numpy() for t in out], refs[4], "fp32", "fp32 stack, replayed")
            ordinary()
        for cta in (5, 40):                         # a CTA of each layer
            m.selftest_timeout(cta, 2_000_000)
            m.forward(xd)
            assert m.status() == pkg.LSTM_ERR_TIMEOUT
            m.selftest_timeout(-1)
            ordinary()
        del graph
    finally:
        m.close()


def test_fp32_narrow_stack_beside_a_smaller_one(oracle):
    """A handle that needs less shared memory, made later, takes nothing from the one made before it."""
    import torch
    import paper_1901_10997_b200 as pkg
    models = []
    try:
        for s in ((2, 256, 256, 3, 32), (2, 160, 160, 3, 32)):
            w, weights, x, _, _ = make(s)
            models.append((pkg.LSTM(weights, layers=2, in_dim=s[1], hidden=s[2], dtype="fp32", max_T=3, max_B=32), torch.from_numpy(x).cuda(),
                           oracle.forward(weights, x, layers=2, bidir=False, hidden=s[2])))
        for m, x, ref in models + models[:1]:
            got = m.forward(x)
            m.check()
            assert_close([t.cpu().numpy() for t in got], ref, "fp32", "fp32 stack, two handles")
    finally:
        for m, _, _ in models:
            m.close()
