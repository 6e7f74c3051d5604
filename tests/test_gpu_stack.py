"""Two layers of a batch in one launch: edges of the partition (units per pair, the second block of accumulator rows, halves of K),
of the row groups, of the chunks and of the rule that takes calls there, dense and pruned, against the oracle (needs a B200)."""
import numpy as np
import pytest

import lstm_workloads as wl
from gpu_util import GUARD, assert_close, csr_weights, run_gpu

pytestmark = pytest.mark.gpu

# (in_dim, H, T, B, density)
SHAPES = [(5, 65, 4, 5, 1.0), (40, 128, 5, 8, 1.0), (33, 129, 9, 9, 1.0), (64, 301, 47, 3, 1.0), (70, 517, 7, 24, 1.0), (24, 600, 11, 32, 1.0), (20, 600, 6, 33, 1.0),
          (30, 1056, 5, 2, 1.0), (30, 1057, 16, 2, 1.0), (16, 1280, 17, 9, 1.0), (24, 1281, 16, 17, 1.0), (40, 1500, 18, 20, 1.0), (16, 1500, 16, 25, 1.0), (16, 1536, 16, 3, 1.0),
          (64, 300, 4, 7, 0.3), (48, 700, 9, 16, 0.1), (32, 1300, 16, 9, 0.1)]


def make(s, seed=0):
    in_dim, H, T, B, density = s
    w = wl.Workload("stack", 2, False, in_dim, H, T, B, "bf16", min(0.3, 1.5 / (H * density) ** 0.5), density=density, seed=H + B + seed)
    return (w, *wl.make(w), *wl.make_states(w))


@pytest.mark.parametrize("s", SHAPES, ids=lambda s: "in{}_H{}_T{}_B{}_p{}".format(*s))
def test_small_shapes_of_stacks(oracle, s):
    w, weights, x, h0, c0 = make(s)
    ref = oracle.forward(weights, x, h0, c0, layers=2, bidir=False, hidden=w.hidden)
    mode, ws = ("dense", weights) if w.density == 1 else ("csr", csr_weights(oracle, weights))
    assert_close(run_gpu(w, ws, x, h0, c0, exec_mode=mode), ref, "bf16", "stack")
    if w.T == 9:
        assert_close(run_gpu(w, ws, x, h0, c0, exec_mode=mode, chunks=[4, 5]), ref, "bf16", "stack, chunked")


# H, T, B -> launches: beside each other three, one after the other five
@pytest.mark.parametrize("H,T,B,launches", [(300, 4, 9, 3), (300, 3, 9, 5), (300, 4, 32, 3), (300, 4, 33, 5), (1200, 16, 9, 3), (1200, 15, 9, 5), (1500, 16, 24, 3), (1500, 16, 25, 5),
                                              (1320, 16, 20, 3), (1320, 16, 21, 5), (1584, 16, 12, 3), (1584, 16, 13, 5), (1056, 4, 32, 3)])
def test_calls_that_run_two_layers_at_once(H, T, B, launches):
    import torch
    import paper_1901_10997_b200 as pkg
    g = torch.Generator(device="cuda").manual_seed(H)
    ws = [{"wx": torch.randn(4 * H, n, generator=g, device="cuda"), "wh": torch.randn(4 * H, H, generator=g, device="cuda")} for n in (16, H)]
    m = pkg.LSTM(ws, layers=2, in_dim=16, hidden=H, dtype="bf16", max_T=16, max_B=B)
    try:
        m.forward(torch.randn(T, B, 16, generator=g, device="cuda"))
        m.check()
        assert m.info()["launches_per_forward"] == launches
    finally:
        m.close()


def test_small_shapes_of_stacks_nan_in_one_unit(oracle):
    w, weights, x, h0, c0 = make((24, 300, 6, 13, 1.0), 3)
    c0[0, 11, 66] = np.nan
    ref = oracle.forward(weights, x, h0, c0, layers=2, bidir=False, hidden=300)
    for name, got, want in zip(("y", "hT", "cT"), run_gpu(w, weights, x, h0, c0), ref):
        assert np.array_equal(np.isnan(got), np.isnan(want)), name
        ok = ~np.isnan(want)
        assert np.abs(got - want)[ok].max() <= wl.TOLERANCE["bf16"], name


@pytest.mark.parametrize("density", [1.0, 0.2])
def test_stacks_recorded_timed_out_and_of_different_lengths(oracle, density):
    """Calls of different lengths and rows on one handle, a recorded one replayed between them, and ones whose words are withheld:
    every call meets cleared words and counts, whatever the calls before it wrote."""
    import torch
    import paper_1901_10997_b200 as pkg
    w, weights, x, _, _ = make((40, 300, 19, 15, density), 5)
    ws, mode = (weights, "dense") if density == 1 else (csr_weights(oracle, weights), "csr")
    m = pkg.LSTM(ws, layers=2, in_dim=40, hidden=300, dtype="bf16", exec_mode=mode, max_T=19, max_B=15)
    try:
        xd = torch.from_numpy(x).cuda()
        xs = [xd[:T, :B].contiguous() for T, B in ((19, 15), (4, 9), (2, 15), (19, 15), (7, 5), (19, 8))]
        refs = [oracle.forward(weights, v.cpu().numpy(), layers=2, bidir=False, hidden=300) for v in xs]

        def ordinary():
            for v, ref in zip(xs, refs):
                got = m.forward(v)
                m.check()
                assert_close([t.cpu().numpy() for t in got], ref, "bf16", "stack, mixed calls")

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
            assert_close([t.cpu().numpy() for t in out], refs[4], "bf16", "stack, replayed")
            ordinary()
        for cta in (5, 60, 0):                      # of the lower and of the upper layer
            m.selftest_timeout(cta, 2_000_000)
            m.forward(xd)
            assert m.status() == pkg.LSTM_ERR_TIMEOUT
            m.selftest_timeout(-1)
            ordinary()
        del graph
    finally:
        m.close()


def test_stack_that_gives_up_while_the_projection_runs(oracle):
    """The upper layer's wait ends long before the lower layer does: the CTAs that project find the status between two chunks, with
    products of theirs under way, at another point of the chunk for every limit."""
    import torch
    import paper_1901_10997_b200 as pkg
    w, weights, x, _, _ = make((40, 300, 256, 15, 1.0), 7)
    ref = oracle.forward(weights, x, layers=2, bidir=False, hidden=300)
    m = pkg.LSTM(weights, layers=2, in_dim=40, hidden=300, dtype="bf16", max_T=256, max_B=15)
    try:
        xd = torch.from_numpy(x).cuda()
        for limit in range(200_000, 300_000, 5_000):         # about 0.1 ms; the call takes 0.6
            m.selftest_timeout(60, limit)
            m.forward(xd)
            assert m.status() == pkg.LSTM_ERR_TIMEOUT
        m.selftest_timeout(-1)
        got = m.forward(xd)
        m.check()
        assert_close([t.cpu().numpy() for t in got], ref, "bf16", "stack, after the waits that gave up")
    finally:
        m.close()


# (in_dim, H, B, density): the lower layer's projection in several planes for calls of up to 128 rows, in one beyond them
@pytest.mark.parametrize("in_dim,H,B,density", [(517, 300, 8, 1.0), (301, 517, 3, 1.0), (1500, 1300, 8, 1.0), (700, 600, 20, 1.0), (600, 400, 16, 0.2)])
def test_stack_behind_a_projection_in_several_planes(oracle, in_dim, H, B, density):
    import torch
    import paper_1901_10997_b200 as pkg
    T = 128 // B
    w, weights, x, _, _ = make((in_dim, H, T + 1, B, density), 9)
    ws, mode = (weights, "dense") if density == 1 else (csr_weights(oracle, weights), "csr")
    ref = oracle.forward(weights, x, layers=2, bidir=False, hidden=H)
    m = pkg.LSTM(ws, layers=2, in_dim=in_dim, hidden=H, dtype="bf16", exec_mode=mode, max_T=T + 1, max_B=B)
    try:
        xd, got = torch.from_numpy(x).cuda(), {}
        for t in (T, T + 1):
            y, hT, cT = m.forward(xd[:t].contiguous())
            m.check()
            info = m.info()
            assert info["launches_per_forward"] == 3
            got[info["proj_splits"] > 1] = y.cpu().numpy()
            if t > T:
                assert_close([v.cpu().numpy() for v in (y, hT, cT)], ref, "bf16", "stack behind one plane")
        assert set(got) == {True, False}
        # the same products in another order: each side within the guard of the oracle, so within twice that of the other
        assert np.abs(got[True] - got[False][:T]).max() <= 2 * GUARD["bf16"] * np.abs(ref[0]).max()
        assert_close([got[True]], [ref[0][:T]], "bf16", "stack behind several planes")
    finally:
        m.close()


def test_small_shapes_of_stacks_nan_in_one_unit_of_the_second_block(oracle):
    """Two blocks of accumulator rows (1300 units): a NaN in one unit of either block reaches what it has to and nothing else."""
    for unit in (3, 36, 1299):                  # of the first pair's first and second block, and of the last pair
        w, weights, x, h0, c0 = make((24, 1300, 16, 5, 1.0), 3)
        c0[0, 2, unit] = np.nan
        ref = oracle.forward(weights, x, h0, c0, layers=2, bidir=False, hidden=1300)
        for name, got, want in zip(("y", "hT", "cT"), run_gpu(w, weights, x, h0, c0), ref):
            assert np.array_equal(np.isnan(got), np.isnan(want)), (name, unit)
            ok = ~np.isnan(want)
            assert np.abs(got - want)[ok].max() <= wl.TOLERANCE["bf16"], (name, unit)


def test_stack_with_two_blocks_whose_words_or_projection_are_withheld(oracle):
    import torch
    import paper_1901_10997_b200 as pkg
    w, weights, x, _, _ = make((24, 1300, 16, 5, 1.0), 4)
    ref = oracle.forward(weights, x, layers=2, bidir=False, hidden=1300)
    m = pkg.LSTM(weights, layers=2, in_dim=24, hidden=1300, dtype="bf16", max_T=16, max_B=5)
    try:
        xd = torch.from_numpy(x).cuda()
        for cta in (1, 66, 132, 147):           # of the lower layer, of the upper one (33 pairs each), two that project
            m.selftest_timeout(cta, 2_000_000)
            m.forward(xd)
            assert m.status() == pkg.LSTM_ERR_TIMEOUT
            m.selftest_timeout(-1)
            got = m.forward(xd)
            m.check()
            assert_close([t.cpu().numpy() for t in got], ref, "bf16", "stack, after a withheld CTA")
    finally:
        m.close()


# narrow layers: (in_dim, H, T, B, density) at the edges of pairs of 24 units and of the projecting CTAs' blocks of rows
@pytest.mark.parametrize("s", [(30, 65, 9, 17, 1.0), (24, 96, 5, 32, 1.0), (300, 97, 8, 8, 1.0), (20, 256, 7, 25, 1.0), (200, 295, 6, 20, 1.0), (40, 296, 13, 9, 1.0), (33, 296, 9, 16, 0.2)],
                         ids=lambda s: "in{}_H{}_T{}_B{}_p{}".format(*s))
def test_small_shapes_of_stacks_that_leave_sms_to_others(oracle, s):
    """Two layers of up to 296 units take less than half of the SMs, so that the calls of two handles run at once."""
    import torch
    import paper_1901_10997_b200 as pkg
    w, weights, x, h0, c0 = make(s)
    ref = oracle.forward(weights, x, h0, c0, layers=2, bidir=False, hidden=w.hidden)
    mode, ws = ("dense", weights) if w.density == 1 else ("csr", csr_weights(oracle, weights))
    xd, hd, cd = (torch.from_numpy(v).cuda() for v in (x, h0, c0))
    models, streams = [], [torch.cuda.Stream() for _ in range(3)]
    try:
        for _ in streams:
            models.append(pkg.LSTM(ws, layers=2, in_dim=w.in_dim, hidden=w.hidden, dtype="bf16", exec_mode=mode, max_T=w.T, max_B=w.B))
        outs = [(torch.empty(w.T, w.B, w.hidden, device="cuda"), torch.empty(2, w.B, w.hidden, device="cuda"), torch.empty(2, w.B, w.hidden, device="cuda")) for _ in streams]
        torch.cuda.synchronize()
        for _ in range(20):
            for m, st, out in zip(models, streams, outs):
                m.forward(xd, hd, cd, out=out, stream=st.cuda_stream)
        for m, out in zip(models, outs):
            m.check()
            assert_close([t.cpu().numpy() for t in out], ref, "bf16", "narrow stack")
            info = m.info()
            assert info["launches_per_forward"] == 3 and 2 * info["kernel_ctas"] <= info["sm_count"]
    finally:
        for m in models:
            m.close()


@pytest.mark.parametrize("H,max_T,holds_more", [(1500, 15, False), (1500, 16, True), (1050, 3, False), (1050, 4, True)])
def test_memory_of_handles_whose_calls_are_too_short(H, max_T, holds_more, monkeypatch):
    """Rows, words and the second G for two layers side by side only where a call of the handle can use them."""
    import torch
    import paper_1901_10997_b200 as pkg
    g = torch.Generator(device="cuda").manual_seed(H)
    ws = [{"wx": torch.randn(4 * H, n, generator=g, device="cuda"), "wh": torch.randn(4 * H, H, generator=g, device="cuda")} for n in (16, H)]

    def held():
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        m = pkg.LSTM(ws, layers=2, in_dim=16, hidden=H, dtype="bf16", max_T=max_T, max_B=20)
        used = free - torch.cuda.mem_get_info()[0]
        m.close()
        return used

    held()                                          # (what the first handle of a process sets up)
    both = held()
    monkeypatch.setenv("LSTM_B200_WAVE", "0")
    assert (both - held() >= 2 * 4 * H * H * 2) == holds_more      # the rows of both layers' recurrent matrices, at least


def test_handle_without_room_for_two_layers_side_by_side(oracle):
    """Memory for everything but the second copy of the rows and the second G: the layers run one after the other."""
    import torch
    import paper_1901_10997_b200 as pkg
    w, weights, x, _, _ = make((16, 1200, 16, 5, 1.0), 8)
    ref = oracle.forward(weights, x, layers=2, bidir=False, hidden=1200)
    shape = dict(layers=2, in_dim=16, hidden=1200, dtype="bf16", max_T=409, max_B=20)      # a second G of 157 MB
    xd = torch.from_numpy(x).cuda()

    def run(m):
        got = m.forward(xd)
        m.check()
        assert_close([t.cpu().numpy() for t in got], ref, "bf16", "stack, little memory")
        return m.info()["launches_per_forward"]

    pkg.LSTM(weights, **shape).close()              # (what the first handle of a process sets up)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    m = pkg.LSTM(weights, **shape)
    needs = before - torch.cuda.mem_get_info()[0]
    try:
        assert run(m) == 3
    finally:
        m.close()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - needs + (100 << 20), dtype=torch.uint8, device="cuda")
    try:
        m = pkg.LSTM(weights, **shape)
        try:
            assert run(m) == 5
        finally:
            m.close()
    finally:
        del fill
        torch.cuda.empty_cache()
