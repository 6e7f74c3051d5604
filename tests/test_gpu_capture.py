"""Calls recorded into a CUDA graph beside ordinary calls on the same handle: the kernels whose exchange words carry a phase bit
(batched, one wide sequence, narrow fp32, H-LSTM tiles) have words of their own for recorded launches, the others' stamped words
are cleared by the graph; single timesteps (needs a B200)."""
import pytest

import lstm_workloads as wl
from gpu_util import csr_weights

pytestmark = pytest.mark.gpu

# (kind, dtype, H, T, B): several steps and a single one of each kernel; pairs and passes of the batched one
CASES = [("lstm", "bf16", 300, 6, 3), ("lstm", "bf16", 200, 4, 70), ("lstm", "bf16", 300, 1, 16), ("lstm", "bf16", 1201, 6, 1), ("lstm", "fp32", 100, 6, 3),
         ("lstm", "fp32", 100, 1, 3), ("hlstm", "bf16", 150, 6, 3), ("hlstm", "bf16", 150, 1, 17), ("lstm", "bf16", 300, 1, 4),
         ("csr", "bf16", 600, 6, 16), ("csr", "bf16", 300, 6, 3),
         # stamped words: weights in registers, wavefront (two layers), lists, shared memory, H-LSTM rows
         ("lstm", "bf16", 300, 6, 1), ("wave", "bf16", 300, 6, 3), ("csr", "bf16", 300, 6, 1), ("csr", "bf16", 300, 2, 3), ("lstm", "fp32", 400, 6, 2),
         ("hlstm", "bf16", 150, 6, 1)]


@pytest.mark.parametrize("c", CASES, ids=lambda c: f"{c[0]}_{c[1]}_H{c[2]}_T{c[3]}_B{c[4]}")
def test_recorded_calls_beside_ordinary_ones(oracle, c):
    import torch
    import paper_1901_10997_b200 as pkg
    kind, dtype, H, T, B = c
    L = 2 if kind == "wave" else 1
    w = wl.Workload("capture", L, False, 40, H, 7, B, dtype, 0.05, density=0.3 if kind == "csr" else 1.0, seed=H + B)
    if kind == "hlstm":
        weights, x = wl.make_hlstm(w, 64)
        m = pkg.HLSTM(weights, layers=1, in_dim=40, hidden=H, gate_hidden=64, dtype=dtype, max_T=7, max_B=B)
    else:
        weights, x = wl.make(w)
        if kind == "csr":
            weights = csr_weights(oracle, weights)
        m = pkg.LSTM(weights, layers=L, in_dim=40, hidden=H, dtype=dtype, exec_mode="csr" if kind == "csr" else "dense", max_T=7, max_B=B)
    try:
        x = torch.from_numpy(x).cuda()
        xg = x[:T].flip(0).contiguous()
        expect = [[t.clone() for t in m.forward(xx)] for xx in (x, xg)]
        out = tuple(torch.empty_like(t) for t in expect[1])
        m.check()

        def ordinary(what):
            got = m.forward(x)
            m.check()
            assert all(torch.equal(a, b) for a, b in zip(got, expect[0])), what

        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            m.forward(xg, out=out)
        ordinary("after recording")
        for i in range(3):
            for _ in range(i + 1):
                for t in out:
                    t.zero_()
                graph.replay()
                m.check()
                torch.cuda.synchronize()
                assert all(torch.equal(a, b) for a, b in zip(out, expect[1])), f"replay {i}"
            ordinary(f"after replay {i}")
        ordinary("again")
        del graph
    finally:
        m.close()
