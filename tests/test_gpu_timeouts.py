"""The bounded waits of every recurrent kernel (needs a B200): one CTA withholds its words, the others' waits run out after a
millisecond, the call reports LSTM_ERR_TIMEOUT, and the next calls on the same handle are right again.  Nothing hangs."""
import pytest

import lstm_workloads as wl
from gpu_util import assert_close, csr_weights

pytestmark = pytest.mark.gpu

# kernel, (dtype, mode, layers, bidir, H, T, B); both forms of the projection for one sequence, both plans of the batched kernel
CASES = [("REGISTERS", ("bf16", "dense", 1, False, 300, 8, 1)), ("REGISTERS", ("bf16", "dense", 1, True, 300, 44, 1)),
         ("ONE", ("bf16", "dense", 1, False, 1201, 8, 1)), ("ONE", ("bf16", "dense", 1, True, 1100, 44, 1)),
         ("SPARSE", ("bf16", "csr", 1, False, 300, 8, 1)), ("SPARSE", ("bf16", "csr", 1, False, 600, 2, 3)),
         ("WAVE", ("bf16", "dense", 2, False, 300, 8, 1)), ("BATCHED", ("bf16", "dense", 1, False, 300, 8, 3)),
         ("BATCHED", ("bf16", "dense", 1, True, 600, 8, 20)), ("BATCHED", ("bf16", "csr", 1, False, 600, 8, 20)),
         ("F32", ("fp32", "dense", 1, False, 200, 8, 1)), ("F32", ("fp32", "dense", 1, True, 100, 8, 20)),
         ("SHARED", ("fp32", "dense", 1, False, 300, 8, 2)), ("HLSTM_ROWS", ("bf16", "hlstm", 1, False, 200, 6, 1)),
         ("HLSTM_TILES", ("bf16", "hlstm", 1, True, 200, 6, 5))]


@pytest.mark.parametrize("kernel,c", CASES, ids=lambda v: v if isinstance(v, str) else "{0}_{1}_L{2}D{3}_H{4}_T{5}_B{6}".format(*v[:3], 1 + v[3], *v[4:]))
def test_withheld_words_time_out_and_later_calls_are_right(oracle, kernel, c):
    import torch
    import paper_1901_10997_b200 as pkg
    dtype, mode, L, bidir, H, T, B = c
    w = wl.Workload("timeouts", L, bidir, 40, H, T, B, dtype, min(0.1, 1 / H ** 0.5), density=0.3 if mode == "csr" else 1.0, seed=H + B)
    shape = dict(layers=L, in_dim=40, hidden=H, bidir=bidir, dtype=dtype, max_T=T, max_B=B)
    if mode == "hlstm":
        weights, x = wl.make_hlstm(w, 160)
        ref = oracle.forward_hlstm(weights, x, layers=L, bidir=bidir, hidden=H, gate_hidden=160)
        m = pkg.HLSTM(weights, gate_hidden=160, **shape)
    else:
        weights, x = wl.make(w)
        ref = oracle.forward(weights, x, layers=L, bidir=bidir, hidden=H)
        m = pkg.LSTM(csr_weights(oracle, weights) if mode == "csr" else weights, exec_mode=mode, **shape)
    try:
        xd = torch.from_numpy(x).cuda()
        for cta in (5, 0):
            m.selftest_timeout(cta, 2_000_000)
            m.forward(xd)
            assert m.status() == pkg.LSTM_ERR_TIMEOUT
            assert m.info()["kernel"] == getattr(pkg, "LSTM_RAN_" + kernel)
            m.selftest_timeout(-1)
            for _ in range(3):                       # both sets of exchange words, and the first again
                got = m.forward(xd)
                m.check()
                assert_close([t.cpu().numpy() for t in got], ref, dtype, f"after the timeout/{kernel}")
    finally:
        m.close()
