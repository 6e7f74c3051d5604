"""Which recurrent kernel serves which call, as the library reports it after the call (needs a B200)."""
import pytest

pytestmark = pytest.mark.gpu


def forward(kind, dtype, bidir, L, H, T, B, density=1.0, max_B=None):
    """One call on fresh weights; the handle's report after it."""
    import torch
    import paper_1901_10997_b200 as pkg
    D, n = 2 if bidir else 1, 24
    g = torch.Generator(device="cuda").manual_seed(H + B)
    ws = []
    for layer in range(L):
        for _ in range(D):
            k = n if layer == 0 else D * H
            if kind == "hlstm":
                ws.append({"ux": torch.randn(4 * 64, k, generator=g, device="cuda"), "uh": torch.randn(4 * 64, H, generator=g, device="cuda"),
                           "w": torch.randn(4 * H, 64, generator=g, device="cuda")})
            else:
                w = {"wx": torch.randn(4 * H, k, generator=g, device="cuda"), "wh": torch.randn(4 * H, H, generator=g, device="cuda")}
                if density < 1:
                    w["mask_x"] = (torch.rand(4 * H, k, generator=g, device="cuda") < density).to(torch.uint8)
                    w["mask_h"] = (torch.rand(4 * H, H, generator=g, device="cuda") < density).to(torch.uint8)
                ws.append(w)
    shape = dict(layers=L, in_dim=n, hidden=H, bidir=bidir, dtype=dtype, max_T=T, max_B=max_B or B)
    m = pkg.HLSTM(ws, gate_hidden=64, **shape) if kind == "hlstm" else pkg.LSTM(ws, exec_mode="csr" if density < 1 else "dense", **shape)
    try:
        assert m.info()["kernel"] == pkg.LSTM_RAN_NONE
        m.forward(torch.randn(T, B, n, generator=g, device="cuda"))
        m.check()
        return m.info()
    finally:
        m.close()


# (kind, dtype, bidir, layers, H, T, B, density) -> kernel, threads
CASES = [
    (("lstm", "fp32", False, 1, 200, 3, 20, 1.0), "F32", 512),
    (("lstm", "fp32", False, 1, 400, 3, 2, 1.0), "SHARED", None),
    (("lstm", "bf16", False, 1, 300, 3, 1, 1.0), "REGISTERS", 256),
    (("lstm", "bf16", False, 1, 1300, 3, 1, 1.0), "ONE", 512),
    (("lstm", "bf16", False, 2, 300, 3, 1, 1.0), "WAVE", 512),
    (("lstm", "bf16", False, 2, 300, 3, 9, 1.0), "BATCHED", 512),
    (("lstm", "bf16", False, 1, 1300, 3, 5, 1.0), "BATCHED", 512),
    (("lstm", "bf16", False, 1, 600, 3, 16, 0.1), "BATCHED", 512),
    (("lstm", "bf16", False, 1, 600, 3, 1, 0.1), "SPARSE", 512),
    (("lstm", "bf16", False, 2, 300, 1, 8, 1.0), "STEP", 256),
    (("hlstm", "bf16", False, 1, 300, 3, 9, 1.0), "HLSTM_TILES", 512),
    (("hlstm", "bf16", False, 1, 300, 3, 2, 1.0), "HLSTM_TILES", 512),
    # two to four rows of stacks that fit the wavefront kernel, and just beyond where it is the faster one
    (("lstm", "bf16", False, 2, 200, 40, 4, 1.0), "WAVE", 512),
    (("lstm", "bf16", False, 2, 300, 40, 3, 1.0), "WAVE", 512),
    (("lstm", "bf16", False, 2, 300, 45, 3, 1.0), "BATCHED", 512),
    (("lstm", "bf16", False, 2, 300, 30, 4, 1.0), "BATCHED", 512),
    (("lstm", "bf16", False, 2, 700, 24, 2, 1.0), "WAVE", 512),
    (("lstm", "bf16", False, 2, 700, 25, 2, 1.0), "BATCHED", 512),
    (("lstm", "bf16", False, 3, 400, 40, 4, 1.0), "WAVE", 512),
    (("lstm", "bf16", False, 4, 300, 40, 4, 1.0, 9), "WAVE", 512),
    # a few rows of a pruned handle for a few steps
    (("lstm", "bf16", False, 2, 600, 1, 4, 0.1), "SPARSE", 512),
    (("lstm", "bf16", True, 1, 600, 4, 2, 0.1, 16), "SPARSE", 512),
    (("lstm", "bf16", False, 2, 600, 3, 3, 0.1), "BATCHED", 512),
    (("lstm", "bf16", False, 2, 600, 1, 5, 0.1), "BATCHED", 512),
    # wide directions in turn: short calls, and widths that would leave a quarter of the SMs idle
    (("lstm", "bf16", True, 1, 1500, 19, 1, 1.0), "REGISTERS", 512),
    (("lstm", "bf16", True, 1, 1500, 20, 1, 1.0), "ONE", 512),
    (("lstm", "bf16", True, 1, 1300, 41, 1, 1.0), "REGISTERS", 512),
    (("lstm", "bf16", True, 1, 1100, 3, 1, 1.0), "ONE", 512),
    # one sequence, on a handle made for one and on one made for several
    (("hlstm", "bf16", False, 1, 300, 3, 1, 1.0), "HLSTM_ROWS", None),
    (("hlstm", "bf16", True, 1, 300, 3, 1, 1.0, 20), "HLSTM_ROWS", None),
]


@pytest.mark.parametrize("case,kernel,threads", CASES, ids=lambda v: "-".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_kernel_of_a_call(case, kernel, threads):
    import paper_1901_10997_b200 as pkg
    info = forward(*case)
    assert pkg.RECUR_KERNELS[info["kernel"]] == pkg.RECUR_KERNELS[getattr(pkg, "LSTM_RAN_" + kernel)]
    assert info["kernel_ctas"] >= 1 and (threads is None or info["kernel_threads"] == threads)
    assert info["kernel_smem_bytes"] <= 227 * 1024


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("ctas", [20, 61, 100])
def test_stacks_on_fewer_ctas(oracle, dtype, ctas, monkeypatch):
    """The limit on the CTAs of a direction holds for the kernels that run the layers of a stack side by side too."""
    import torch
    import lstm_workloads as wl
    import paper_1901_10997_b200 as pkg
    from gpu_util import assert_close
    monkeypatch.setenv("LSTM_B200_CTAS", str(ctas))
    w = wl.Workload("ctas", 2, False, 40, 200, 9, 10, dtype, 0.1, seed=ctas)
    weights, x = wl.make(w)
    m = pkg.LSTM(weights, layers=2, in_dim=40, hidden=200, dtype=dtype, max_T=9, max_B=10)
    try:
        got = m.forward(torch.from_numpy(x).cuda())
        m.check()
        assert 1 <= m.info()["kernel_ctas"] <= ctas
        assert_close([t.cpu().numpy() for t in got], oracle.forward(weights, x, layers=2, bidir=False, hidden=200), dtype, "fewer CTAs")
    finally:
        m.close()


@pytest.mark.parametrize("value,side_by_side", [(None, True), ("", True), ("0", False), ("1", False)])
@pytest.mark.parametrize("dtype,launches", [("bf16", (3, 5)), ("fp32", (1, 4))])
def test_switch_that_keeps_the_layers_of_a_stack_apart(dtype, launches, value, side_by_side, monkeypatch):
    if value is None:
        monkeypatch.delenv("LSTM_B200_WAVE", raising=False)
    else:
        monkeypatch.setenv("LSTM_B200_WAVE", value)
    monkeypatch.setenv("LSTM_B200_RECUR", "")              # an empty switch is an unset one
    info = forward("lstm", dtype, False, 2, 200, 6, 9)
    assert info["launches_per_forward"] == launches[0 if side_by_side else 1]


# (dtype, layers, H, T, B) -> kernel, layers of its last launch
@pytest.mark.parametrize("dtype,L,H,T,B,kernel,layers", [("bf16", 2, 200, 6, 9, "BATCHED", 2), ("bf16", 3, 200, 6, 9, "BATCHED", 1), ("bf16", 3, 200, 6, 1, "WAVE", 3),
                                                         ("fp32", 3, 100, 6, 9, "F32", 3), ("fp32", 1, 100, 6, 9, "F32", 1), ("bf16", 2, 200, 1, 3, "STEP", 1)])
def test_layers_of_a_launch(dtype, L, H, T, B, kernel, layers):
    import paper_1901_10997_b200 as pkg
    info = forward("lstm", dtype, False, L, H, T, B)
    assert (info["kernel"], info["kernel_layers"]) == (getattr(pkg, "LSTM_RAN_" + kernel), layers)
