"""The sequence kernel (a thread-block cluster per sequence) against the oracle where it can go wrong: slices and chunks
that are empty, ragged or exactly full, clusters of one to sixteen CTAs, no drafts, masked and bad rows, and draws that
all go to the evaluation in double."""
import numpy as np
import pytest
import torch

import bebop_gen as G
import oracle
import paper_2606_12370_b200 as P
from parity import TOL, check_properties, compare_verify, oracle_on, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(autouse=True)
def _sequence_kernel():
    P.bebop_debug_force_general_path(4)
    yield
    P.bebop_debug_set_draw_kappa(-1.0)
    P.bebop_debug_force_general_path(0)


def run(x, **kw):
    return P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], draft_len=x["draft_len"],
                          temperature=x["temperature"], temperature_all=x["temperature_all"], **kw)


# one vector; one chunk short of, exactly, one beyond 128 vectors; slices that leave the last CTA empty; sixteen CTAs
SHAPES = [("bf16", 5, 2, 8), ("bf16", 9, 1, 1016), ("bf16", 9, 1, 1024), ("f32", 9, 3, 516), ("bf16", 140, 3, 4101), ("f32", 3, 32, 2047),
          ("bf16", 2, 3, 151936), ("f32", 1, 2, 151937), ("bf16", 1, 2, 262144), ("bf16", 600, 1, 2049)]


@pytest.mark.parametrize("redraw", [False, True])
@pytest.mark.parametrize("dtype,B,K,V", SHAPES)
def test_verify(dtype, B, K, V, redraw):
    cfg = G.Config("seq", B, K, V, dtype, 2.0, V >= 16, 0.8, (0.6, 1.2), ragged=K > 1, seed=B + K)
    x = G.make_inputs(cfg, DEV, pad_ld=(-V) % 8)
    if K > 1:
        x["draft_len"] = torch.tensor([(i * 5) % (K + 1) for i in range(B)], dtype=torch.int32, device=DEV)
    if redraw:
        P.bebop_debug_set_draw_kappa(1e9)          # no fp32 draw clears its bound
    got = run(x)
    assert P.bebop_debug_last_kernel() == 3
    ref = oracle_on(x)
    check_properties(got, x)
    compare_verify(got, ref, dtype, context=str(cfg))
    tokens_only = run(x, want_tv=False, want_probs=False, want_status=False)
    assert tokens_only["tv"] is None
    assert torch.equal(tokens_only["accept_len"], got["accept_len"]) and torch.equal(tokens_only["out_tokens"], got["out_tokens"])


@pytest.mark.parametrize("dtype,B,K,V", SHAPES)
def test_tv_and_greedy(dtype, B, K, V):
    cfg = G.Config("seq", B, K, V, dtype, 2.0, V >= 16, 0.8, 1.0, seed=B + K)
    x = G.make_inputs(cfg, DEV, draft_mode="argmax", pad_ld=(-V) % 8)
    tgt, drf = x["target"][:, 0], x["draft"][:, K - 1]
    tau = torch.linspace(0.6, 1.2, B, device=DEV)
    tau[0] = -1.0 if B > 1 else 1.0
    got = P.bebop_tv(tgt, drf, temperature=tau)
    assert P.bebop_debug_last_kernel_name() == "k_seq"
    ref = oracle.tv(tgt.float().cpu().numpy(), drf.float().cpu().numpy(), temperature=to_np(tau))
    np.testing.assert_array_equal(to_np(got["row_status"]), ref["row_status"])
    assert np.abs(to_np(got["tv"]) - ref["tv"]).max() <= TOL[dtype]
    assert np.abs(to_np(got["s_aux"]) - ref["s_aux"]).max() <= TOL[dtype]
    x["target"][0, 0, V - 1] = float("nan")
    x["target"][B - 1, K, :] = float("-inf")
    g = P.bebop_greedy_verify(x["target"], x["draft_tokens"])
    assert P.bebop_debug_last_kernel_name() == "k_seq_greedy"
    r = oracle.greedy_verify(x["target"].float().cpu().numpy(), to_np(x["draft_tokens"]))
    for k in ("accept_len", "out_tokens", "row_status"):
        np.testing.assert_array_equal(to_np(g[k]), r[k], err_msg=k)


@pytest.mark.parametrize("V", [2048, 40000])
def test_status_and_masks(V):
    cfg = G.Config("st", 10, 2, V, "f32", 1.0, False, 0.5, 1.0, seed=4)
    x = G.make_inputs(cfg, DEV)
    x["target"][1, 0, 17] = float("nan")
    x["draft"][2, 1, :] = float("-inf")
    x["draft_tokens"][3, 1] = V
    x["temperature"] = torch.ones(10, device=DEV)
    x["temperature"][4] = 0.0
    x["target"][5, 1, V - 1] = float("inf")
    # 6: p == q with the drafted token masked in both (no residual mass at a reject); 7: NaN only in the bonus row
    x["draft"][6] = x["target"][6, :2]
    x["target"][6, 0, 9] = float("-inf"); x["draft"][6, 0, 9] = float("-inf")
    x["draft_tokens"][6, 0] = 9
    x["draft"][7] = x["target"][7, :2]
    x["target"][7, 2, 100] = float("nan")
    # 8, 9: supports that do not meet
    x["target"][8:, :, : V // 2] = float("-inf"); x["draft"][8:, :, V // 2:] = float("-inf")
    x["draft_tokens"][8:] = 1
    got = run(x)
    compare_verify(got, oracle_on(x), "f32")
    st = to_np(got["row_status"])
    assert st[1] & 1 and st[2] & 2 and st[3] & 4 and st[4] & 16 and st[5] & 1 and st[6] == 8 and st[7] & 1
    assert (to_np(got["accept_len"])[8:] == 0).all()


def test_back_to_back_calls_on_changing_inputs():
    """The launch of a call overlaps the end of what is before it in the stream: inputs written by a kernel right before the
    call are seen, and outputs of one call are not overtaken by the next."""
    cfg = G.Config("b2b", 64, 3, 8192, "bf16", 2.0, True, 1.0, 1.0, seed=3)
    xs = [G.make_inputs(G.replace(cfg, seed=s), DEV) for s in range(3)]
    want = [run(x) for x in xs]
    torch.cuda.synchronize()
    buf = {k: torch.empty_like(xs[0][k]) for k in ("target", "draft", "draft_tokens", "u_accept", "u_final")}
    got = []
    for i in range(9):
        for k in buf:
            buf[k].copy_(xs[i % 3][k])
        got.append(P.bebop_verify(buf["target"], buf["draft"], buf["draft_tokens"], buf["u_accept"], buf["u_final"]))
    for i, g in enumerate(got):
        for k in ("accept_len", "out_tokens", "tv", "p_draft", "q_draft", "row_status"):
            assert torch.equal(g[k], want[i % 3][k]), (i, k)


def test_a_wait_that_runs_out_returns_with_the_status_bit():
    cfg = G.Config("wait", 16, 3, 8192, "bf16", 2.0, True, 1.0, 1.0, seed=63)
    x = G.make_inputs(cfg, DEV)
    ok = run(x)
    P.bebop_debug_expire_wait(1)
    bad = run(x)
    torch.cuda.synchronize()
    assert (to_np(bad["row_status"]) & 32 == 32).all() and (to_np(bad["out_tokens"]) == -1).all()
    again = run(x)
    for k in ("accept_len", "out_tokens", "tv", "row_status"):
        assert torch.equal(again[k], ok[k]), k
