"""The stream (fused and pipelined kernel with a TV output) where its cuts fall: chunks of 128 and 256 16-byte vectors, one CTA
to eight per row, ragged last vectors, empty and ragged sequences, more and fewer units than clusters, rows short of a CTA's
slice; and the pipelined kernel's sweeps, which a call without a TV output takes.  Against the oracle."""
import numpy as np
import pytest
import torch

import bebop_gen as G
import oracle
import paper_2606_12370_b200 as P
from parity import TOL, check_properties, compare_verify, oracle_on, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(params=[2, 3])
def path(request):
    P.bebop_debug_force_general_path(request.param)
    yield request.param
    P.bebop_debug_force_general_path(0)


def vocab(dtype, vectors, tail):
    return (4 if dtype == "f32" else 8) * vectors - tail


# vectors per row: a chunk and its neighbours, one and more stages, ragged ends.  The calls are small, so rows of more than 3,072 vectors
# go over four or eight CTAs; 10,241 vectors over eight in chunks of 256 (path 2) leave the last of them one vector.  The limits of
# one, two and eight CTAs and of their chunk tables are test_the_limits_of_a_slice's.
# (V = 1 is left out: p = q = 1 there, and whether q <= p, by which S jumps from 1 to 0, is a matter of the last bit)
SIZES = [("bf16", 1, 3), ("f32", 128, 0), ("bf16", 129, 3), ("bf16", 257, 0), ("f32", 3073, 1), ("bf16", 7499, 5), ("f32", 7500, 2),
         ("bf16", 10240, 0), ("bf16", 10241, 1), ("f32", 15001, 3), ("bf16", 40960, 0), ("bf16", 40961, 7), ("f32", 81921, 1)]


@pytest.mark.parametrize("dtype,vectors,tail", SIZES)
def test_verify(path, dtype, vectors, tail):
    V = vocab(dtype, vectors, tail)
    cfg = G.Config("stream", 5 if vectors > 20000 else 11, 3, V, dtype, 2.0, V >= 64, 0.8, (0.6, 1.2), ragged=True, seed=vectors)
    x = G.make_inputs(cfg, "cuda", pad_ld=(-V) % 8)
    x["draft_len"][1] = 0                                   # a sequence that is its bonus row
    got = P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], draft_len=x["draft_len"],
                         temperature=x["temperature"], temperature_all=x["temperature_all"])
    assert P.bebop_debug_last_kernel_name() == ("k_pipe" if path == 2 else "k_fuse")
    ref = oracle_on(x)
    compare_verify(got, ref, dtype, context=str(cfg))
    check_properties(got, x)
    if path == 2:                                           # the same call without a TV output: the sweeps
        again = P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], draft_len=x["draft_len"],
                               temperature=x["temperature"], temperature_all=x["temperature_all"], want_tv=False)
        compare_verify({k: v for k, v in again.items() if k != "tv"}, ref, dtype, context=str(cfg) + " without tv")


@pytest.mark.parametrize("dtype,vectors,tail", SIZES)
def test_tv(path, dtype, vectors, tail):
    V, N = vocab(dtype, vectors, tail), 4 if vectors > 20000 else 300 if vectors < 200 else 9
    g = torch.Generator(device="cuda").manual_seed(vectors)
    store = torch.zeros((2, N, V + (-V) % 8), device="cuda")
    store[0, :, :V] = 2.0 * torch.randn((N, V), generator=g, device="cuda")
    store[1, :, :V] = store[0, :, :V] + torch.randn((N, V), generator=g, device="cuda")
    store = store.to(torch.float32 if dtype == "f32" else torch.bfloat16)
    got = P.bebop_tv(store[0, :, :V], store[1, :, :V])
    ref = oracle.tv(store[0, :, :V].float().cpu().numpy(), store[1, :, :V].float().cpu().numpy())
    assert np.abs(to_np(got["tv"]) - ref["tv"]).max() <= TOL[dtype]
    assert np.abs(to_np(got["s_aux"]) - ref["s_aux"]).max() <= TOL[dtype]
    assert (to_np(got["row_status"]) == 0).all()


@pytest.mark.parametrize("B,K", [(1, 1), (2, 32), (900, 1), (2000, 4)])
def test_shares(path, B, K):
    """Fewer units than clusters, a sequence cut by many of them, more sequences than threads of a CTA."""
    cfg = G.Config("shares", B, K, 1030, "bf16", 2.0, True, 0.8, 1.0, ragged=K > 1, seed=B + K)
    x = G.make_inputs(cfg, "cuda", pad_ld=2)
    got = P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], draft_len=x["draft_len"],
                         temperature=x["temperature"], temperature_all=x["temperature_all"])
    check_properties(got, x)
    idx = np.unique(np.linspace(0, B - 1, 200).astype(np.int64))
    compare_verify(got, oracle_on(x, idx), "bf16", idx=idx, context=str(cfg))


@pytest.mark.parametrize("B,K,V", [(6, 2, 1030), (300, 3, 20000)])
def test_a_wait_that_runs_out_leaves_no_output_unwritten(path, B, K, V):
    """Every CTA gives up on its first unit (test hook), so no sequence is completed: all outputs say so, and none keeps what
    the caller's buffer held."""
    x = G.make_inputs(G.Config("failed", B, K, V, "bf16", 2.0, True, 0.8, 1.0, seed=B), "cuda", pad_ld=(-V) % 8)
    P.bebop_debug_expire_wait(2)
    got = P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"])
    assert (to_np(got["row_status"]) & 32 == 32).all()
    assert (to_np(got["accept_len"]) == 0).all() and (to_np(got["out_tokens"]) == -1).all()
    for k in ("tv", "p_draft", "q_draft"):
        assert (to_np(got[k]) == 0).all(), k
    P.bebop_debug_expire_wait(2)
    tv = P.bebop_tv(x["target"][:, 0], x["draft"][:, 0])
    assert (to_np(tv["row_status"]) & 32 == 32).all() and (to_np(tv["tv"]) == 0).all() and (to_np(tv["s_aux"]) == 0).all()


@pytest.mark.parametrize("dtype,B,K,V,n", [("bf16", 230, 3, 89999, 100), ("f32", 300, 3, 27999, 200)])
def test_one_rule_for_the_chunks_whatever_the_name(dtype, B, K, V, n):
    """A batch on one side of the line between the names and a part of it on the other: the same bits for the same sequences."""
    x = G.make_inputs(G.Config("name", B, K, V, dtype, 2.0, True, 0.8, 0.9, seed=B), "cuda", pad_ld=(-V) % 8)
    part = {k: None if x[k] is None else x[k][:n].contiguous() if k not in ("target", "draft") else x[k][:n] for k in ("target", "draft", "draft_tokens", "u_accept", "u_final")}
    a, b = (P.bebop_verify(y["target"], y["draft"], y["draft_tokens"], y["u_accept"], y["u_final"], temperature_all=0.9) for y in (x, part))
    for k in ("accept_len", "out_tokens", "tv", "p_draft", "q_draft", "row_status"):
        assert torch.equal(a[k][:n], b[k]), k


def sampled(cfg, x, got, n, context=""):
    idx = np.unique(np.linspace(0, cfg.B - 1, n).astype(np.int64))
    compare_verify(got, oracle_on(x, idx), cfg.dtype, idx=idx, context=str(cfg) + context)
    check_properties(got, x)


# the resident form: rows of one chunk, of a chunk and a vector, around half and all of what fits (1,536 vectors: four stages), and the
# first row beyond it; sequences of no drafts, cut by clusters, temperatures of their own; with and without a TV output
@pytest.mark.parametrize("dtype,vectors,tail,B,K", [("bf16", 1, 3, 400, 5), ("f32", 128, 0, 500, 3), ("bf16", 129, 5, 900, 4), ("bf16", 769, 7, 400, 8),
                                                     ("f32", 1024, 1, 300, 2), ("bf16", 1535, 7, 300, 2), ("bf16", 1536, 0, 200, 4), ("f32", 1536, 3, 160, 32),
                                                     ("bf16", 1537, 0, 300, 3)])
def test_resident_rows(dtype, vectors, tail, B, K):
    V = vocab(dtype, vectors, tail)
    cfg = G.Config("resident", B, K, V, dtype, 2.0, V >= 64, 0.8, (0.6, 1.2), ragged=True, seed=vectors)
    x = G.make_inputs(cfg, "cuda", pad_ld=(-V) % 8)
    x["draft_len"][::7] = 0
    P.bebop_debug_force_general_path(3)
    try:
        for tv in (True, False):
            got = P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], draft_len=x["draft_len"],
                                 temperature=x["temperature"], temperature_all=x["temperature_all"], want_tv=tv)
            assert P.bebop_debug_last_kernel_name() == "k_fuse"
            sampled(cfg, x, got, 96)
    finally:
        P.bebop_debug_force_general_path(0)


def test_resident_rows_masked_and_broken():
    """What the chunks of the resident form meet besides ordinary logits: masks, NaN, empty rows, bad tokens and temperatures."""
    cfg = G.Config("res", 40, 3, 9000, "bf16", 2.0, True, 0.8, 1.0, seed=9)
    x = G.make_inputs(cfg, "cuda")
    t, d = x["target"], x["draft"]
    t[1, :, 3000:] = float("-inf"); d[1, :, 3000:] = float("-inf")
    t[2, 0, :8192] = -1e9; d[3, 1, 64:] = -1e4
    t[4, 1, 8999] = float("nan"); d[5, 0, 0] = float("inf"); d[6, 2] = float("-inf"); t[7, 3] = float("-inf")
    x["draft_tokens"][1:4] = 5
    x["draft_tokens"][8, 1] = 9000
    x["temperature"] = torch.ones(40, device="cuda"); x["temperature"][9] = -1.0; x["temperature"][10] = float("nan")
    d[11] = t[11, :3]                                       # p = q: everything is accepted
    P.bebop_debug_force_general_path(3)
    try:
        got = P.bebop_verify(t, d, x["draft_tokens"], x["u_accept"], x["u_final"], temperature=x["temperature"])
        compare_verify(got, oracle_on(x), "bf16")
        P.bebop_debug_set_draw_kappa(1e9)                   # no fp32 draw clears its bound: the re-draw kernel does them all
        compare_verify(P.bebop_verify(t, d, x["draft_tokens"], x["u_accept"], x["u_final"], temperature=x["temperature"]), oracle_on(x), "bf16")
    finally:
        P.bebop_debug_set_draw_kappa(-1.0)
        P.bebop_debug_force_general_path(0)


# rows at the limits of a CTA's slice, in batches for which one, two and eight CTAs share a row: 10,240 vectors over one (40 large chunks) and
# one more, over two; 7,500 over one in small chunks (59); 40,960 over two, whose tables of 80 large chunks they fill; 163,840 over eight,
# the longest rows of the stream
@pytest.mark.parametrize("dtype,vectors,tail,B,K", [("bf16", 10240, 0, 120, 3), ("bf16", 10241, 1, 120, 3), ("f32", 7500, 0, 300, 3),
                                                     ("bf16", 40960, 3, 60, 3), ("f32", 163840, 0, 6, 2)])
def test_the_limits_of_a_slice(dtype, vectors, tail, B, K):
    V = vocab(dtype, vectors, tail)
    cfg = G.Config("limits", B, K, V, dtype, 2.0, True, 0.8, 0.9, seed=vectors)
    x = G.make_inputs(cfg, "cuda", pad_ld=(-V) % 8)
    P.bebop_debug_force_general_path(3)
    try:
        got = P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], temperature_all=0.9)
        assert P.bebop_debug_last_kernel_name() == "k_fuse"
        sampled(cfg, x, got, 6 if vectors > 20000 else 24)
    finally:
        P.bebop_debug_force_general_path(0)


def test_the_limits_of_a_slice_tv():
    N, V = 100, 8 * 40960
    g = torch.Generator(device="cuda").manual_seed(3)
    tgt = (2.0 * torch.randn((N, V), generator=g, device="cuda")).to(torch.bfloat16)
    drf = (tgt.float() + torch.randn((N, V), generator=g, device="cuda")).to(torch.bfloat16)
    P.bebop_debug_force_general_path(3)
    got = P.bebop_tv(tgt, drf)
    P.bebop_debug_force_general_path(0)
    sel = [0, 1, 50, 98, 99]
    ref = oracle.tv(tgt[sel].float().cpu().numpy(), drf[sel].float().cpu().numpy())
    assert np.abs(to_np(got["tv"])[sel] - ref["tv"]).max() <= TOL["bf16"] and np.abs(to_np(got["s_aux"])[sel] - ref["s_aux"]).max() <= TOL["bf16"]


# ---- the sweeps (path 2 without a TV output), which the suites of the other files reach through calls with TV no longer
@pytest.fixture
def sweeps():
    P.bebop_debug_force_general_path(2)
    yield lambda x, **kw: P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], draft_len=x["draft_len"],
                                         temperature=x["temperature"], temperature_all=x["temperature_all"], want_tv=False, **kw)
    P.bebop_debug_set_draw_kappa(-1.0)
    P.bebop_debug_force_general_path(0)


def test_sweeps_fast_draw_bound_over_many_seeds(sweeps):
    """As the calibration of the other kernels: no unflagged mismatch, and none with a quarter of the factor either."""
    B, K, V = 224, 3, 151936
    off = P.bebop_debug_fallback_offset(B, K, V, 1)
    redrawn = seen = wrong = 0
    for seed in range(8):
        flat = seed % 2 == 1
        cfg = G.Config("cert", B, K, V, "bf16", 1.0 if flat else 3.0, not flat, 1.5 if flat else 1.0, (0.6, 0.7, 1.0, 1.2)[seed % 4], seed=2000 + seed)
        x = G.make_inputs(cfg, "cuda")
        if seed % 3 == 0:
            x["draft_len"] = torch.tensor([i % 2 for i in range(B)], dtype=torch.int32, device="cuda")
        got = sweeps(x)
        assert P.bebop_debug_last_kernel_name() == "k_pipe"
        redrawn += int(got["workspace"][off:off + 4].view(torch.int32).item())
        ref = oracle_on(x)
        compare_verify(got, ref, "bf16", context=str(cfg))
        P.bebop_debug_set_draw_kappa(1.0)
        again = sweeps(x, workspace=got["workspace"])
        P.bebop_debug_set_draw_kappa(-1.0)
        wrong += int(((to_np(again["out_tokens"]) != ref["out_tokens"]).any(axis=1) & ~ref["flagged"]).sum())
        seen += B
    print("\nfast-draw bound (sweeps): %d sequences, %d (%.2f %%) re-drawn in fp64" % (seen, redrawn, 100.0 * redrawn / seen))
    assert wrong == 0 and redrawn <= 0.06 * seen


@pytest.mark.parametrize("which", [1, 2])
def test_sweeps_a_wait_that_runs_out_returns_with_the_status_bit(sweeps, which):
    cfg = G.Config("wait", 64, 3, 8192, "bf16", 2.0, True, 1.0, 1.0, seed=63)
    x = G.make_inputs(cfg, "cuda")
    ok = sweeps(x)
    P.bebop_debug_expire_wait(which)
    bad = sweeps(x, workspace=ok["workspace"])
    torch.cuda.synchronize()                                # returns: nothing hangs
    assert (to_np(bad["row_status"]) & 32 == 32).all()
    again = sweeps(x, workspace=ok["workspace"])
    for k in ("accept_len", "out_tokens", "row_status"):
        assert torch.equal(again[k], ok[k]), k
    compare_verify(again, oracle_on(x), cfg.dtype)


def test_sweeps_status_bits_and_masks(sweeps):
    cfg = G.Config("st", 12, 2, 20000, "f32", 1.0, False, 0.5, 1.0, seed=4)
    x = G.make_inputs(cfg, "cuda")
    t, d = x["target"], x["draft"]
    x["temperature"] = torch.ones(12, device="cuda"); x["temperature"][4] = 0.0
    t[1, 0, 17] = float("nan"); d[2, 1, :] = float("-inf"); x["draft_tokens"][3, 1] = 20000; t[5, 1, 5] = float("inf")
    d[6] = t[6, :2]; t[6, 0, 9] = float("-inf"); d[6, 0, 9] = float("-inf"); x["draft_tokens"][6, 0] = 9        # p = q: no residual at the reject
    d[7] = t[7, :2]; t[7, 2, 100] = float("nan")                                                                  # a bad bonus row
    t[8, :, :10000] = float("-inf"); d[8, :, 10000:] = float("-inf"); x["draft_tokens"][8] = 11                  # supports that do not meet
    t[9, :, : 5000] = -1e9; t[10, 1, 300:] = -1e4
    got = sweeps(x)
    compare_verify(got, oracle_on(x), "f32")
    st = to_np(got["row_status"])
    assert st[1] & 1 and st[2] & 2 and st[3] & 4 and st[4] & 16 and st[5] & 1 and st[6] == 8 and st[7] & 1 and st[0] == 0


@pytest.mark.parametrize("dtype,B,K,V", [("bf16", 600, 2, 20000), ("f32", 600, 2, 20000), ("bf16", 5, 2, 16383), ("bf16", 3, 1, 131072), ("f32", 3, 1, 65537)])
def test_sweeps_every_sequence_goes_to_the_fp64_redraw(sweeps, dtype, B, K, V):
    cfg = G.Config("redraw", B, K, V, dtype, 2.0, True, 0.8, (0.6, 1.2), ragged=True, seed=B + K)
    x = G.make_inputs(cfg, "cuda", pad_ld=(-V) % 8)
    P.bebop_debug_set_draw_kappa(1e9)
    got = sweeps(x)
    off = P.bebop_debug_fallback_offset(B, K, V, 0 if dtype == "f32" else 1)
    assert int(got["workspace"][off:off + 4].view(torch.int32).item()) == B
    sampled(cfg, x, {k: v for k, v in got.items() if k != "tv"}, 64)
