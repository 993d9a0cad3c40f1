"""Finite logits far from zero, through every kernel, against the oracle: masks of a large negative number on one side of a
row pair, rows that hold nothing but such a mask, and temperatures that carry ordinary logits far out.  Every case is
well defined (the softmax subtracts the maximum), so no status bit and no tolerance is given away."""
import numpy as np
import pytest
import torch

import bebop_gen as G
import oracle
import paper_2606_12370_b200 as P
from parity import TOL, compare_verify, oracle_on, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda"
PATHS = {"auto": 0, "pipe": 2, "fuse": 3, "seq": 4}
TYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


@pytest.fixture(autouse=True, params=list(PATHS))
def kernel_path(request):
    P.bebop_debug_force_general_path(PATHS[request.param])
    yield request.param
    P.bebop_debug_force_general_path(0)


def check_tv(tgt, drf, tau, dtype):
    got = P.bebop_tv(tgt, drf, temperature=tau)
    ref = oracle.tv(tgt.float().cpu().numpy(), drf.float().cpu().numpy(), temperature=to_np(tau))
    np.testing.assert_array_equal(to_np(got["row_status"]), ref["row_status"])
    assert np.abs(to_np(got["tv"]) - ref["tv"]).max() <= TOL[dtype], (to_np(got["tv"]), ref["tv"])
    assert np.abs(to_np(got["s_aux"]) - ref["s_aux"]).max() <= TOL[dtype], (to_np(got["s_aux"]), ref["s_aux"])


# a quarter of the vocabulary lies under the mask in the rows named; masks as programs write them
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mask", [-60.0, -1e4, -1e9, "lowest"])
def test_a_finite_mask_on_one_side(dtype, mask):
    """The other side has its mass under the mask: p and q do not meet there, and the ratio of the two rows' scales over that
    part of the vocabulary is far beyond fp32."""
    N, V = 24, 16384
    low = float(torch.finfo(TYPES[dtype]).min) if mask == "lowest" else mask
    g = torch.Generator(device=DEV).manual_seed(5)
    tgt, drf = 0.01 * torch.randn(N, V, generator=g, device=DEV), torch.randn(N, V, generator=g, device=DEV)
    drf[:, 7] = 14.0; drf[:, 3000] = 13.0                    # nearly all of q: the sums around the maxima differ by 2^13
    tgt[:8, : V // 4] = low                                  # p flat outside the mask
    tgt[8:16], drf[8:16] = drf[8:16].clone(), tgt[8:16].clone()
    drf[8:16, : V // 4] = low                                # the other way round
    tgt[16:, : V // 4] = low; drf[16:, : V // 4] = low       # on both sides
    tgt, drf = tgt.to(TYPES[dtype]), drf.to(TYPES[dtype])
    tau = torch.linspace(0.6, 1.2, N, device=DEV)
    check_tv(tgt, drf, tau, dtype)
    # the same pairs as the draft positions of sequences of two (bonus row: the first target row again)
    B = N // 2
    x = dict(cfg=G.Config("m", B, 2, V, dtype, 1.0, False, 1.0, 1.0, seed=5), draft=drf.view(B, 2, V),
             target=torch.cat([tgt.view(B, 2, V), tgt.view(B, 2, V)[:, :1]], 1).contiguous(),
             draft_tokens=drf.float().argmax(-1).int().view(B, 2), draft_len=None, temperature=tau[:B].contiguous(), temperature_all=1.0,
             u_accept=torch.rand(B, 2, generator=g, device=DEV) * 0.98 + 0.01, u_final=torch.rand(B, generator=g, device=DEV) * 0.98 + 0.01)
    compare_verify(run_verify(x), oracle_on(x), dtype)


def run_verify(x, **kw):
    return P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], draft_len=x["draft_len"],
                          temperature=x["temperature"], temperature_all=x["temperature_all"], **kw)


FAR_PATHS = ("auto", "seq")


def far_inputs(dtype, V):
    """Ten sequences of two drafts, most with rows whose scaled logits lie beyond +-4e6."""
    B, K = 10, 2
    cfg = G.Config("far", B, K, V, dtype, 2.0, False, 0.5, 1.0, seed=V)
    x = G.make_inputs(cfg, DEV, pad_ld=(-V) % 8)
    t, d, low = x["target"], x["draft"], float(torch.finfo(TYPES[dtype]).min)
    tau = torch.ones(B, device=DEV)
    t[1, 0] = low                                            # a target row that is nothing but mask: p uniform
    d[2, 1] = -1e9; t[2, 1] = -1e9                           # both rows of a position
    t[3] = 1e9; d[3] = 1e9; t[3, :, : V // 2] = 1.1e9        # far up: p uniform over one half, q over all
    tau[4] = 1e-6                                            # ordinary logits, carried out by the temperature
    tau[5] = 1e-6; t[5] -= 20; d[5] -= 20
    d[6] = t[6, :2]; t[6, 2] = -1e9                          # the bonus row alone
    t[7, :, V // 3:] = low; d[7, :, V // 3:] = -1e9          # masks beside ordinary logits: nothing is far out
    t[8, 1] = 3e38; t[8, 1, 5:] = -3e38; d[8, 1] = t[8, 1]   # both ends of the type
    t[9, 0] = -1e9; t[9, 1, 3] = float("nan")                # a bad row behind a far one
    x["temperature"] = tau
    x["draft_tokens"] = d.float().argmax(-1).int().contiguous()
    x["draft_tokens"][3, 0] = V - 1                          # p(x) = 0 there: rejected
    x["u_accept"][6] = 0.5
    return x


@pytest.mark.parametrize("dtype,V", [("f32", 1024), ("bf16", 1024), ("bf16", 2051), ("f32", 30001), ("bf16", 65536)])
@pytest.mark.parametrize("kappa", [-1.0, 1e9])               # (1e9: no fp32 draw clears its bound)
def test_rows_far_from_zero(kernel_path, dtype, V, kappa):
    if kernel_path not in FAR_PATHS:
        pytest.skip("not through this kernel")
    x = far_inputs(dtype, V)
    ref = oracle_on(x)
    P.bebop_debug_set_draw_kappa(kappa)
    try:
        got = run_verify(x)
        bare = run_verify(x, want_tv=False, want_probs=False, want_status=False)
    finally:
        P.bebop_debug_set_draw_kappa(-1.0)
    compare_verify(got, ref, dtype)
    assert to_np(got["row_status"])[9] == 1 and (to_np(got["out_tokens"])[:9, 0] >= 0).all()
    for k in ("accept_len", "out_tokens"):                   # the optional outputs change nothing
        assert torch.equal(bare[k], got[k]), k
    # the call after it, on the same workspace, with ordinary rows
    y = G.make_inputs(x["cfg"], DEV, pad_ld=(-V) % 8)
    compare_verify(run_verify(y, workspace=got["workspace"]), oracle_on(y), dtype)


@pytest.mark.parametrize("dtype,V", [("f32", 1024), ("bf16", 2051), ("f32", 30001), ("bf16", 65536)])
def test_tv_of_rows_far_from_zero(kernel_path, dtype, V):
    if kernel_path not in FAR_PATHS:
        pytest.skip("not through this kernel")
    x = far_inputs(dtype, V)
    n = x["target"].shape[0] * 2
    tgt = torch.cat([x["target"][:, 0], x["target"][:, 1]])
    drf = torch.cat([x["draft"][:, 0], x["draft"][:, 1]])
    pad = lambda r: torch.cat([r, torch.zeros(n, (-V) % 8, dtype=r.dtype, device=DEV)], 1)[:, :V]
    check_tv(pad(tgt), pad(drf), x["temperature"].repeat(2), dtype)
