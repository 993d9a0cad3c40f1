"""Finite logits far from zero, through every kernel, against the oracle: masks of a large negative number on one side of a
row pair.  Every case is well defined (the softmax subtracts the maximum), so no status bit and no tolerance is given
away."""
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
