"""Sequences too large for eight CTAs, in more sequences than run at a time: the cluster size chosen by waves, against the
oracle, with the fp32 draw and with every draw evaluated in double; and the fp64 re-draw kernel on rows of few slices."""
import pytest

import bebop_gen as G
import paper_2606_12370_b200 as P
from parity import check_properties, compare_verify, oracle_on

pytestmark = pytest.mark.gpu


# (kernel path, shape): one wave of large clusters, a wave and one more sequence, ragged fp32; rows of one, eight and nine slices
@pytest.mark.parametrize("redraw", [False, True])
@pytest.mark.parametrize("path,dtype,B,K,V", [(4, "bf16", 8, 3, 151936), (4, "bf16", 9, 3, 151936), (4, "f32", 9, 5, 49999),
                                              (2, "bf16", 5, 2, 16383), (2, "bf16", 3, 1, 131072), (2, "f32", 3, 1, 65537)])
def test_against_the_oracle(path, dtype, B, K, V, redraw):
    cfg = G.Config("waves", B, K, V, dtype, 2.0, True, 0.8, (0.6, 1.2), ragged=K > 1, seed=B + K)
    x = G.make_inputs(cfg, "cuda", pad_ld=(-V) % 8)
    P.bebop_debug_force_general_path(path)
    try:
        if redraw:
            P.bebop_debug_set_draw_kappa(1e9)      # no fp32 draw clears its bound
        got = P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], draft_len=x["draft_len"],
                             temperature=x["temperature"], temperature_all=x["temperature_all"])
        assert P.bebop_debug_last_kernel() == (3 if path == 4 else 2)
        compare_verify(got, oracle_on(x), dtype, context=str(cfg))
        check_properties(got, x)
    finally:
        P.bebop_debug_set_draw_kappa(-1.0)
        P.bebop_debug_force_general_path(0)
