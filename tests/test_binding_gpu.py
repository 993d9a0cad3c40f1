"""What the Python binding promises beside the numbers: the outputs it makes (as programs get them: the sentinel that the other
tests fill them with is off here), the buffers it is given, and the exceptions it raises."""
import pytest
import torch

import bebop_gen as G
import paper_2606_12370_b200 as P
import paper_2606_12370_b200.binding as binding

pytestmark = pytest.mark.gpu
DEV = "cuda"
VERIFY = {"accept_len": ((5,), torch.int32), "out_tokens": ((5, 4), torch.int32), "tv": ((5, 3), torch.float32),
          "p_draft": ((5, 3), torch.float32), "q_draft": ((5, 3), torch.float32), "row_status": ((5,), torch.int32)}


@pytest.fixture(autouse=True)
def _no_sentinel(_poison_outputs):
    binding.POISON_OUTPUTS = False


@pytest.fixture(scope="module")
def x():
    return G.make_inputs(G.Config("b", 5, 3, 2048, "f32", 2.0, True, 0.8, 1.0, seed=1), DEV)


def verify(x, **kw):
    return P.bebop_verify(x["target"], x["draft"], x["draft_tokens"], x["u_accept"], x["u_final"], **kw)


def calls(x):
    return {"verify": verify(x), "tv": P.bebop_tv(x["target"][:, 0], x["draft"][:, 0]),
            "tv_static": P.bebop_tv_static(x["target"][:, 0], x["draft"][:, 0]), "greedy": P.bebop_greedy_verify(x["target"], x["draft_tokens"])}


# ------------------------------------------------------------------ outputs
def test_every_output_has_a_storage_of_its_own(x):
    for name, r in calls(x).items():
        out = {k: v for k, v in r.items() if k != "workspace"}
        assert len({v.untyped_storage().data_ptr() for v in out.values()}) == len(out), name
        for k, v in out.items():
            assert v.is_contiguous() and v.storage_offset() == 0 and not v.requires_grad and v.device == x["target"].device, (name, k)
            assert v.untyped_storage().nbytes() <= (4 * v.numel() + 511) // 512 * 512, (name, k)
    r = verify(x)
    keep = {k: v.clone() for k, v in r.items() if k != "workspace"}
    r["accept_len"].resize_(4096).fill_(-5)                  # what a program does to one output does not reach another
    for k in keep:
        if k != "accept_len":
            assert torch.equal(r[k], keep[k]), k


def test_new_outputs_given_outputs_and_none_agree(x):
    full = verify(x)
    for k, (shape, dtype) in VERIFY.items():
        assert tuple(full[k].shape) == shape and full[k].dtype == dtype, k
    given = {k: torch.full(s, -77, dtype=d, device=DEV) for k, (s, d) in VERIFY.items()}
    for keys in (list(VERIFY), ["accept_len", "tv"], ["out_tokens", "row_status"], []):
        out = {k: given[k].fill_(-77) for k in keys}
        r = verify(x, out=out)
        for k in VERIFY:
            assert torch.equal(r[k], full[k]), (keys, k)
            assert (r[k] is out[k]) if k in out else r[k].data_ptr() not in [v.data_ptr() for v in out.values()]
    r = verify(x, out={"tv": given["tv"]}, want_tv=False, want_probs=False, want_status=False)      # (a given buffer is always written)
    assert r["tv"] is given["tv"] and r["p_draft"] is None and r["q_draft"] is None and r["row_status"] is None
    assert torch.equal(r["tv"], full["tv"]) and torch.equal(r["out_tokens"], full["out_tokens"])
    t = P.bebop_tv(x["target"][:, 0], x["draft"][:, 0], want_s_aux=False, want_status=False)
    assert t["s_aux"] is None and t["row_status"] is None and t["tv"].shape == (5,)


# ------------------------------------------------------------------ exceptions
def test_an_allocation_that_fails_raises_what_torch_raises(x):
    """Programs catch torch.cuda.OutOfMemoryError to free memory and call again.  The allocator's limit for this process is set to
    what it holds already (and put back)."""
    torch.cuda.synchronize(); torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    hold = []
    torch.cuda.set_per_process_memory_fraction(torch.cuda.memory_reserved() / total)
    try:
        for n in (1 << 21, 1 << 9):                          # what is free inside the blocks held
            with pytest.raises(torch.cuda.OutOfMemoryError):
                while True:
                    hold.append(torch.empty(n, dtype=torch.uint8, device=DEV))
        with pytest.raises(torch.cuda.OutOfMemoryError):
            verify(x)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
        hold.clear()
    assert verify(x)["accept_len"].shape == (5,)


def test_what_the_binding_takes_and_refuses(x):
    t, d = x["target"][:, 0], x["draft"][:, 0]
    want = P.bebop_tv(t, d, temperature_all=0.5)["tv"]
    for tau in (0.5, "0.5", torch.tensor(0.5), torch.tensor([0.5], device=DEV)):      # whatever float() takes
        assert torch.equal(P.bebop_tv(t, d, temperature_all=tau)["tv"], want)
    assert torch.equal(P.bebop_tv(t, d, temperature_all=1)["tv"], P.bebop_tv(t, d)["tv"])
    for bad in (lambda: P.bebop_tv(x["target"], x["draft"]), lambda: P.bebop_greedy_verify(t, x["draft_tokens"]), lambda: P.bebop_verify(
            t, d, x["draft_tokens"], x["u_accept"], x["u_final"])):
        with pytest.raises(ValueError):
            bad()
    for bad in (False, True, 0, "no"):                       # a workspace is a tensor or None
        with pytest.raises((TypeError, AttributeError)):
            P.bebop_tv(t, d, workspace=bad)
    with pytest.raises(P.BebopError) as e:
        P.bebop_tv(t, d, workspace=torch.empty(256, dtype=torch.uint8, device=DEV))
    assert e.value.code == 5
    with pytest.raises(P.BebopError) as e:
        P.bebop_tv(t.half(), d.half())
    assert e.value.code == 3
