"""The calls whose speed counts: what users of the verify step have it do, over the sizes they do it at.

A case names an entry point ("verify", "tv" or "greedy"), its sizes (B sequences, or row pairs for "tv"; K drafts;
V logits per row), the type of the logits and the recipe of their values.  Inputs are the seeded ones of `bebop_gen`
(draft = target + noise, drafts sampled from the draft distribution, supplied uniforms); rows whose length is not a
whole number of 16-byte vectors are padded, as the entry points ask for.
"""
import math

import torch

import bebop_gen as G
import paper_2606_12370_b200 as P

MAX_BYTES = 1.9e9          # logits of the largest listed case, rounded up: drawn cases stay below

# How logits are distributed: "plain" N(0, 2^2) with close drafts, "peaked" N(0, 3^2) plus eight Zipf-ranked peaks per
# row (a trained model's rollout), "flat" N(0, 1) with far drafts (high-entropy regime).
RECIPES = {"plain": (2.0, False, 0.5), "peaked": (3.0, True, 1.0), "flat": (1.0, False, 1.5)}


def _case(name, op, B, K, V, dtype="bf16", recipe="peaked", temperature="one", ragged=False, tv=True):
    """temperature: "one" (1.0 for all), "half" (0.7 for half of the rows) or "rows" (per row, 0.6 to 1.2);
    ragged: draft counts uniform in 1..K; tv: the call asks for TV and for p, q of the drafts."""
    return dict(name=name, op=op, B=B, K=K, V=V, dtype=dtype, recipe=recipe, temperature=temperature, ragged=ragged, tv=tv)


def listed():
    return [
        # the smallest call: a toy vocabulary, latency and launches only
        _case("verify_tiny", "verify", 4, 3, 1024, dtype="f32", recipe="plain"),
        # one stream of interactive decoding over a production vocabulary
        _case("verify_one_stream", "verify", 1, 3, 151936),
        # fp32 logits, a vocabulary that is no round number, ragged drafts, a temperature per request
        _case("verify_f32_odd", "verify", 24, 5, 49999, dtype="f32", temperature="rows", ragged=True),
        # a middle-sized vocabulary at a serving batch, long drafts
        _case("verify_mid_vocab", "verify", 192, 7, 32000, temperature="half", ragged=True),
        # rollout batches of RL training
        _case("verify_rollout", "verify", 64, 3, 151936),
        _case("verify_headline", "verify", 256, 3, 151936),
        # the high-entropy regime where only the tokens are wanted (a serving engine keeps no statistics)
        _case("verify_tokens_only", "verify", 256, 5, 151936, recipe="flat", tv=False),
        # the largest vocabulary
        _case("verify_large_vocab", "verify", 512, 3, 262144, temperature="half"),
        # the full rollout batch: ragged drafts, a temperature per row
        _case("verify_full_batch", "verify", 1024, 4, 151936, temperature="rows", ragged=True),
        # forward value of the TV loss (and the scalar its gradient needs) over the rows of a training batch
        _case("tv_loss", "tv", 768, 1, 151936),
        # the same on a small evaluation batch with fp32 logits and an odd vocabulary
        _case("tv_f32_odd", "tv", 100, 1, 32003, dtype="f32", temperature="rows"),
        # greedy drafts compared with the argmax of the target
        _case("greedy_high_entropy", "greedy", 256, 5, 151936, recipe="flat"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["verify", "verify", "verify", "tv", "greedy"])
    c = _case("", op, _log_int(rng, 1, 1024), 1 if op == "tv" else rng.randint(1, 8), _log_int(rng, 1024, 262144),
              dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]), recipe=rng.choice(list(RECIPES)),
              temperature=rng.choice(["one", "half", "rows"]), ragged=op != "tv" and rng.random() < 0.5,
              tv=op != "verify" or rng.random() < 0.75)
    del c["name"]
    while _logits(dict(c, ragged=False)) * _size(c) > MAX_BYTES:
        c["B"] = c["B"] * 3 // 4
    return c


def _size(c):
    return 4 if c["dtype"] == "f32" else 2


def _logits(c):
    """Logits the method reads: per sequence L target rows, L draft rows and the bonus row (greedy: no draft rows; TV:
    no bonus row); ragged drafts count with their mean."""
    L = (1 + c["K"]) / 2 if c["ragged"] else c["K"]
    rows = {"verify": 2 * L + 1, "tv": 2, "greedy": L + 1}[c["op"]]
    return c["B"] * rows * c["V"]


def _rows_of(c, seed):
    """[N, V] target and draft rows for the TV entry point, in padded storage."""
    std, peaks, noise = RECIPES[c["recipe"]]
    dt, N, V = G.torch_dtype(c["dtype"]), c["B"], c["V"]
    ld = V + (-V) % (16 // _size(c))
    g = torch.Generator(device="cuda").manual_seed(seed)
    store = torch.zeros((2, N, ld), dtype=dt, device="cuda")
    heights = 8.0 * torch.arange(1, 9, device="cuda", dtype=torch.float32) ** (-2.0 / 3.0)
    for a in range(0, N, 64):
        n = min(64, N - a)
        t = torch.randn((n, V), generator=g, device="cuda") * std
        if peaks:
            t.scatter_add_(1, torch.randint(0, V, (n, 8), generator=g, device="cuda"), heights.expand(n, 8))
        store[0, a:a + n, :V] = t
        store[1, a:a + n, :V] = t + noise * torch.randn((n, V), generator=g, device="cuda")
    tau = None
    if c["temperature"] == "rows":
        tau = 0.6 + 0.6 * torch.rand(N, generator=g, device="cuda")
    elif c["temperature"] == "half":
        tau = torch.ones(N, device="cuda")
        tau[: N // 2] = 0.7
    return store[0, :, :V], store[1, :, :V], tau


def prepare(case, seed):
    c = case
    dt = P.BEBOP_F32 if c["dtype"] == "f32" else P.BEBOP_BF16
    # the workspace and the outputs' buffers are what a program that calls the step in a loop keeps
    s = dict(op=c["op"], ws=torch.empty(P.bebop_workspace_bytes(c["B"], c["K"], c["V"], dt), dtype=torch.uint8, device="cuda"))
    if c["op"] == "tv":
        s["target"], s["draft"], s["temperature"] = _rows_of(c, seed)
        return s
    std, peaks, noise = RECIPES[c["recipe"]]
    cfg = G.Config("case", c["B"], c["K"], c["V"], c["dtype"], std, peaks, noise,
                   {"one": 1.0, "half": "half_0.7_1.0", "rows": (0.6, 1.2)}[c["temperature"]], ragged=c["ragged"], seed=seed)
    x = G.make_inputs(cfg, "cuda", draft_mode="argmax" if c["op"] == "greedy" else "sample", pad_ld=(-c["V"]) % (16 // _size(c)))
    s.update({k: x[k] for k in ("target", "draft", "draft_tokens", "draft_len", "temperature", "u_accept", "u_final")})
    if c["op"] == "verify":
        new = lambda shape, t: torch.empty(shape, dtype=t, device="cuda")
        B, K = c["B"], c["K"]
        s["tv"] = c["tv"]
        s["out"] = dict(accept_len=new((B,), torch.int32), out_tokens=new((B, K + 1), torch.int32), row_status=new((B,), torch.int32))
        if c["tv"]:
            s["out"].update({k: new((B, K), torch.float32) for k in ("tv", "p_draft", "q_draft")})
    else:
        s["draft"] = None
    return s


def run(state):
    s = state
    if s["op"] == "verify":
        r = P.bebop_verify(s["target"], s["draft"], s["draft_tokens"], s["u_accept"], s["u_final"], draft_len=s["draft_len"],
                           temperature=s["temperature"], out=s["out"], workspace=s["ws"], want_tv=s["tv"], want_probs=s["tv"])
        r.pop("workspace")
        return r
    if s["op"] == "tv":
        return P.bebop_tv(s["target"], s["draft"], temperature=s["temperature"], workspace=s["ws"])
    return P.bebop_greedy_verify(s["target"], s["draft_tokens"], draft_len=s["draft_len"], workspace=s["ws"])


def work(case):
    c = case
    n = _logits(c)
    # every logit once, and the tokens, uniforms and results of a sequence
    small = 4 * c["B"] * ({"verify": 6 * c["K"] + 6, "tv": 4, "greedy": 2 * c["K"] + 4}[c["op"]])
    # per logit: scale, exponential, sum, normalise, residual (greedy: one comparison)
    return {"bytes": float(n * _size(c) + small), "flops": float(n * (1 if c["op"] == "greedy" else 5))}


def tolerance(case):
    if case["op"] == "greedy":
        return "exact"
    # sums of fp32 exponentials; tokens are decided in double or certified, and may differ where the draw is a tie
    return {"rel": 1e-5, "differ": 1e-3}
