"""The work a user of this library has it do, as timed cases: one routing step per pass, through the public entry points.

A case names the kind of call and its sizes.  Kinds:
  route   bf16 head, device buffers (`Router.route`), optionally with a learned router, per-row thresholds, the
          opposite polarity and the first routed position of every sequence
  route8  the same on the 8-bit (e4m3) head, decode batches of up to 128 rows
  host    `tlr_route_host`: hidden states and results in pinned host memory
  shard   one rank's part of a vocabulary-sharded decode step: its summaries, then the merge of all ranks'

The hidden states mix rows of every confidence, as a decoder sees them: for each row one random token is given a
logit between one below and eight above the log of the vocabulary size, so that confidences run from about 0.2 to
0.9997 and roughly one row in five falls under the threshold of 0.7.
"""
import math

import torch

import paper_2504_07878_b200 as tlr

TAU = 0.7


def _case(kind, n, d, V, **options):
    return dict({"kind": kind, "n": n, "d": d, "V": V}, **options)


def listed():
    cases = [
        # the smallest call: one session's next token on a small head (launches and host work count)
        ("single_small", _case("route", 1, 256, 20000)),
        # one session on a large head: the time to read W
        ("single_wide", _case("route", 1, 2048, 128256)),
        # a small decode batch, the 0.5B-class head, bf16 and 8-bit
        ("decode16", _case("route", 16, 896, 151936)),
        ("decode16_8bit", _case("route8", 16, 896, 151936)),
        # a ragged decode batch on the 8-bit head whose decision is the learned router's
        ("decode100_8bit_router", _case("route8", 100, 2048, 128256, router=256)),
        # a hidden size whose rows are no multiple of 16 bytes (word-level heads of width 300)
        ("odd_hidden", _case("route", 64, 300, 33000)),
        # the benchmark workload: 256 sessions, one token each
        ("decode256", _case("route", 256, 896, 151936)),
        # the same batch from and to host memory
        ("host256", _case("host", 256, 896, 151936)),
        # the same batch on one of eight vocabulary shards
        ("shard256_of_8", _case("shard", 256, 896, 151936, shards=8, rank=3)),
        # seven returned contexts of 111 tokens re-scored: learned router, a threshold per session, first routed position
        ("rescore777_router", _case("route", 777, 1536, 151936, router=256, seq_len=111, per_row_tau=True)),
        # prefill scoring: 16 sequences of 512 tokens
        ("prefill8192", _case("route", 8192, 896, 151936, seq_len=512)),
        # the largest batch
        ("prefill16384", _case("route", 16384, 2048, 128256)),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log_int(rng, lo, hi, step=1):
    """An integer between lo and hi, spread over its logarithm, a multiple of step."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi // step, max(-(-lo // step), round(x / step))) * step


def draw(rng):
    kind = rng.choice(["route", "route", "route", "route", "options", "odd", "route8", "route8", "host", "shard"])
    V = _log_int(rng, 20000, 151936)
    if kind == "odd":
        d = _log_int(rng, 100, 1000)
        return _case("route", _log_int(rng, 1, 256), d + 1 if d % 8 == 0 else d, min(V, 60000))
    if kind == "route8":
        c = _case("route8", _log_int(rng, 1, 128), _log_int(rng, 256, 2048, 16), V)
        return dict(c, router=_log_int(rng, 64, 512)) if rng.random() < 0.3 else c
    d = _log_int(rng, 256, 2048, 8)
    if kind == "host":
        return _case("host", _log_int(rng, 1, 4096), d, V)
    if kind == "shard":
        shards = rng.choice([2, 4, 8])
        return _case("shard", _log_int(rng, 1, 512), d, V, shards=shards, rank=rng.randrange(shards))
    if kind == "options":
        seq_len = _log_int(rng, 1, 512)
        c = _case("route", seq_len * rng.randint(1, 16), d, V, seq_len=seq_len, per_row_tau=rng.random() < 0.5,
                  route_above=rng.random() < 0.3)
        return dict(c, router=_log_int(rng, 64, 512)) if rng.random() < 0.5 else c
    return _case("route", _log_int(rng, 1, 16384), d, min(V, 128256))


def _std(case):
    # large enough that a row can be confident: the 0.5B-class head's 0.02 and wider, more on narrow heads
    return 0.02 * max(1.0, 896.0 / case["d"])


def _head(case, gen):
    """W as the caller holds it: (bf16 [V, d], None) or (e4m3 codes, one scale per row); and its values as float."""
    V, d = case["V"], case["d"]
    W = torch.randn((V, d), generator=gen, device="cuda") * _std(case)
    if case["kind"] != "route8":
        return W.to(torch.bfloat16), None
    scale = W.abs().amax(dim=1) / 448.0
    return (W / scale[:, None]).to(torch.float8_e4m3fn), scale


def _hidden(case, W, scale, gen):
    """bf16 [n, d] rows of root mean square 1, each leaning towards one random token (see the head of this file)."""
    n, d, V = case["n"], case["d"], case["V"]
    g = torch.randn((n, d), generator=gen, device="cuda")
    w = W[torch.randint(0, V, (n,), generator=gen, device="cuda")].float()
    u = w / w.square().mean(dim=1, keepdim=True).sqrt()
    want = math.log(V) + torch.empty((n, 1), device="cuda").uniform_(-1.0, 8.0, generator=gen)
    r = (want / (_std(case) * d)).clamp(max=0.99)              # share of the row that points at the token
    h = g * (1.0 - r * r).sqrt() + u * r
    return (h / h.square().mean(dim=1, keepdim=True).sqrt()).to(torch.bfloat16)


def _peer_summaries(case, W, h):
    """[shards, n] summaries (max logit, its index, sum e^(z-m), sum e^(z-m)(z-m)) as the all-gather delivers them."""
    out = torch.empty((case["shards"], case["n"], 4), device="cuda")
    for g, (v0, v1) in enumerate(_bounds(case)):
        z = h.float() @ W[v0:v1].float().T
        m, i = z.max(dim=1)
        y = z - m[:, None]
        e = y.exp()
        out[g, :, 0], out[g, :, 2], out[g, :, 3] = m, e.sum(dim=1), (e * y).sum(dim=1)
        out.view(torch.int32)[g, :, 1] = (i + v0).to(torch.int32)
    return out


def _bounds(case):
    return [tlr.shard_bounds(case["V"], case["shards"], g) for g in range(case["shards"])]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, n, d = case["kind"], case["n"], case["d"]
    W, scale = _head(case, gen)
    h = _hidden(case, W, scale, gen)
    s = {"case": case, "h": h}
    if kind == "shard":
        v0, v1 = _bounds(case)[case["rank"]]
        s["gathered"] = _peer_summaries(case, W, h)
        s["v0"] = v0
        W = W[v0:v1].clone()                                   # the rank holds its own rows only
    router = s["router"] = tlr.Router(W, max_n=n, wscale=scale)
    router.routed_idx.zero_()
    if kind == "host":
        host = lambda dtype, size: torch.zeros(size, dtype=dtype, pin_memory=True)  # noqa: E731
        s["h"] = h.cpu().pin_memory()
        s["out"] = [host(torch.int32, n), host(torch.float32, n), host(torch.float32, n), host(torch.uint8, n),
                    host(torch.int32, n), host(torch.int32, 1)]
        return s
    options = {}
    if case.get("router"):
        width = case["router"]
        rand = lambda *size: torch.randn(size, generator=gen, device="cuda")  # noqa: E731
        router.set_router_mlp((rand(width, d) / d ** 0.5).to(torch.bfloat16), rand(width) * 0.1, rand(width) * 0.2, 0.3)
        options.update(score_source=tlr.TLR_SCORE_MLP, mlp_score=torch.zeros(n, device="cuda"))
    if case.get("per_row_tau"):
        options["tau_per_row"] = 0.4 + 0.4 * torch.rand(n, generator=gen, device="cuda")
    if case.get("route_above"):
        options["route_above"] = True
    if case.get("seq_len"):
        options.update(seq_len=case["seq_len"],
                       first_routed=torch.zeros(n // case["seq_len"], dtype=torch.int32, device="cuda"))
    s["options"] = options
    return s


def run(s):
    case, router = s["case"], s["router"]
    n = case["n"]
    if case["kind"] == "host":
        tlr.tlr_route_host(router.ctx, s["h"], n, TAU, *s["out"])
        return s["out"]
    if case["kind"] == "shard":
        mine = s["gathered"][case["rank"]]
        tlr.tlr_shard_summary(router.ctx, s["h"], n, s["v0"], mine)
        tlr.tlr_shard_finish(router.ctx, s["gathered"], case["shards"], n, TAU, router.token, router.conf,
                             router.entropy, router.route_mask, router.routed_idx, router.routed_count)
        return [router.token, router.conf, router.entropy, router.route_mask, router.routed_idx, router.routed_count]
    out = list(router.route(s["h"], TAU, **s["options"]))
    return out + [s["options"][k] for k in ("mlp_score", "first_routed") if k in s["options"]]


def work(case):
    n, d, V = case["n"], case["d"], case["V"]
    width = case.get("router", 0)
    out = 17 * n + 4 + (4 * n + 8 * width if width else 0) + (4 * n if case.get("per_row_tau") else 0)
    if case.get("seq_len"):
        out += 4 * (n // case["seq_len"])
    if case["kind"] == "shard":
        v0, v1 = _bounds(case)[case["rank"]]
        V = v1 - v0
        out += 16 * n * case["shards"]
    head = V * d + 4 * V if case["kind"] == "route8" else 2 * V * d
    return {"bytes": head + 2 * n * d + 2 * width * d + out, "flops": 2.0 * n * d * (V + width)}


def tolerance(case):
    # fp32 accumulation of exact products and fp32 sums over the vocabulary: against 64-bit arithmetic the confidences
    # are off by up to 4e-6 and the entropies (small differences of sums near 1) by up to 3e-5.  A row whose two best
    # logits, or whose score and threshold, are closer than that may go either way, and shifts the list behind it.
    return {"rel": 1.2e-4, "max": 2.4e-4, "differ": 0.005}
