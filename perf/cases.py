"""The work that a program using this package has it do, as cases that can be timed and compared.

A verification step reads B x (K+1) rows of V logits and writes a few values per row, so three things decide what a
case stresses: how many bytes a step streams (latency at a few rows, bandwidth at thousands), whether rows have
16-byte structure, and which entry point the program calls.  Kinds:

  logits  verify() on a handle, or run_static() where the program cannot allocate; plain decode loops
  fused   verify_fused(): hidden states and the LM-head weight instead of logits
  shard   one rank of a vocabulary-parallel target: reduce_shard() on its slice, then run_partials()
  pld     pld_draft(): the drafter's n-gram retrieval before the step
  host    verify(host=True): logits in page-locked host memory
"""
import math

import torch

from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, binding, synthetic, verify, verify_fused

LLAMA_V, SERVING_V, TINY_V = synthetic.LLAMA3.V, synthetic.SERVING.V, synthetic.TINY.V
MAX_LOGIT_BYTES = synthetic.SERVING.rows * SERVING_V * 2     # the largest listed step
MAX_POSITIONS = synthetic.FUSED.rows                          # one pass over the weight


def _logits(**kw):
    case = dict(kind="logits", B=1, K=8, V=LLAMA_V, dtype="bf16", theta=1.0, unit="nats", W=3, carry=False,
                temperature=0.0, sampled=False, ready=False, static=False)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest step a program makes: one short fp32 round, all latency
        _logits(name="tiny_f32", V=TINY_V, dtype="f32"),
        # the paper's own operating point: one sequence of a 70B target, K = 15, W = 6, normalised threshold 0.3
        _logits(name="paper_one_sequence", K=15, theta=0.3, unit="normalized", W=6),
        # the paper's 405B draft length at temperature 1 with tokens the program sampled itself, from a server whose
        # memory pool owns the device (no handle)
        _logits(name="paper_sampled_static", B=4, K=25, theta=0.3, unit="normalized", W=6, temperature=1.0,
                sampled=True, static=True),
        # an ordinary decode batch over the Llama-3 vocabulary; the benchmark's default
        _logits(name="llama3_batch", B=16),
        # many long drafts at once
        _logits(name="long_draft", B=64, K=16),
        # high-batch serving with deferred state carried from round to round: the largest step
        _logits(name="serving_carry", B=256, V=SERVING_V, carry=True),
        # a vocabulary whose rows have no 16-byte structure, packed as the LM head writes them
        _logits(name="odd_vocab", B=32, V=50257),
        # LM head and verification in one: a few sequences (the weight, stored as linear layers store it, is the work)
        dict(name="fused_few", kind="fused", B=4, K=8, D=8192, V=LLAMA_V, vocab_major=True, theta=1.0, W=3),
        # the same at the batch that fills the tensor cores
        dict(name="fused_full", kind="fused", B=32, K=8, D=8192, V=LLAMA_V, vocab_major=False, theta=1.0, W=3),
        # one rank of the paper's 405B target over four GPUs: its slice of the vocabulary, then the merge
        dict(name="vocab_shard", kind="shard", B=4, K=25, V=LLAMA_V, world=4, dtype="bf16", theta=0.3, W=6),
        # drafting for a batch of long contexts
        dict(name="pld_long", kind="pld", B=32, L=32768, K=15, max_ngram=3, min_ngram=1),
        # logits that arrive in host memory: the copy over the bus and the step
        dict(name="host_batch", kind="host", B=16, K=8, V=LLAMA_V, dtype="bf16", theta=1.0, W=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng, multiple=1):
    """A vocabulary of the repository's configurations, or any size between 1000 and the largest of them."""
    if rng.random() < 0.5:
        v = rng.choice([TINY_V, 50264, LLAMA_V, SERVING_V] + ([50257] if multiple == 1 else []))
    else:
        v = _log(rng, 1000, SERVING_V)
    return max(multiple, v // multiple * multiple)


def draw(rng):
    kind = rng.choices(["logits", "fused", "shard", "pld", "host"], [6, 3, 1, 1, 1])[0]
    if kind == "logits":
        dtype = rng.choices(["bf16", "f32"], [3, 1])[0]
        V, K, B = _vocab(rng), rng.choice([1, 3, 5, 8, 10, 15, 16, 20, 25, 30]), _log(rng, 1, 256)
        B = max(1, min(B, MAX_LOGIT_BYTES // ((K + 1) * V * (4 if dtype == "f32" else 2))))
        static = rng.random() < 0.15
        carry = rng.random() < 0.3
        theta, unit = rng.choice([(0.5, "nats"), (1.0, "nats"), (2.0, "nats"), (0.3, "normalized")])
        W = min(rng.choice([0, 1, 3, 5, 6]), K) if carry else rng.choice([0, 1, 3, 5, 6])
        sampled = rng.random() < 0.2
        return _logits(B=B, K=K, V=V, dtype=dtype, theta=theta, unit=unit, W=W, carry=carry, static=static,
                       sampled=sampled, temperature=rng.choice([0.7, 1.0, 1.5]) if sampled else 0.0,
                       ready=rng.random() < 0.25)   # a queue of steps over logits that are all in memory already
    if kind == "fused":
        K = rng.choice([1, 3, 5, 8, 15])
        B = max(1, min(_log(rng, 1, 64), MAX_POSITIONS // (K + 1)))
        return dict(kind="fused", B=B, K=K, D=max(64, _log(rng, 512, 8192) // 8 * 8), V=min(LLAMA_V, max(4096, _vocab(rng, 8))),
                    vocab_major=rng.random() < 0.5, theta=rng.choice([0.5, 1.0, 2.0]), W=rng.choice([1, 3, 6]))
    if kind == "shard":
        return dict(kind="shard", B=_log(rng, 1, 64), K=rng.choice([3, 8, 15, 25]), V=max(8000, _vocab(rng)),
                    world=rng.choice([2, 4, 8]), dtype=rng.choices(["bf16", "f32"], [3, 1])[0], theta=rng.choice([0.3, 0.1]),
                    W=rng.choice([3, 6]))
    if kind == "pld":
        mn = rng.choice([1, 1, 2])
        return dict(kind="pld", B=_log(rng, 1, 64), L=_log(rng, 256, 16384), K=rng.choice([5, 8, 15, 25]),
                    max_ngram=rng.choice([2, 3, 4, 5]), min_ngram=mn)
    return dict(kind="host", B=_log(rng, 1, 16), K=rng.choice([3, 5, 8]), V=rng.choice([TINY_V, 50257, LLAMA_V]),
                dtype="bf16", theta=rng.choice([0.5, 1.0, 2.0]), W=rng.choice([1, 3]))


# ---- inputs -----------------------------------------------------------------------------------------------------

def _recipe(case, seed, V=None):
    """The repository's recipe for rows of this kind; its seeds derive from the name."""
    fp32 = case.get("dtype") == "f32"
    base = synthetic.TINY if fp32 else synthetic.SERVING if case.get("carry") else synthetic.LLAMA3
    return synthetic.shrink(base, name="%s seed %d" % (base.name, seed), B=case["B"], K=case["K"], V=V or case["V"],
                            dtype=case.get("dtype", "bf16"))


def _logits_and_draft(case, seed, device="cuda"):
    w = _recipe(case, seed)
    logits = synthetic.make_logits(w, 0, device=device)
    return logits, synthetic.make_draft(w, 0, synthetic.rank5(logits.view(-1, w.V)))


def _sample(logits, temperature, seed):
    """Tokens [B, K+1] drawn from softmax(logits / T), as a sampling loop draws them."""
    g = torch.Generator(device=logits.device)
    g.manual_seed(seed)
    u = torch.rand(logits.shape, generator=g, device=logits.device).clamp_(min=1e-20)
    return (logits.float() / temperature - torch.log(-torch.log(u))).argmax(-1).to(torch.int32)


def _tokens(case, seed):
    """Contexts [B, L] of skewed token ids; most end in tokens that occurred before, as text does."""
    B, L = case["B"], case["L"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    u = torch.rand(B, L, generator=g, device="cuda")
    tokens = (LLAMA_V * u ** 3).to(torch.int32).clamp_(max=LLAMA_V - 1)
    lengths = (L * (0.5 + 0.5 * torch.rand(B, generator=g, device="cuda"))).to(torch.int64).clamp_(min=16)
    repeat = torch.randint(0, 6, (B,), generator=g, device="cuda")          # how many of the last tokens recur
    back = (torch.rand(B, generator=g, device="cuda") * (lengths - 12)).to(torch.int64)
    rows = torch.arange(B, device="cuda")
    for i in range(5):
        sel = repeat > i
        tokens[rows[sel], (lengths - 1 - i)[sel]] = tokens[rows[sel], (back + 5 - i)[sel]]
    return tokens, lengths.to(torch.int32)


def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    s = {"case": case, "stream": stream}
    kind = case["kind"]
    if kind == "pld":
        s["tokens"], s["lengths"] = _tokens(case, seed)
        return s
    B, K, V = case["B"], case["K"], case["V"]
    out = s["out"] = VerifyBuffers(B, K, "cuda", pinned=kind == "host")
    if kind == "fused":
        w = synthetic.shrink(synthetic.FUSED, name="fused seed %d" % seed, B=B, K=K, V=V, hidden=case["D"],
                             weight_std=0.02 * math.sqrt(synthetic.FUSED.hidden / case["D"]))
        hidden, weight = synthetic.make_hidden(w, 0, device="cuda"), synthetic.make_weight(w, device="cuda")
        top = (hidden @ weight).float().argmax(1, keepdim=True)
        s["fv"] = FlyVerify(B, K, V, "bf16", hidden=case["D"])
        if case["vocab_major"]:
            s["fv"].set_weight_layout(True)
            weight = weight.t().contiguous()
        s.update(hidden=hidden, weight=weight, draft=synthetic.make_draft(w, 0, top))
        return s
    logits, draft = _logits_and_draft(case, seed)
    if kind == "host":
        s.update(fv=FlyVerify(B, K, V, case["dtype"]), logits=logits.cpu().pin_memory(), draft=draft.cpu().pin_memory())
        return s
    if kind == "shard":
        rows, world = B * (K + 1), case["world"]
        flat = logits.view(rows, V)
        width = -(-(-(-V // world)) // 8) * 8                   # slices start at multiples of 8 tokens
        gathered = torch.empty(world, rows, 4, dtype=torch.float32, device="cuda")
        for rank in range(world - 1, -1, -1):                   # the other ranks' states, as the all-gather brings them
            lo = rank * width
            mine = flat[:, lo:min(V, lo + width)].contiguous()
            fv = FlyVerify(B, K, mine.shape[1], case["dtype"])
            fv.reduce_shard(mine, lo, gathered[rank], stream)
        s.update(fv=fv, logits=mine, offset=lo, gathered=gathered, draft=draft)
        s["args"] = fv.make_args(B, K, draft, out.accept_len, out.out_tokens, theta=case["theta"], theta_unit="normalized",
                                 W=case["W"], state_out=out.state, rollback=out.rollback,
                                 target_argmax=out.target_argmax, entropy=out.entropy, row_flags=out.row_flags)
        torch.cuda.synchronize()
        return s
    s.update(logits=logits, draft=draft, target=_sample(logits, case["temperature"], seed) if case["sampled"] else None)
    if not case["static"]:
        s["fv"] = FlyVerify(B, K, V, case["dtype"])
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------

def _outputs(out):
    return {"accept_len": out.accept_len, "rollback": out.rollback, "out_tokens": out.out_tokens, "state": out.state,
            "target_argmax": out.target_argmax, "entropy": out.entropy, "row_flags": out.row_flags}


def run(s):
    case, stream = s["case"], s["stream"]
    kind = case["kind"]
    if kind == "pld":
        return binding.pld_draft(s["tokens"], s["lengths"], case["K"], case["max_ngram"], case["min_ngram"], stream=stream)
    out = s["out"]
    if kind == "fused":
        verify_fused(s["fv"], s["hidden"], s["weight"], s["draft"], out, theta=case["theta"], W=case["W"], stream=stream)
        return _outputs(out)
    if kind == "host":
        verify(s["fv"], s["logits"], s["draft"], out, theta=case["theta"], W=case["W"], stream=stream, host=True)
        return _outputs(out)
    if kind == "shard":
        mine = s["gathered"][0]
        s["fv"].reduce_shard(s["logits"], s["offset"], mine, stream)
        s["fv"].run_partials(s["args"], s["gathered"], case["world"], case["V"], stream)
        return dict(_outputs(out), partial=mine[:, :3], partial_argmax=mine.view(torch.int32)[:, 3])
    boundary = "carry" if case["carry"] else "reject"
    if s["target"] is None and not case["static"]:
        verify(s["fv"], s["logits"], s["draft"], out, theta=case["theta"], W=case["W"], theta_unit=case["unit"],
               boundary=boundary, stream=stream, temperature=case["temperature"], inputs_ready=case["ready"])
        return _outputs(out)
    # caller-sampled tokens and the entry point without a handle take the argument struct itself
    kw = dict(logits=s["logits"], theta=case["theta"], theta_unit=case["unit"], W=case["W"], boundary=boundary,
              state_in=out.state if case["carry"] else None, state_out=out.state, rollback=out.rollback,
              target_argmax=out.target_argmax, entropy=out.entropy, row_flags=out.row_flags,
              target_tokens=s["target"], temperature=case["temperature"], inputs_ready=case["ready"])
    B, K = case["B"], case["K"]
    if case["static"]:
        binding.run_static(binding.static_args(B, K, s["draft"], out.accept_len, out.out_tokens, **kw), case["V"],
                           case["dtype"], 0, stream)
    else:
        s["fv"].run(s["fv"].make_args(B, K, s["draft"], out.accept_len, out.out_tokens, **kw), stream)
    return _outputs(out)


# ---- what a pass cannot do without, and how exact it is -----------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "pld":
        # every token of every context (3/4 of L on average) once, the proposals out
        return {"bytes": case["B"] * (3 * case["L"] + 4 * case["K"] + 16), "flops": 0}
    B, K, V = case["B"], case["K"], case["V"]
    rows = B * (K + 1)
    small = 4 * B * K + 16 * rows + 32 * B        # drafts in; tokens, argmax, entropy, flags, lengths and state out
    if kind == "fused":
        return {"bytes": 2 * case["D"] * (V + rows) + small, "flops": 2 * rows * case["D"] * V}
    size = 4 if case["dtype"] == "f32" else 2
    if kind == "shard":
        return {"bytes": rows * (V // case["world"]) * size + 16 * rows * (case["world"] + 1) + small, "flops": 0}
    return {"bytes": rows * V * size + small + (4 * rows if case.get("sampled") else 0), "flops": 0}


def tolerance(case):
    if case["kind"] == "pld":
        return "exact"
    # measured against the same statistics in fp64: entropies off by at most 8e-8 (one value 5e-7) where the logits are
    # given and 2.6e-6 (one value 3.1e-6) where the tensor cores form them in fp32; about four times that.  An entropy that
    # lies that close to the threshold, or two fused logits that close to each other, may decide a round the other way.
    if case["kind"] == "fused":
        return {"rel": 1e-5, "max": 1.5e-5, "differ": 0.002}
    return {"rel": 4e-7, "max": 2e-6, "differ": 0.002}
