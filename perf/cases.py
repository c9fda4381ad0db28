"""The work this library is measured on: denoising steps, cached steps, whole generations and the sampling epilogue, called
the way a decoding program calls them, from the two-layer test model up to a batch of eight at the 8B width.

Shapes are those of the package's own workloads (`workloads.TINY`, `workloads.LLADA_8B`, the benchmark's prompt / response
lengths) and sizes between them.  Some cases cut the 8B shape to fewer layers: every layer runs the same kernels on the same
sizes, and bf16 rounding noise, which grows with depth, stays well inside the tolerance."""
import math

import torch

from paper_2506_10848_b200 import binding as sfs
from paper_2506_10848_b200 import workloads as W

DEV = "cuda"
FULL_DEPTH = W.LLADA_8B.n_layers


# ---- the cases ------------------------------------------------------------------------------------------------------

def _forward(name, model, layers, batch, prompt, gen, done, rows, dtype="bf16"):
    """One uncached denoising step's predictor: positions before `done` are decoded, logits are asked for the next `rows`."""
    return dict(name=name, kind="forward", model=model, layers=layers, batch=batch, prompt=prompt, gen=gen, done=done, rows=rows, dtype=dtype)


def _cached(name, model, layers, batch, prompt, gen, done, steps, k_prompt, k_response, rho=0.25, span=0):
    """The first `steps` steps of a cached generation, one more token decoded per step; `span` > 0: the partial steps are
    accelerated ones with a span of that many positions."""
    return dict(name=name, kind="cached", model=model, layers=layers, batch=batch, prompt=prompt, gen=gen, done=done, steps=steps,
                k_prompt=k_prompt, k_response=k_response, rho=rho, span=span)


def _generate(name, model, layers, batch, prompt, gen, sampler="slowfast", max_steps=0):
    """A whole sfs_generate call; predictions are as confident as a trained model's (see _fit_head)."""
    return dict(name=name, kind="generate", model=model, layers=layers, batch=batch, prompt=prompt, gen=gen, sampler=sampler,
                max_steps=max_steps)


def _select(name, vocab, batch, prompt, gen, done, rows, phase, dtype="bf16", sampler="slowfast"):
    """The sampling epilogue and transition rule on given logits (a program with its own predictor)."""
    return dict(name=name, kind="select", vocab=vocab, batch=batch, prompt=prompt, gen=gen, done=done, rows=rows, phase=phase,
                dtype=dtype, sampler=sampler)


def _row_stats(name, vocab, rows, dtype="bf16"):
    """Argmax, canonical denominator and confidence of every row."""
    return dict(name=name, kind="row_stats", vocab=vocab, rows=rows, dtype=dtype)


def listed():
    return [
        # the smallest model and sequence: what a step costs when launches and latency are all of it
        _forward("forward_tiny", "tiny", 2, 1, 32, 32, 0, 32),
        # a chat-sized prompt and a short answer at full depth: the weights stream through for a hundred rows
        _forward("forward_short", "8b", FULL_DEPTH, 1, 40, 64, 0, 64),
        # the benchmark's step: 256 + 256, every response row masked
        _forward("forward_256_256", "8b", FULL_DEPTH, 1, 256, 256, 0, 256),
        # an accelerated step late in a long answer: odd lengths, logits of a short span only, fp32 for a sampler of one's own
        _forward("forward_span_f32", "8b", 8, 1, 693, 307, 211, 29, "f32"),
        # the long response
        _forward("forward_1024_1024", "8b", 8, 1, 1024, 1024, 0, 1024),
        # a serving batch
        _forward("forward_batch8", "8b", 8, 8, 512, 256, 0, 256),
        # the paper's cached setting (K_p = 100, K_r = 5), half of the answer decoded: full refresh, four partial steps, response
        # refresh
        _cached("cached_1024_512", "8b", 4, 1, 1024, 512, 256, 6, 100, 5),
        # whole SlowFast generations: a small one (host and launch latency per step), and one at the 8B width
        _generate("generate_tiny", "tiny", 2, 2, 160, 64),
        _generate("generate_8b_width", "8b", 8, 1, 512, 256),
        # the epilogue microbenchmark: all rows of a 256-token response, exploratory step
        _select("select_slow_256", W.LLADA_8B.vocab, 1, 256, 256, 0, 256, "slow"),
        # fp32 logits of an odd vocabulary from another predictor, two sequences, accelerated step
        _select("select_fast_f32", 50257, 2, 19, 96, 13, 61, "fast", "f32"),
        # confidences of every row for a ranking of one's own
        _row_stats("row_stats_64", W.LLADA_8B.vocab, 64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _to8(prompt, gen):
    """The nearest prompt length that makes the sequence a multiple of eight tokens."""
    return max(1, prompt + (-(prompt + gen)) % 8)


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "cached", "generate", "select", "select", "row_stats"])
    if kind == "forward":
        model = rng.choice(["tiny", "8b", "8b", "8b"])
        batch = rng.choice([1, 1, 1, 2, 3, 5, 8])
        gen = _log(rng, 24, 1024 if batch == 1 else 320)
        prompt = _to8(_log(rng, 16, 1024 if batch == 1 else 512), gen)
        done = rng.choice([0, rng.randrange(gen // 2)])
        rows = rng.choice([gen - done, _log(rng, 1, gen - done)])
        c = _forward("", model, 2 if model == "tiny" else rng.randint(2, 8), batch, prompt, gen, done, rows, rng.choice(["bf16", "bf16", "f32"]))
    elif kind == "cached":
        batch = rng.choice([1, 1, 2])
        gen = _log(rng, 48, 768 if batch == 1 else 256)
        prompt = _to8(_log(rng, 48, 1024 if batch == 1 else 512), gen)
        steps = rng.randint(4, 7)
        k_p, k_r = rng.choice([(100, 5), (500, 30), (4, 2)])
        c = _cached("", "8b", rng.randint(2, 4), batch, prompt, gen, rng.randrange(gen // 3), steps, k_p, k_r, rng.choice([0.25, 0.25, 0.1]),
                    rng.choice([0, 0, gen // 3]))
    elif kind == "generate":
        model = rng.choice(["tiny", "8b"])
        batch = rng.choice([1, 1, 2]) if model == "tiny" else 1
        gen = _log(rng, 24, 96) if model == "tiny" else _log(rng, 32, 256)
        prompt = _to8(2 * gen + rng.randrange(256), gen)
        sampler = rng.choice(["slowfast", "slowfast", "random"]) if model == "8b" else "slowfast"
        c = _generate("", model, 2 if model == "tiny" else rng.randint(2, 8), batch, prompt, gen, sampler, rng.choice([4, 8]) if sampler == "random" else 0)
    elif kind == "select":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        vocab = rng.choice([W.LLADA_8B.vocab, W.LLADA_8B.vocab, 50257, 32000, _log(rng, 4000, 130000)])
        batch = rng.choice([1, 1, 2, 4, 8])
        gen = _log(rng, 24, 512 if batch == 1 else 256)
        done = rng.choice([0, rng.randrange(gen // 2)])
        rows = rng.choice([gen - done, _log(rng, 2, gen - done)])
        phase = "slow" if rows == gen - done and rng.random() < 0.5 else "fast"
        c = _select("", vocab, batch, rng.randint(8, 512), gen, done, rows, phase, dtype)
    else:
        vocab = rng.choice([W.LLADA_8B.vocab, W.LLADA_8B.vocab, 50257, 32000, _log(rng, 4000, 130000)])
        c = _row_stats("", vocab, _log(rng, 4, 768), rng.choice(["bf16", "bf16", "f32"]))
    del c["name"]
    return c


# ---- inputs ---------------------------------------------------------------------------------------------------------

class _Engine:
    """A model with its weights and one session; gives the library's memory back when the program drops it."""

    def __init__(self, case, seed, peak=1.0):
        shape = W.TINY if case["model"] == "tiny" else W.with_layers(W.LLADA_8B, case["layers"])
        self.shape, self.session = shape, None
        weights = W.model_weights(shape, seed, device=DEV)
        for layer in weights["layers"]:
            layer["wq"].mul_(peak)
            layer["wk"].mul_(peak)
        self.model = sfs.Model(shape, weights)
        self.session = sfs.sfs_session_create(self.model, case["batch"], case["prompt"] + case["gen"])

    def __del__(self):
        if self.session is not None and sfs is not None:
            sfs.sfs_session_destroy(self.session)
            self.session = None
            self.model.close()


class _Selector:
    def __init__(self, vocab, batch, length):
        self.session = sfs.sfs_select_session_create(vocab, batch, length)

    def __del__(self):
        if getattr(self, "session", None) is not None and sfs is not None:
            sfs.sfs_session_destroy(self.session)
            self.session = None


def _rng(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _tokens(case, shape, seed):
    """(all tokens decoded, the same with every response position masked)."""
    B, P, L = case["batch"], case["prompt"], case["gen"]
    full = torch.randint(0, shape.vocab - 2, (B, P + L), generator=_rng(seed, 1), device=DEV, dtype=torch.int32)
    masked = full.clone()
    masked[:, P:] = shape.mask_id
    return full, masked


def _masked_from(full, masked, P, done):
    t = masked.clone()
    t[:, P:P + done] = full[:, P:P + done]
    return t


def _row_list(B, S, first, count):
    r = torch.arange(count, device=DEV, dtype=torch.int32)[None, :] + first
    return (r + S * torch.arange(B, device=DEV, dtype=torch.int32)[:, None]).reshape(-1).contiguous()


def _prepare_forward(case, seed):
    e = _Engine(case, seed)
    B, P, L = case["batch"], case["prompt"], case["gen"]
    full, masked = _tokens(case, e.shape, seed)
    n = B * case["rows"]
    rows = torch.zeros(B * L, device=DEV, dtype=torch.int32)
    rows[:n] = _row_list(B, P + L, P + case["done"], case["rows"])
    f32 = case["dtype"] == "f32"
    return dict(kind="forward", engine=e, B=B, S=P + L, tokens=_masked_from(full, masked, P, case["done"]), rows=rows, n=n,
                n_rows=torch.tensor([n], device=DEV, dtype=torch.int32), max_rows=B * L, dtype=sfs.LOGITS_F32 if f32 else sfs.LOGITS_BF16,
                logits=torch.zeros((B * L, e.shape.vocab), device=DEV, dtype=torch.float32 if f32 else torch.bfloat16))


def _prepare_cached(case, seed):
    e = _Engine(case, seed)
    sfs.sfs_cache_enable(e.session, case["k_prompt"], case["k_response"], case["rho"])
    B, P, L = case["batch"], case["prompt"], case["gen"]
    full, masked = _tokens(case, e.shape, seed)
    steps = []
    for t in range(case["steps"]):
        done = case["done"] + t
        count = min(case["span"], L - done) if case["span"] and t else L - done
        state = None
        if case["span"] and t:
            state = torch.zeros((B, sfs.STATE_INTS), device=DEV, dtype=torch.int32)
            state[:, sfs.STATE_FIELDS.index("phase")] = sfs.PHASE_FAST
            state[:, sfs.STATE_FIELDS.index("s_cycle")] = done
            state[:, sfs.STATE_FIELDS.index("hi")] = done + count
        n = B * count
        rows = torch.zeros(B * L, device=DEV, dtype=torch.int32)
        rows[:n] = _row_list(B, P + L, P + done, count)
        steps.append(dict(tokens=_masked_from(full, masked, P, done), state=state, rows=rows, n=n,
                          n_rows=torch.tensor([n], device=DEV, dtype=torch.int32),
                          logits=torch.zeros((B * L, e.shape.vocab), device=DEV, dtype=torch.bfloat16)))
    return dict(kind="cached", engine=e, B=B, P=P, S=P + L, max_rows=B * L, steps=steps)


SAMPLERS = {"slowfast": sfs.SAMPLER_SLOWFAST, "low_confidence": sfs.SAMPLER_LOW_CONFIDENCE, "random": sfs.SAMPLER_RANDOM}


def _fit_head(engine, prompt, B, P, L, seed):
    """Random weights predict nothing in particular: one near-tie decides for all positions at once.  A trained model tells its
    positions apart, so the head's rows of L distinct tokens are fitted to the hidden states of the fully masked response."""
    shape, head = engine.shape, engine.model.weights["lm_head"]
    d = shape.d_model
    keep = head[:d].clone()
    head[:d] = torch.eye(d, device=DEV, dtype=head.dtype)           # now the logits are the hidden states
    tokens = torch.cat([prompt, torch.full((B, L), shape.mask_id, device=DEV, dtype=torch.int32)], dim=1)
    rows = _row_list(B, P + L, P, L)
    out = torch.empty((B * L, shape.vocab), device=DEV, dtype=torch.float32)
    sfs.sfs_forward(engine.session, tokens, B, P + L, rows, None, B * L, out, sfs.LOGITS_F32)
    h = out[:, :d].clone() / shape.logit_scale
    head[:d] = keep
    mean = h.mean(dim=0, keepdim=True)
    mean = mean / mean.norm()
    apart = h - (h @ mean.t()) * mean
    proto = apart / apart.norm(dim=1, keepdim=True)
    score = apart @ proto.t()
    rival = (score - 1e30 * torch.eye(B * L, device=DEV)).amax(dim=1)
    gain = CONFIDENT / (score.diagonal() - rival).median() / shape.logit_scale
    ids = torch.randperm(shape.vocab - 2, generator=_rng(seed, 5), device=DEV)[:B * L]
    head[ids] = (gain * proto).to(head.dtype)


CONFIDENT = 30.0        # the fitted head's median margin over the runner-up, in logits
PEAK = 8.0              # W_q and W_k of the narrow model: attention as peaked as it is at the 8B width, where positions differ


def _prepare_generate(case, seed):
    e = _Engine(case, seed, PEAK if case["model"] == "tiny" else 1.0)
    B, P, L = case["batch"], case["prompt"], case["gen"]
    full, _ = _tokens(case, e.shape, seed)
    prompt = full[:, :P].contiguous()
    _fit_head(e, prompt, B, P, L, seed)
    return dict(kind="generate", engine=e, B=B, P=P, L=L, prompt=prompt,
                params=sfs.Params.default(sampler=SAMPLERS[case["sampler"]], max_steps=case["max_steps"], seed=seed),
                out=torch.zeros((B, P + L), device=DEV, dtype=torch.int32))


def _logits(rows, vocab, seed, dtype):
    """N(0, 4^2) noise and one planted winner per row, U(0, 12) above the noise maximum: confidences from 0.2 to 1."""
    g = _rng(seed, 3)
    x = torch.randn((rows, vocab), generator=g, device=DEV, dtype=torch.float32).mul_(4.0)
    col = torch.randint(0, vocab, (rows, 1), generator=g, device=DEV)
    x.scatter_(1, col, x.amax(dim=1, keepdim=True) + 12.0 * torch.rand((rows, 1), generator=g, device=DEV))
    return x if dtype == "f32" else x.to(torch.bfloat16)


def _prepare_select(case, seed):
    B, P, L, V = case["batch"], case["prompt"], case["gen"], case["vocab"]
    S, done, count = P + L, case["done"], case["rows"]
    params = sfs.Params.default(sampler=SAMPLERS[case["sampler"]])
    # tokens, mask and scheduler state in one buffer: a step updates them in place, a pass starts from the same ones
    nt, nm, ns = 4 * B * S, (B * S + 15) // 16 * 16, 4 * B * sfs.STATE_INTS
    begin = torch.zeros(nt + nm + ns, device=DEV, dtype=torch.uint8)

    def views(buf):
        return (buf[:nt].view(torch.int32).view(B, S), buf[nt:nt + B * S].view(B, S), buf[nt + nm:].view(torch.int32).view(B, sfs.STATE_INTS))

    tok, mask, state = views(begin)
    full = torch.randint(0, V - 2, (B, S), generator=_rng(seed, 1), device=DEV, dtype=torch.int32)
    tok.copy_(full)
    tok[:, P + done:] = V - 1
    mask[:, P + done:] = 1
    fields = {"phase": sfs.PHASE_FAST if case["phase"] == "fast" else sfs.PHASE_SLOW, "s_cycle": done, "hi": done + count if case["phase"] == "fast" else 0,
              "k_remaining": L - done, "n_masked": L - done, "steps_done": done}
    for k, v in fields.items():
        state[:, sfs.STATE_FIELDS.index(k)] = v
    work = begin.clone()
    tok_w, mask_w, state_w = views(work)
    new = lambda *shape: torch.full(shape, -1, device=DEV, dtype=torch.int32)  # noqa: E731
    n = B * count
    return dict(kind="select", selector=_Selector(V, B, S), B=B, S=S, P=P, V=V, params=params, begin=begin, work=work, tokens=tok_w, mask=mask_w,
                state=state_w, logits=_logits(n, V, seed, case["dtype"]), dtype=sfs.LOGITS_F32 if case["dtype"] == "f32" else sfs.LOGITS_BF16,
                rows=_row_list(B, S, P + done, count), n=n, sel_count=new(B), sel_pos=new(B, L), sel_tok=new(B, L), next_rows=new(B * L), next_n=new(1))


def _prepare_row_stats(case, seed):
    n = case["rows"]
    return dict(kind="row_stats", logits=_logits(n, case["vocab"], seed, case["dtype"]), V=case["vocab"], n=n,
                dtype=sfs.LOGITS_F32 if case["dtype"] == "f32" else sfs.LOGITS_BF16, argmax=torch.zeros(n, device=DEV, dtype=torch.int32),
                sq=torch.zeros(n, device=DEV, dtype=torch.int64), conf=torch.zeros(n, device=DEV, dtype=torch.float32))


def prepare(case, seed):
    return {"forward": _prepare_forward, "cached": _prepare_cached, "generate": _prepare_generate, "select": _prepare_select,
            "row_stats": _prepare_row_stats}[case["kind"]](case, seed)


# ---- one pass -------------------------------------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "forward":
        sfs.sfs_forward(s["engine"].session, s["tokens"], s["B"], s["S"], s["rows"], s["n_rows"], s["max_rows"], s["logits"], s["dtype"])
        return s["logits"][:s["n"]]
    if kind == "cached":
        session = s["engine"].session
        sfs.sfs_cache_reset(session)
        for t in s["steps"]:
            sfs.sfs_forward_cached(session, t["tokens"], s["B"], s["S"], s["P"], t["state"], t["rows"], t["n_rows"], s["max_rows"], t["logits"],
                                   sfs.LOGITS_BF16)
        return [t["logits"][:t["n"]] for t in s["steps"]]
    if kind == "generate":
        sfs.sfs_generate(s["engine"].session, s["prompt"], s["B"], s["P"], s["L"], s["params"], s["out"])
        return s["out"]
    if kind == "select":
        s["work"].copy_(s["begin"])
        sfs.sfs_select(s["selector"].session, s["logits"], s["dtype"], s["V"], s["rows"], None, s["n"], s["tokens"], s["mask"], s["B"], s["S"], s["P"],
                       s["state"], s["params"], s["sel_count"], s["sel_pos"], s["sel_tok"], s["next_rows"], s["next_n"])
        return {k: s[k] for k in ("tokens", "mask", "state", "sel_count", "sel_pos", "sel_tok", "next_rows", "next_n")}
    sfs.sfs_row_stats(s["logits"], s["dtype"], s["V"], s["V"], None, s["n"], s["argmax"], s["sq"], s["conf"])
    return {k: s[k] for k in ("argmax", "sq", "conf")}


# ---- what a pass cannot do without ----------------------------------------------------------------------------------

def _step_work(shape, B, S, q, kv, rows, logit_bytes):
    """Bytes and FLOPs of one step that computes `q` query tokens per sequence against `kv` keys and `rows` logits rows."""
    d, ff, V, nl = shape.d_model, shape.d_ff, shape.vocab, shape.n_layers
    weights = 2.0 * (nl * (4 * d * d + 3 * d * ff + 2 * d) + V * d + d)
    flops = nl * (2.0 * B * q * (4 * d * d + 3 * d * ff) + 4.0 * B * q * kv * d) + 2.0 * rows * d * V
    return weights + 2.0 * min(B * S, V) * d + 4.0 * B * S + 4.0 * rows + float(logit_bytes) * rows * V, flops


def work(case):
    kind = case["kind"]
    if kind in ("select", "row_stats"):
        n = case["rows"] * case.get("batch", 1)
        extra = case["batch"] * (2 * (5 * (case["prompt"] + case["gen"]) + 128) + 12 * case["gen"]) if kind == "select" else 16 * n
        return {"bytes": float(n) * case["vocab"] * (4 if case["dtype"] == "f32" else 2) + extra, "flops": 4.0 * n * case["vocab"]}
    shape = W.TINY if case["model"] == "tiny" else W.with_layers(W.LLADA_8B, case["layers"])
    B, P, L = case["batch"], case["prompt"], case["gen"]
    S = P + L
    if kind == "forward":
        b, f = _step_work(shape, B, S, S, S, B * case["rows"], 4 if case["dtype"] == "f32" else 2)
        return {"bytes": b, "flops": f}
    if kind == "generate":
        # SlowFast: two exploratory steps and one accelerated step are the fewest that decode everything
        n = case["max_steps"] if case["sampler"] == "random" else 3
        steps = [_step_work(shape, B, S, S, S, B * (L * (n - t) // n if case["sampler"] == "random" else L - t), 0) for t in range(n)]
        return {"bytes": sum(b for b, _ in steps), "flops": sum(f for _, f in steps)}
    tot_b = tot_f = 0.0
    for t in range(case["steps"]):
        done = case["done"] + t
        rows = min(case["span"], L - done) if case["span"] and t else L - done
        q = (P if t % case["k_prompt"] == 0 else 0) + (L if t % case["k_response"] == 0 else math.ceil(case["rho"] * L))
        b, f = _step_work(shape, B, S, q, S, B * rows, 2)
        if t % case["k_response"]:
            f += shape.n_layers * 2.0 * B * L * shape.d_model ** 2      # fresh values of the candidates
        tot_b, tot_f = tot_b + b, tot_f + f
    return {"bytes": tot_b, "flops": tot_f}


def tolerance(case):
    """Measured with the same model under a permutation of its hidden dimensions, i.e. with every sum in another order: a bf16
    rounding that flips in one layer moves the next, so the distance grows with depth."""
    if case["kind"] in ("select", "row_stats"):
        return "exact"                      # decisions are taken on integers that do not depend on the order of summation
    if case["kind"] == "generate":
        return {"rel": 0.0, "differ": 0.01}             # tokens; measured: 0, at most 0.0067 with one near-tie in the narrow model
    if case["model"] == "tiny":
        return {"rel": 0.01}                            # measured: 1.3e-3 to 2.6e-3
    return {"rel": 0.03}        # measured: 7e-3 to 1.2e-2 for 2 to 8 layers, 1.4e-2 for 32, 2.2e-2 where nearly tied rows are recomputed
