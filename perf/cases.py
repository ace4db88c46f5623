"""Performance cases of the stairs framework: what its users have it do, through the public entry
points, over the range of sizes it serves.

The models are the shapes of `paper_2407_19947_b200.workloads` (configs 1 to 4; config 5 is config
4's model with a long prefix), some at a reduced depth so that making the inputs stays quick.
Weights are random, but the language-model head carries a planted successor relation: after token t
the main model prefers succ(t) by a clear margin, as a trained model prefers its next token.  The
assistant of a generation agrees with it on about three quarters of the tokens, so that drafts are
kept or dropped in earnest and the tokens do not hang on the last bits of a logit.

A case is a dict of plain values:
  op        accept | validate | validate_host | prefill | draft | generate
  model     number of the config whose widths, vocabulary and weight type are used (1 is fp32, the
            others bf16); layers: depth of the main model
  assistant layers of the assistant (0: none); it has the main model's first layers (early exit)
            in configs 1 to 3 and layers of its own in config 4
  requests  requests of one call; prefix: tokens in the cache, of the longest request
  ragged    1: the requests' prefixes (down to half) and draft lengths (down by two) differ
  k         drafted tokens per request; page: tokens per K/V page; new: tokens generated
  adaptive  generate: 1 for the draft length that follows the acceptance
  vocab     accept: width of the logits
"""
import math

import numpy as np
import torch

from paper_2407_19947_b200 import stairs, workloads as wl

DEVICE = "cuda:0"
EMB_STD = 1.0          # embedding elements; the layers' outputs add up to about the same
AGREEMENT = 0.75       # share of the tokens after which the assistant agrees with the main model


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def _case(name=None, **kw):
    base = dict(op="validate", model=2, layers=24, assistant=0, requests=1, prefix=0, ragged=0, k=0, page=64,
                new=0, adaptive=0, vocab=0)
    if kw["op"] == "accept":
        base.update(model=0, layers=0)
    base.update(kw)
    return dict(base, name=name) if name else base


def listed():
    return [
        # a caller that holds logits already: one request's 5 rows over a Llama-sized vocabulary
        _case("accept, 5 rows", op="accept", requests=1, k=4, vocab=32000),
        # the same for a full serving batch: 64 requests of 9 rows, config 2's vocabulary
        _case("accept, 576 rows", op="accept", requests=64, k=8, vocab=32128),
        # config 1 (fp32): a whole short generation, where latency and launches are everything
        _case("generate tiny fp32", op="generate", model=1, layers=4, assistant=1, prefix=32, k=4, page=16, new=32),
        # config 2: the validation call of the benchmark's default run
        _case("validate 0.4B p2048 k8", op="validate", model=2, layers=24, prefix=2048, k=8),
        # config 3: the validation call through host buffers (drafts in, tokens out, every call)
        _case("validate_host 3B p512 k4", op="validate_host", model=3, layers=32, prefix=512, k=4),
        # config 4: one validation call of the 7B model
        _case("validate 7B p1024 k8", op="validate", model=4, layers=32, prefix=1024, k=8),
        # config 5 at a reduced depth: four requests with 16384 cached tokens each, 36 rows
        _case("validate 7B/4 4x16384 k8", op="validate", model=4, layers=4, requests=4, prefix=16384, k=8),
        # a serving batch: 16 requests of different lengths and draft lengths, more than 64 rows
        _case("validate 3B 16 requests", op="validate", model=3, layers=32, requests=16, prefix=300, ragged=1, k=6, page=16),
        # time to first token: config 2's prompt, and config 4's
        _case("prefill 0.4B 2048", op="prefill", model=2, layers=24, prefix=2048),
        _case("prefill 7B 1024", op="prefill", model=4, layers=32, prefix=1024),
        # the assistant's part of a step: config 4's two-layer assistant drafts 4 tokens
        _case("draft 7B assistant k4", op="draft", model=4, layers=4, assistant=2, prefix=512, k=4),
        # a whole generation: config 3 with its early-exit assistant
        _case("generate 3B 512+96 k4", op="generate", model=3, layers=32, assistant=4, prefix=512, k=4, new=96),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))


def draw(rng):
    op = rng.choice(["accept", "validate", "validate", "validate_host", "prefill", "prefill", "draft", "generate"])
    if op == "accept":
        k = rng.randint(0, 16)
        return _case(op=op, requests=_log_int(rng, 1, min(64, 576 // (k + 1))), k=k, vocab=_log_int(rng, 1000, 32128))
    page = rng.choice([16, 32, 64, 128])
    k = rng.randint(0, 8)
    if op == "draft":
        model = rng.choice([1, 2, 3, 4])
        return _case(op=op, model=model, layers=4, assistant=rng.randint(1, 4) if model != 1 else rng.randint(1, 2),
                     prefix=_log_int(rng, 3, 90 if model == 1 else 900), k=max(1, k), page=page)
    if op == "generate":
        model = rng.choice([1, 2, 3])
        layers = {1: 4, 2: rng.randint(6, 24), 3: rng.randint(4, 24)}[model]
        return _case(op=op, model=model, layers=layers, assistant=rng.randint(1, 2), prefix=_log_int(rng, 3, 60 if model == 1 else 512),
                     k=max(1, k), page=page, new=_log_int(rng, 8, 40 if model == 1 else 64), adaptive=rng.randint(0, 1))
    model = rng.choice([2, 3, 4] if op == "prefill" else [1, 2, 3, 4])
    layers = {1: 4, 2: rng.randint(6, 24), 3: rng.randint(4, 32), 4: rng.randint(2, 32)}[model]
    # (position limits of configs 1 to 3; the 7B shape goes further where it is shallow enough to prepare quickly)
    top = {1: 100, 2: 2048, 3: 960, 4: 16384 if layers <= 4 else 4096 if layers <= 8 else 1024}[model]
    if op == "prefill":
        top = min(top, 4096)
        return _case(op=op, model=model, layers=layers, prefix=_log_int(rng, 16, top), page=page)
    prefix = _log_int(rng, 8, top)
    most = max(1, min(16, 120 // (k + 1), 16384 * 4 // prefix if model == 4 else 4800 // prefix))
    return _case(op=op, model=model, layers=layers, requests=_log_int(rng, 1, most), prefix=prefix, ragged=rng.randint(0, 1), k=k, page=page)


# ------------------------------------------------------------------------------------------------
# weights, prompts, drafts
# ------------------------------------------------------------------------------------------------
def _successors(vocab, seed):
    """(main model's successor of every token, the assistant's)."""
    rng = np.random.default_rng(seed)
    main = rng.permutation(vocab)
    helper = main.copy()
    other = rng.permutation(vocab)[: int((1.0 - AGREEMENT) * vocab)]
    helper[other] = main[np.roll(other, 1)]
    return main.astype(np.int64), helper.astype(np.int64)


class _Weights(wl.WeightSource):
    """Weights of one model, made on the GPU."""

    def __init__(self, shape, seed, succ, depth, layers_of=None, globals_of=None):
        super().__init__(shape, seed, "torch-cuda", share_layers_with=layers_of, share_globals_with=globals_of)
        self.succ, self.depth = succ, depth

    def _draw(self, layer, name):
        shape = self.shape.tensor_shape(name)
        g = torch.Generator(device=DEVICE)
        k = self._key(layer, name)
        g.manual_seed((k[0] * 1_000_003 + k[1]) * 64 + k[2])
        if len(shape) == 1:   # gains near 1, biases near 0
            return torch.randn(shape, generator=g, device=DEVICE) * 0.05 + (0.0 if name.endswith("_b") else 1.0)
        std = 0.02
        if name in ("tok_emb", "pos_emb"):
            std = EMB_STD if name == "tok_emb" else 0.1
        elif name in ("wo", "w_down_or_fc2"):
            std = 0.02 / math.sqrt(2.0 * self.depth)
        dtype = torch.bfloat16 if self.shape.wdtype == wl.WDTYPE_BF16 else torch.float32
        return torch.empty(shape, dtype=dtype, device=DEVICE).normal_(0.0, std, generator=g)

    def torch_tensor(self, layer, name, device="cpu"):
        src, layer = self._resolve(layer, name) if name != "lm_head" else (self, layer)
        if not src.shape.has_tensor(name):
            return None
        key = f"{layer}:{name}"
        if key not in src._cache:
            if name == "lm_head":
                emb = self.torch_tensor(-1, "tok_emb", device)
                rho = min(1.0, 16.0 / math.sqrt(self.shape.d_model))
                t = src._draw(layer, name).mul_(math.sqrt(1.0 - rho * rho))
                # row succ(t) leans towards the embedding of t (rows that are nobody's successor stay noise)
                t.index_put_((torch.from_numpy(self.succ).to(DEVICE),), emb * (0.02 * rho / EMB_STD), accumulate=True)
            else:
                t = src._draw(layer, name)
            src._cache[key] = t.contiguous()
        return src._cache[key]


def _shapes(case):
    w = wl.workload(case["model"])
    main = w.target.replace(n_layers=case["layers"])
    if case["model"] == 4:
        main = main.replace(max_pos=16384 + 256)
    return w, main, main.replace(n_layers=case["assistant"]) if case["assistant"] else None


def _lengths(case):
    """Cached prefix and draft length of every request of a call."""
    n, p, k = case["requests"], case["prefix"], case["k"]
    if not case["ragged"]:
        return [p] * n, [k] * n
    return [p - (r * p) // (2 * n) for r in range(n)], [max(0, k - r % 3) for r in range(n)]


def prepare(case, seed):
    rng = np.random.default_rng([7, seed])
    if case["op"] == "accept":
        n, k, vocab = case["requests"], case["k"], case["vocab"]
        g = torch.Generator(device=DEVICE)
        g.manual_seed(seed)
        logits = torch.randn((n * (k + 1), vocab), generator=g, device=DEVICE)
        best = logits.argmax(dim=1).view(n, k + 1)[:, :k]
        keep = torch.rand((n, k), generator=g, device=DEVICE) < AGREEMENT
        draft = torch.where(keep, best, (best + 1) % vocab).to(torch.int32).contiguous()
        return {"case": case, "logits": logits, "k": [k] * n, "k_max": k, "draft": draft if k else None}
    w, main, helper = _shapes(case)
    succ, succ_h = _successors(main.vocab, seed)
    tsrc = _Weights(main, seed, succ, main.n_layers)
    dsrc = None
    if helper is not None:
        early = case["model"] != 4
        dsrc = _Weights(helper, seed + 1, succ_h, main.n_layers, layers_of=tsrc if early else None, globals_of=tsrc)
    prefixes, ks = _lengths(case)
    room = case["prefix"] + 1 + max(case["new"], case["k"] + 1) + 1
    eng = stairs.Stairs(tsrc, dsrc, max_requests=case["requests"], max_seq_len=room, k_max=case["k"], kv_page_tokens=case["page"])
    tokens = wl.uniform_tokens if w.prompt_dist == "uniform" else wl.zipf_tokens
    prompts = [tokens(p + 1, main.vocab, int(rng.integers(1 << 31))) for p in prefixes]
    st = {"case": case, "eng": eng, "prompts": prompts, "ks": ks, "reqs": list(range(case["requests"]))}
    if case["op"] in ("validate", "validate_host", "draft"):
        for r, p in enumerate(prompts):
            eng.prefill(r, p)
    if case["op"] in ("validate", "validate_host"):
        # drafts that follow the main model for a while and then leave it
        draft = rng.integers(0, main.vocab, size=(case["requests"], max(case["k"], 1))).astype(np.int32)
        for r, p in enumerate(prompts):
            t = int(p[-1])
            for j in range(int(rng.integers(0, ks[r] + 1))):
                t = int(succ[t])
                draft[r, j] = t
        st["draft"] = torch.from_numpy(draft).to(DEVICE) if case["op"] == "validate" else draft
    eng.sync()
    return st


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "accept":
        return stairs.accept_static(st["logits"], st["k"], st["draft"], st["k_max"])
    eng = st["eng"]
    if op == "validate":
        return eng.validate(st["reqs"], st["ks"], st["draft"], want_logits=True)
    if op == "validate_host":
        return eng.validate_host(st["reqs"], st["ks"], st["draft"] if case["k"] else None)
    if op == "prefill":      # the prompt, then the first token and its scores
        eng.prefill(0, st["prompts"][0])
        return eng.validate([0], [0], None, want_logits=True)
    if op == "draft":
        return eng.draft(0, case["k"])
    out, stats = eng.generate(0, st["prompts"][0], case["k"], case["new"], adaptive=bool(case["adaptive"]))
    return np.asarray(out, np.int32), [stats[n] for n in ("iterations", "drafted", "accepted", "emitted")]


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far apart two correct results may be
# ------------------------------------------------------------------------------------------------
def _layer_params(shape):
    es = 4 if shape.wdtype == wl.WDTYPE_F32 else 2
    return shape.weight_bytes_per_call() // es - shape.vocab * shape.d_model


def _forward(shape, prefixes, rows, logits, head=True):
    """Bytes and operations of one pass of `rows[i]` new positions after prefixes[i] cached ones."""
    es = 4 if shape.wdtype == wl.WDTYPE_F32 else 2
    n, head_params = sum(rows), shape.vocab * shape.d_model if head else 0
    kv = shape.kv_bytes_per_token()
    b = es * (_layer_params(shape) + head_params) + kv * sum(p + r for p, r in zip(prefixes, rows)) + n * shape.d_model * es
    f = 2.0 * n * (_layer_params(shape) + head_params)
    f += sum(4.0 * shape.n_layers * shape.n_heads * shape.head_dim * (r * p + r * (r + 1) / 2.0) for p, r in zip(prefixes, rows))
    return b + (4 * n * shape.vocab if logits else 0), f


def work(case):
    op, k = case["op"], case["k"]
    if op == "accept":
        rows = case["requests"] * (k + 1)
        return {"bytes": 4 * rows * (case["vocab"] + 2), "flops": rows * case["vocab"]}
    _, main, helper = _shapes(case)
    prefixes, ks = _lengths(case)
    p = case["prefix"]
    total = [0.0, 0.0]

    def add(bf, times=1.0):
        total[0] += times * bf[0]
        total[1] += times * bf[1]

    if op in ("validate", "validate_host"):
        add(_forward(main, prefixes, [x + 1 for x in ks], op == "validate"))
    elif op == "draft":
        add(_forward(helper, [p], [1], False), k)
    else:
        # (an early-exit assistant finds the prompt in the main model's cache; the last prompt token comes with the first call)
        add(_forward(main, [0], [p], False, head=False))
        if op == "prefill":
            add(_forward(main, [p], [1], True))
        else:
            # passes of a generation whose drafts are kept with probability AGREEMENT each
            per_pass = sum(AGREEMENT ** j for j in range(k + 1))
            passes = case["new"] / per_pass
            add(_forward(main, [p], [k + 1], False), passes)
            add(_forward(helper, [p], [1], False), passes * k)
    return {"bytes": total[0], "flops": total[1]}


def tolerance(case):
    if case["op"] in ("validate", "prefill"):
        # scores: sums of 32-bit floats in another order, or of bf16 operands and an fp16 cache
        return {"rel": 1e-5, "max": 2e-4} if case["model"] == 1 else {"rel": 1e-2, "max": 1e-1}
    return "exact"   # token ids and counts
