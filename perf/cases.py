"""The calls a serving program makes of this library, as cases that can be timed.

Every case is made of the public entry points (`SuffixStore` and its methods) on seeded text:

  draft    one `speculate` for a batch whose requests are in the store: the cost of a draft alone
  decode   a batch from its prompts to the end of its outputs: `build_requests`, then one `step`
           (append the accepted tokens + draft) per decode step
  refill   a few new requests enter a running batch: `build_requests` and their first draft
  serve    a service from its start: `SuffixStore` from a corpus, the first prompts, then decode
           steps in the two-call form (`speculate`, `append`) in which requests finish, their
           outputs go into the global tree and new requests take their slots
  build    offline: `SuffixStore` from a corpus, then n-gram counts looked up in it
  entropy  offline: `entropy` of a store's global tree (does speculation pay on this text?)

The text follows workload/generator.py's model, made on the GPU: a text is a series of events, each
a span copied from earlier text (probability `copy`, geometric length of mean `span`) or a fresh
Zipf(1.1) token.  `corpus_share` (when above 0): that share of a prompt's events copies from the
corpus, the others only from the prompt itself.
"""
import math

import numpy as np
import torch

import paper_2411_04975_b200 as sfx

SEQ = 1024                 # tokens of a corpus sequence
ZIPF = 1.1
HEAD = 1024                # fresh tokens at the start of a corpus
MEAN_EXTRA, MAX_ACCEPT = 3.0, 16   # accepted tokens per step: 1 + geometric of that mean, at most that many

LARGE = dict(vocab=128256, corpus=4096 * SEQ, copy=0.7, span=32.0, corpus_share=0.0, depth=32, P=32, alpha=2.0,
             max_spec=64, flags=0, tau=0.0)
AGENTIC = dict(LARGE, vocab=32000, corpus=4000 * SEQ, copy=0.8, span=48.0, corpus_share=0.5, P=24)
LOW = dict(LARGE, copy=0.15, span=8.0)
TINY = dict(LARGE, vocab=32000, corpus=64 * 512, P=16, alpha=1.0, max_spec=32)


def listed():
    return [
        # one user's draft in a small deployment: launch and latency are all of it
        dict(TINY, name="draft_1", kind="draft", batch=1, prompt=256),
        # the headline batch: 256 requests with 4,096-token prompts
        dict(LARGE, name="draft_256", kind="draft", batch=256, prompt=4096),
        # one agent with a long context, token after token
        dict(AGENTIC, name="decode_1_agentic", kind="decode", batch=1, prompt=8192, steps=64),
        # 64 agents: long repetitive contexts
        dict(AGENTIC, name="decode_64_agentic", kind="decode", batch=64, prompt=8192, steps=48),
        # the headline batch, prompts to outputs of about 256 tokens
        dict(LARGE, name="decode_256", kind="decode", batch=256, prompt=4096, steps=64),
        # open-ended chat, little repetition, more requests than two per SM
        dict(LOW, name="decode_512_low_repetition", kind="decode", batch=512, prompt=4096, steps=32),
        # four requests finished: four new ones enter the running batch of 256
        dict(LARGE, name="refill_4", kind="refill", batch=256, new=4, prompt=4096),
        # a small service from its start
        dict(TINY, name="serve_16_small", kind="serve", batch=16, prompt=256, steps=32, out_lo=32, out_hi=128),
        # the headline batch as a service, with a corpus of half a million tokens at its start
        dict(LARGE, name="serve_256", kind="serve", batch=256, corpus=512 * SEQ, prompt=4096, steps=64, out_lo=128,
             out_hi=512),
        # the smallest and the headline corpus, built offline
        dict(TINY, name="build_32k", kind="build", queries=1024),
        dict(LARGE, name="build_4m", kind="build", queries=65536),
        # what the headline corpus's tree says about its predictability
        dict(LARGE, name="entropy_4m", kind="entropy"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    base = rng.choice([LARGE, AGENTIC, LOW, TINY])
    case = dict(base, kind=rng.choice(["draft", "decode", "decode", "refill", "serve", "build", "entropy"]))
    case["vocab"] = log(8000, 151000)
    case["corpus"] = log(30000, 4 << 20)
    case["depth"] = rng.choice([32, 32, 24, 17])
    case["P"] = rng.randint(8, 32)
    case["alpha"] = rng.choice([1.0, 1.5, 2.0, 4.0])
    case["max_spec"] = rng.choice([16, 32, 48, 64, 64])
    case["flags"] = rng.choice([0, 0, 0, 0, sfx.FLAG_LINEAR, sfx.FLAG_GLOBAL_ONLY, sfx.FLAG_REQUEST_ONLY])
    case["tau"] = rng.choice([0.0, 0.0, 2.0])
    kind = case["kind"]
    if kind in ("draft", "decode", "refill", "serve"):
        case["prompt"] = log(200, 8192)
        most = min(512, (4 << 20) // 2 // case["prompt"])      # the prompts of a batch hold at most two million tokens
        case["batch"] = log(1, most)
    if kind == "decode":
        case["steps"] = rng.randint(8, 64)
    if kind == "refill":
        case["new"] = rng.randint(1, min(8, case["batch"]))
    if kind == "serve":
        case["corpus"] = log(30000, 1 << 19)
        case["batch"] = min(case["batch"], 256)
        case["steps"] = rng.randint(8, 48)
        case["out_lo"] = log(16, 128)
        case["out_hi"] = case["out_lo"] * rng.randint(2, 4)
    if kind == "build":
        case["queries"] = log(256, 65536)
    return case


# ------------------------------------------------------------------------------------------ text
class _Text:
    """Seeded text on the GPU."""

    def __init__(self, case, seed):
        self.c, self.dev = case, torch.device("cuda", torch.cuda.current_device())
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(seed)
        w = torch.arange(1, case["vocab"] + 1, device=self.dev, dtype=torch.float64) ** (-ZIPF)
        self.cdf = torch.cumsum(w, 0)
        self.cdf /= self.cdf[-1].clone()
        self.perm = torch.randperm(case["vocab"], device=self.dev, generator=self.g)

    def _rand(self, *shape):
        return torch.rand(*shape, device=self.dev, dtype=torch.float64, generator=self.g)

    def _fresh(self, u):
        return self.perm[torch.searchsorted(self.cdf, u).clamp_(max=self.c["vocab"] - 1)]

    def _spans(self, u):
        mean = self.c["span"]
        return (torch.log1p(-u) / math.log(1.0 - 1.0 / mean)).floor_().to(torch.int64) + 1

    def corpus(self):
        """int32[corpus].  Its head is fresh throughout: a text that copied from its first word on would be that word."""
        n = self.c["corpus"]
        head = self._fresh(self._rand(min(n, HEAD)))
        if n <= HEAD:
            return head.to(torch.int32)
        rest = self._write(1, n - HEAD, head, 0.0)
        return torch.cat([head, rest.reshape(-1)]).to(torch.int32)

    def texts(self, n, length, corpus):
        """int32[n][length]: texts that copy from the corpus and from themselves."""
        return self._write(n, length, corpus.to(torch.int64), self.c["corpus_share"]).to(torch.int32)

    def _write(self, n, length, pool, pool_share):
        """int64[n][length].  An event copies from `pool` and the text's own earlier part as one."""
        kind, where = self._rand(n, length), self._rand(n, length)
        spans = self._spans(self._rand(n, length))
        copies = kind < (self.c["copy"] if pool_share == 0.0 else pool_share + (1.0 - pool_share) * self.c["copy"])
        size = torch.where(copies, spans, 1)
        start = torch.cumsum(size, 1) - size                    # of every event; those behind the end do not count
        mark = torch.zeros(n, length + 1, device=self.dev, dtype=torch.int64)
        mark.scatter_(1, start.clamp(max=length), 1)
        event = torch.cumsum(mark[:, :length], 1) - 1           # of every token
        at = torch.gather(start, 1, event)                      # start of the token's event
        off = torch.arange(length, device=self.dev)[None, :] - at
        kind, where, copies = torch.gather(kind, 1, event), torch.gather(where, 1, event), torch.gather(copies, 1, event)
        have = pool.numel()
        if pool_share > 0.0:
            src = torch.where(kind < pool_share, (where * have).to(torch.int64),
                              have + (where * at).to(torch.int64))
            copies &= (kind < pool_share) | (at > 0)
        else:
            src = (where * (have + at)).to(torch.int64)
        own = src >= have
        row = torch.arange(n, device=self.dev)[:, None] * length
        # a span that runs into its own event goes on from the span's start again
        own_src = row + (src - have) + off % (at - (src - have)).clamp(min=1)
        here = row + torch.arange(length, device=self.dev)[None, :]
        text = torch.where(copies & ~own, pool[(src + off) % have],
                           self._fresh(self._rand(n, length)))
        link = torch.where(copies & own, own_src, here).reshape(-1)
        for _ in range(max(1, length.bit_length())):            # copies of copies
            link = link[link]
        return text.reshape(-1)[link].reshape(n, length)


def _accepted(rng, shape):
    p = 1.0 / (MEAN_EXTRA + 1.0)
    extra = np.floor(np.log1p(-rng.random(shape)) / math.log(1.0 - p)).astype(np.int64)
    return 1 + np.minimum(extra, MAX_ACCEPT - 1)


def _ragged(rng, n, longest):
    """Prompt lengths between half the longest and the longest."""
    return rng.integers((longest + 1) // 2, longest + 1, n)


def _offsets(lengths):
    return np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)


def _pieces(rows, begins, lengths, stride):
    """Indices into flat [n][stride] text of the pieces [begin, begin + length) of rows, back to back."""
    rows, begins, lengths = (np.asarray(a, dtype=np.int64) for a in (rows, begins, lengths))
    first = rows * stride + begins
    off = _offsets(lengths)
    return np.repeat(first - off[:-1], lengths) + np.arange(off[-1])


def _outputs(case, n_calls, n):
    """Output tensors of n_calls drafts for n requests, one row per call."""
    M, dev = case["max_spec"], torch.device("cuda", torch.cuda.current_device())
    z = lambda dt, *s: torch.zeros(n_calls, n, *s, dtype=dt, device=dev)  # noqa: E731
    return {"n_draft": z(torch.int32), "tokens": z(torch.int32, M), "parents": z(torch.int32, M),
            "positions": z(torch.int32, M), "mask": z(torch.int32, M, (M + 31) // 32), "chosen_tree": z(torch.int32),
            "chosen_p": z(torch.int32), "score": z(torch.float64), "status": z(torch.int32)}


def _store(case, corpus, offsets, batch, tokens):
    return sfx.SuffixStore(corpus, offsets, vocab=case["vocab"], depth_cap=case["depth"], max_requests=batch,
                           max_req_tokens=tokens, max_spec_cap=case["max_spec"])


def _spec(case):
    return dict(P=case["P"], alpha=case["alpha"], max_spec=case["max_spec"], flags=case["flags"], tau=case["tau"])


# --------------------------------------------------------------------------------------- prepare
def prepare(case, seed):
    text = _Text(case, seed)
    rng = np.random.default_rng(seed + 1)
    dev, kind = text.dev, case["kind"]
    corpus = text.corpus()
    n_seqs = -(-case["corpus"] // SEQ)
    seq_offsets = torch.from_numpy(np.minimum(np.arange(n_seqs + 1, dtype=np.int64) * SEQ, case["corpus"])).to(dev)
    s = {"case": case, "spec": _spec(case), "corpus": corpus, "seq_offsets": seq_offsets}
    if kind in ("build", "entropy"):
        if kind == "entropy":
            s["store"] = _store(case, corpus, seq_offsets, 1, 256)
            return s
        # paths of 1 .. depth tokens: spans of the corpus, every fourth with a last token of its own
        q = case["queries"]
        lengths = rng.integers(1, case["depth"] + 1, q)
        begins = rng.integers(0, case["corpus"] - case["depth"], q)
        paths = corpus[torch.from_numpy(_pieces(np.zeros(q), begins, lengths, 0)).to(dev)]
        off = _offsets(lengths)
        last = torch.from_numpy(off[1::4] - 1).to(dev)
        paths[last] = torch.randint(0, case["vocab"], (last.numel(),), device=dev, dtype=torch.int32, generator=text.g)
        s.update(paths=paths, path_offsets=torch.from_numpy(off).to(dev), path_tree=torch.full((q,), -1, dtype=torch.int32, device=dev))
        return s

    B, prompt = case["batch"], case["prompt"]
    if kind == "serve":
        return _prepare_serve(case, text, rng, s)
    steps = case.get("steps", 0)
    taken = _accepted(rng, (steps, B)) if steps else np.zeros((0, B), dtype=np.int64)
    lengths = _ragged(rng, B, prompt)
    new = int(taken.sum(0).max()) if steps else 0
    stride = prompt + new
    texts = text.texts(B, stride, corpus).reshape(-1)
    s["slots"] = torch.arange(B, dtype=torch.int32, device=dev)
    s["store"] = _store(case, corpus, seq_offsets, B, stride)
    s["host_slots"], s["host_offsets"] = np.arange(B, dtype=np.int32), _offsets(lengths)
    s["prompts"] = texts[torch.from_numpy(_pieces(np.arange(B), np.zeros(B), lengths, stride)).to(dev)]
    if kind in ("draft", "refill"):
        s["store"].build_requests(s["host_slots"], s["host_offsets"], s["prompts"])
    if kind == "refill":
        n = case["new"]
        slots = rng.choice(B, n, replace=False).astype(np.int32)
        lengths = _ragged(rng, n, prompt)
        texts = text.texts(n, prompt, corpus).reshape(-1)
        s["host_slots"], s["host_offsets"] = slots, _offsets(lengths)
        s["prompts"] = texts[torch.from_numpy(_pieces(np.arange(n), np.zeros(n), lengths, prompt)).to(dev)]
        s["slots"] = torch.from_numpy(slots).to(dev)
    s["out"] = _outputs(case, max(1, steps), s["slots"].numel())
    s["calls"] = [{k: v[i] for k, v in s["out"].items()} for i in range(max(1, steps))]
    begins = lengths.copy()
    s["steps"] = []
    for i in range(steps):
        off = torch.from_numpy(_offsets(taken[i])).to(dev)
        s["steps"].append((off, texts[torch.from_numpy(_pieces(np.arange(B), begins, taken[i], stride)).to(dev)]))
        begins += taken[i]
    return s


def _prepare_serve(case, text, rng, s):
    """The calls of a service's first steps: which tokens every slot takes, which requests finish."""
    B, prompt, dev = case["batch"], case["prompt"], text.dev
    taken = _accepted(rng, (case["steps"], B))
    request = np.arange(B)
    plen = list(_ragged(rng, B, prompt))
    olen = list(rng.integers(min(16, case["out_lo"]), case["out_hi"] + 1, B))    # the first ones are at all stages of theirs
    done = np.zeros(B, dtype=np.int64)
    plan = []
    for i in range(case["steps"]):
        slots, rows, begins, lengths, ends, refill = [], [], [], [], [], []
        for b in range(B):
            r = request[b]
            take = min(int(taken[i, b]), int(olen[r]) - int(done[b]))
            if done[b] + take < olen[r]:
                slots.append(b); rows.append(r); begins.append(plen[r] + done[b]); lengths.append(take)
                done[b] += take
            else:
                ends.append(r)
                plen.append(int(_ragged(rng, 1, prompt)[0]))
                olen.append(int(rng.integers(case["out_lo"], case["out_hi"] + 1)))
                request[b], done[b] = len(plen) - 1, 0
                refill.append((b, len(plen) - 1))
        for r in ends:
            slots.append(-1); rows.append(r); begins.append(plen[r]); lengths.append(olen[r])
        plan.append((slots, rows, begins, lengths, refill))
    stride = prompt + case["out_hi"]
    texts = text.texts(len(plen), stride, s["corpus"]).reshape(-1)

    def piece(rows, begins, lengths):
        return texts[torch.from_numpy(_pieces(rows, begins, lengths, stride)).to(dev)]

    s["stride"] = stride
    s["host_slots"], s["host_offsets"] = np.arange(B, dtype=np.int32), _offsets(plen[:B])
    s["prompts"] = piece(np.arange(B), np.zeros(B), plen[:B])
    s["slots"] = torch.arange(B, dtype=torch.int32, device=dev)
    s["out"] = _outputs(case, case["steps"], B)
    s["calls"] = [{k: v[i] for k, v in s["out"].items()} for i in range(case["steps"])]
    s["steps"] = []
    for slots, rows, begins, lengths, refill in plan:
        items = (torch.tensor(slots, dtype=torch.int32, device=dev), torch.from_numpy(_offsets(lengths)).to(dev),
                 piece(rows, begins, lengths))
        new = None
        if refill:
            rr = [r for _, r in refill]
            pl = [plen[r] for r in rr]
            new = (np.array([b for b, _ in refill], dtype=np.int32), _offsets(pl), piece(rr, np.zeros(len(rr)), pl))
        s["steps"].append((items, new))
    return s


# ------------------------------------------------------------------------------------------- run
def run(s):
    case, spec, kind = s["case"], s["spec"], s["case"]["kind"]
    if kind == "draft":
        s["store"].speculate(s["slots"], out=s["calls"][0], **spec)
    elif kind == "decode":
        store = s["store"]
        store.build_requests(s["host_slots"], s["host_offsets"], s["prompts"])
        for (offsets, tokens), out in zip(s["steps"], s["calls"]):
            store.step(s["slots"], offsets, tokens, out=out, **spec)
    elif kind == "refill":
        s["store"].build_requests(s["host_slots"], s["host_offsets"], s["prompts"])
        s["store"].speculate(s["slots"], out=s["calls"][0], **spec)
    elif kind == "serve":
        store = _store(case, s["corpus"], s["seq_offsets"], case["batch"], s["stride"])
        store.build_requests(s["host_slots"], s["host_offsets"], s["prompts"])
        for (items, new), out in zip(s["steps"], s["calls"]):
            store.speculate(s["slots"], out=out, **spec)
            store.append(*items)
            if new is not None:
                store.build_requests(*new)
        stats = store.stats()
        store.free()
        return dict(s["out"], nodes=stats["global_nodes"], tokens_in=stats["global_tokens"])
    elif kind == "build":
        store = _store(case, s["corpus"], s["seq_offsets"], 1, 256)
        counts = store.query_counts(s["path_tree"], s["path_offsets"], s["paths"])
        stats = store.stats()
        store.free()
        return {"counts": counts, "nodes": stats["global_nodes"], "tokens": stats["global_tokens"]}
    else:
        return s["store"].entropy(-1)
    return s["out"]


# ------------------------------------------------------------------------------ work and tolerance
def _nodes_per_token(case):
    """Tree nodes a token of this text adds: new strings begin only around the ends of the copied spans."""
    D = case["depth"]
    event = (1.0 - case["copy"]) + case["copy"] * case["span"]
    return min(0.85 * D, 0.45 * D * D / 2.0 / event + 1.0)


def work(case):
    kind, D, M = case["kind"], case["depth"], case["max_spec"]
    accepted = MEAN_EXTRA + 1.0
    built = case["corpus"] * (4.0 + 16.0 * _nodes_per_token(case))              # tokens in, 16-byte nodes out
    # a draft: its outputs, one sector per pattern and tree for the match, one node and its child run per drafted node
    draft = 24.0 + M * (12.0 + 4.0 * ((M + 31) // 32)) + 32.0 * 2 * min(case["P"], D) + 64.0 * M
    token = 4.0 + 32.0 * D                                                       # one count read and written per depth
    prompt = lambda n: n * 0.75 * case["prompt"] * (8.0 + 16.0 * _nodes_per_token(case))  # noqa: E731  (prompts are ragged)
    ops = 4.0 * M                                                                # a division, a product and an addition per drafted node
    if kind == "draft":
        return {"bytes": case["batch"] * draft, "flops": case["batch"] * ops}
    if kind == "decode":
        n = case["steps"] * case["batch"]
        return {"bytes": prompt(case["batch"]) + n * (draft + accepted * token), "flops": n * ops}
    if kind == "refill":
        return {"bytes": prompt(case["new"]) + case["new"] * draft, "flops": case["new"] * ops}
    if kind == "serve":
        n = case["steps"] * case["batch"]
        ends = n * accepted / (0.5 * (case["out_lo"] + case["out_hi"]))
        return {"bytes": built + prompt(case["batch"] + ends) + n * (draft + 2 * accepted * token), "flops": n * ops}
    if kind == "build":
        return {"bytes": built + case["queries"] * D * 20.0, "flops": 0.0}
    return {"bytes": case["corpus"] * 16.0 * _nodes_per_token(case), "flops": case["corpus"] * 4.0 * _nodes_per_token(case)}


def tolerance(case):
    # drafts, counts and scores are the same bits whatever the order of the work; the entropy is a sum
    # of some tens of millions of binary64 terms in an order that is not fixed
    return {"rel": 1e-11} if case["kind"] == "entropy" else "exact"
