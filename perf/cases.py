"""The work that this library is measured on.

One case is one pass of a program that serves a large multimodal model with
speculative decoding: the verification step (attention of the draft rows over
the paged KV cache, layer by layer, then the acceptance rule), the draft
side's distribution tail (LM head, softmax, sampling), the target LM head
fused with the acceptance, and the visual token compressor.  Sizes are those
of the library's workloads (paper_2505_12728_gb300/workloads.py) and of its
tests; `draw` spreads over the same ranges.

Two ways of calling occur, as in use.  A program keeps its output buffers
and workspaces either way.  ``captured`` cases hold the step's calls, one per
layer, in a CUDA graph that was recorded once and is replayed for every step
(the entry points are asynchronous and allocation-free, and a decoding loop of
28 or 32 layers is run like that); the others make the calls one by one.

sf_kv_commit moves its state on with every call, so it can't be repeated on one
state and has no case of its own; it is one launch over a few integers.
"""
import math

import torch

from paper_2505_12728_gb300 import specflash_verify as sfv

PAGE = sfv.PAGE_SIZE
DEVICE = "cuda"


# --------------------------------------------------------------------------- #
# the cases                                                                   #
# --------------------------------------------------------------------------- #
def _step(name, **kw):
    """Attention over `layers` layers (kind "attend": no acceptance after them)."""
    c = dict(name=name, kind="step", captured=False, layers=1, B=1, heads=8, kv_heads=8, d=64, rows=4,
             prefix_lo=640, prefix_hi=640, V=32000, mode="sampling", sharpness=1.0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one short sequence, one attention layer and the
        # acceptance, called one by one; latency and launches are all of it
        _step("tiny_step", heads=8, kv_heads=8, d=64, rows=4, prefix_lo=640, prefix_hi=640, V=32000),
        # a chat about five images on a 32-layer model with one KV head per
        # query head: the whole verification step
        _step("image_step", captured=True, layers=32, heads=32, kv_heads=32, d=128, rows=5,
              prefix_lo=3008, prefix_hi=3008, V=32000),
        # a ragged batch of image chats on a 28-layer model with 7 query heads
        # per KV head, greedy and sampled sequences mixed
        _step("ragged_step", captured=True, layers=28, B=8, heads=28, kv_heads=4, d=128, rows=6,
              prefix_lo=1200, prefix_hi=3600, V=152064, mode="alternate"),
        # captioning of four 32-frame videos, draft sharper than the target
        _step("video_step", captured=True, layers=28, B=4, heads=28, kv_heads=4, d=128, rows=8,
              prefix_lo=4864, prefix_hi=4864, V=152064, sharpness=1.5),
        # long videos, large batch: one layer's attention at the longest and
        # at the shortest draft block (56 and 14 query rows per KV head)
        _step("long_attend_8", kind="attend", B=16, heads=28, kv_heads=4, d=128, rows=8, prefix_lo=8192,
              prefix_hi=32768),
        _step("long_attend_2", kind="attend", B=16, heads=28, kv_heads=4, d=128, rows=2, prefix_lo=8192,
              prefix_hi=32768),
        # the acceptance alone at the largest batch and vocabulary
        dict(name="long_accept", kind="accept", B=16, k=8, V=152064, mode="alternate", sharpness=1.0),
        # the draft side: LM head, softmax and sampling of one sequence's
        # drafts, and of a batch of 16 sequences with the larger head
        dict(name="draft_one", kind="draft", R=5, hidden=4096, V=32000, mode="sampling"),
        dict(name="draft_batch", kind="draft", R=128, hidden=3584, V=152064, mode="alternate"),
        # the target's LM head fused with the acceptance, four sequences
        dict(name="head_accept", kind="head", B=4, k=8, hidden=3584, V=152064, mode="sampling", sharpness=1.0),
        # the visual compressor over the images of one prompt, and over the
        # frames of four videos
        dict(name="compress_images", kind="compress", F=5, N=576, C=64, d=4096),
        dict(name="compress_video", kind="compress", F=128, N=144, C=16, d=3584),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# bytes of KV that a drawn case reads at most (below the largest listed case)
_MOST_KV = 1.2e9


def draw(rng):
    kind = rng.choice(["step", "step", "attend", "accept", "draft", "head", "compress"])
    mode = rng.choice(["sampling", "sampling", "greedy", "alternate"])
    if kind in ("step", "attend"):
        heads, kv_heads, d = rng.choice([(8, 8, 64), (32, 32, 128), (28, 4, 128), (28, 4, 128), (16, 4, 64)])
        rows = rng.randint(1, 8)
        hi = _log_int(rng, 500, 32768)
        lo = rng.randint(max(200, hi // 4), hi)
        per_layer = 4.0 * kv_heads * d * 0.5 * (lo + hi)  # one sequence, one layer
        B = min(_log_int(rng, 1, 16), max(1, int(_MOST_KV / per_layer)))
        layers = 1
        if kind == "step":
            layers = min(rng.randint(4, 32), max(1, int(_MOST_KV / (per_layer * B))))
        c = _step(None, kind=kind, captured=kind == "step", layers=layers, B=B, heads=heads, kv_heads=kv_heads, d=d,
                  rows=rows, prefix_lo=lo, prefix_hi=hi, V=_log_int(rng, 1000, 152064), mode=mode,
                  sharpness=rng.choice([1.0, 1.5]))
        del c["name"]
        return c
    if kind == "accept":
        return dict(kind=kind, B=_log_int(rng, 1, 16), k=rng.randint(1, 8), V=_log_int(rng, 1000, 152064), mode=mode,
                    sharpness=rng.choice([1.0, 1.5]))
    if kind == "draft":
        return dict(kind=kind, R=_log_int(rng, 1, 128), hidden=8 * _log_int(rng, 64, 448),
                    V=_log_int(rng, 1000, 152064), mode=mode)
    if kind == "head":
        k = rng.randint(1, 8)
        return dict(kind=kind, B=_log_int(rng, 1, 128 // (k + 1)), k=k, hidden=8 * _log_int(rng, 64, 448),
                    V=_log_int(rng, 1000, 152064), mode=mode, sharpness=1.0)
    N = _log_int(rng, 32, 700)
    return dict(kind=kind, F=_log_int(rng, 1, max(1, 18432 // N)), N=N, C=min(128, max(1, N // rng.randint(6, 12))),
                d=128 * rng.randint(8, 32))


# --------------------------------------------------------------------------- #
# inputs                                                                      #
# --------------------------------------------------------------------------- #
def _prefixes(c):
    """Cached tokens of each sequence: fixed by the case (a low-discrepancy
    spread over the range), so that every seed's inputs are the same work."""
    span = c["prefix_hi"] - c["prefix_lo"]
    return [c["prefix_lo"] + int(span * ((0.5 + b * 0.6180339887498949) % 1.0)) for b in range(c["B"])]


def _taus(mode, n, per=1):
    """Temperature of each sequence: 1, 0 (greedy), or alternating from 0."""
    t = {"sampling": [1.0] * n, "greedy": [0.0] * n, "alternate": [float(b % 2) for b in range(n)]}[mode]
    return torch.tensor([x for x in t for _ in range(per)], dtype=torch.float32, device=DEVICE)


def _randn(g, *shape, dtype=torch.float32, std=1.0):
    x = torch.randn(*shape, generator=g, device=DEVICE, dtype=dtype)
    return x if std == 1.0 else x.mul_(std)


def _draft_inputs(g, c, B, k, logits):
    """The draft's distributions (a noisy, possibly sharper view of the target's
    logits), the tokens drawn from them, uniforms and temperatures."""
    V = c["V"]
    probs = torch.empty(B, k, V, device=DEVICE)
    for b in range(B):
        probs[b] = torch.softmax(c["sharpness"] * logits[b, :k].float() + _randn(g, k, V), dim=-1)
    tau = _taus(c["mode"], B)
    drawn = torch.multinomial(probs.view(B * k, V), 1, generator=g).view(B, k)
    tokens = torch.where(tau[:, None] > 0, drawn, probs.argmax(-1)).to(torch.int32)
    return dict(draft_probs=probs, draft_tokens=tokens, u=torch.rand(B, k + 1, generator=g, device=DEVICE), tau=tau)


def _inputs(c, seed):
    """A case's inputs, from the seed alone."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    kind, bf16 = c["kind"], torch.bfloat16
    x = {}
    if kind in ("step", "attend"):
        lens = [p + c["rows"] for p in _prefixes(c)]
        pages = [-(-t // PAGE) for t in lens]
        pool = sum(pages)
        # a sequence's pages lie anywhere in the pool
        order = torch.randperm(pool, generator=g, device=DEVICE).to(torch.int32)
        table = torch.full((c["B"], max(pages)), -1, dtype=torch.int32, device=DEVICE)
        for b, m in enumerate(pages):
            table[b, :m] = order[sum(pages[:b]):sum(pages[:b]) + m]
        x.update(table=table, lens=torch.tensor(lens, dtype=torch.int32, device=DEVICE), layers=[])
        for _ in range(c["layers"]):
            kv = (pool, c["kv_heads"], PAGE, c["d"])
            x["layers"].append((_randn(g, c["B"], c["rows"], c["heads"], c["d"], dtype=bf16),
                                _randn(g, *kv, dtype=bf16), _randn(g, *kv, dtype=bf16)))
    if kind in ("step", "accept"):
        k = _drafts(c)
        x["logits"] = _randn(g, c["B"], k + 1, c["V"], std=3.0)
        x.update(_draft_inputs(g, c, c["B"], k, x["logits"]))
    if kind in ("draft", "head"):
        x["weight"] = _randn(g, c["V"], c["hidden"], dtype=bf16, std=3.0 / math.sqrt(c["hidden"]))
    if kind == "draft":
        x.update(hidden=_randn(g, c["R"], c["hidden"], dtype=bf16),
                 u=torch.rand(c["R"], generator=g, device=DEVICE), tau=_taus(c["mode"], c["R"]))
    if kind == "head":
        x["hidden"] = _randn(g, c["B"], c["k"] + 1, c["hidden"], dtype=bf16)
        x.update(_draft_inputs(g, c, c["B"], c["k"], x["hidden"] @ x["weight"].t()))
    if kind == "compress":
        x.update(queries=_randn(g, c["C"], c["d"], dtype=bf16, std=2.0 / math.sqrt(c["d"])),
                 features=_randn(g, c["F"], c["N"], c["d"], dtype=bf16))
    return x


def _drafts(c):
    return c["rows"] if c["kind"] == "step" else c["k"]


# --------------------------------------------------------------------------- #
# one pass                                                                    #
# --------------------------------------------------------------------------- #
def prepare(case, seed):
    c, kind = case, case["kind"]
    s = dict(case=c, graph=None, **_inputs(c, seed))
    zeros = lambda *shape, dtype=torch.float32: torch.zeros(*shape, dtype=dtype, device=DEVICE)  # noqa: E731
    o = s["out"] = {}
    if kind in ("step", "attend"):
        o["attention"] = zeros(c["layers"], c["B"], c["rows"], c["heads"], c["d"], dtype=torch.bfloat16)
        o["lse"] = zeros(c["layers"], c["B"], c["rows"], c["heads"])
        s["layer_outputs"] = list(zip(o["attention"].unbind(0), o["lse"].unbind(0)))
        s["workspace"] = sfv.new_workspace(sfv.verify_attention_workspace_size(
            c["B"], c["rows"], c["heads"], c["kv_heads"], c["d"], s["table"].shape[1]))
    if kind in ("step", "accept"):
        s["accept_workspace"] = sfv.new_workspace(sfv.accept_workspace_size(c["B"], _drafts(c), c["V"]))
    if kind == "draft":
        o.update(logits=zeros(c["R"], c["V"]), probs=zeros(c["R"], c["V"]), tokens=zeros(c["R"], dtype=torch.int32))
        s["workspace"] = sfv.new_workspace(sfv.draft_tail_workspace_size(c["R"], c["V"]))
    if kind == "head":
        o["logits"] = zeros(c["B"], c["k"] + 1, c["V"])
        s["workspace"] = sfv.new_workspace(sfv.verify_lm_head_accept_workspace_size(c["B"], c["k"], c["V"]))
    if kind in ("step", "accept", "head"):
        o.update(num_accepted=zeros(c["B"], dtype=torch.int32), accept_ratio=zeros(c["B"], _drafts(c)),
                 out_tokens=zeros(c["B"], _drafts(c) + 1, dtype=torch.int32))
    if kind == "compress":
        o["compressed"] = zeros(c["F"], c["C"], c["d"], dtype=torch.bfloat16)
        s["workspace"] = sfv.new_workspace(sfv.visual_compress_workspace_size(c["F"], c["N"], c["C"], c["d"]))
    if c.get("captured"):
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _calls(s)  # the library's one-time set-up, outside the recording
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _calls(s)
    return s


def _calls(s):
    """The case's calls, in order, on the current stream."""
    c, o = s["case"], s["out"]
    kind = c["kind"]
    if kind in ("step", "attend"):
        for (q, k, v), (out, lse) in zip(s["layers"], s["layer_outputs"]):
            sfv.verify_attention(q, k, v, s["table"], s["lens"], out=out, lse=lse, workspace=s["workspace"])
    if kind in ("step", "accept"):
        sfv.accept(s["logits"], s["draft_probs"], s["draft_tokens"], s["u"], s["tau"],
                   num_accepted=o["num_accepted"], out_tokens=o["out_tokens"], accept_ratio=o["accept_ratio"],
                   workspace=s["accept_workspace"])
    if kind == "draft":
        sfv.draft_sample(s["hidden"], s["weight"], s["u"], s["tau"], logits=o["logits"], probs=o["probs"],
                         tokens=o["tokens"], workspace=s["workspace"])
    if kind == "head":
        sfv.verify_lm_head_accept(s["hidden"], s["weight"], s["draft_probs"], s["draft_tokens"], s["u"], s["tau"],
                                  logits=o["logits"], num_accepted=o["num_accepted"], out_tokens=o["out_tokens"],
                                  accept_ratio=o["accept_ratio"], workspace=s["workspace"])
    if kind == "compress":
        sfv.visual_compress(s["queries"], s["features"], out=o["compressed"], workspace=s["workspace"])


def run(state):
    if state["graph"] is not None:
        state["graph"].replay()
    else:
        _calls(state)
    return state["out"]


# --------------------------------------------------------------------------- #
# what a pass cannot do without                                               #
# --------------------------------------------------------------------------- #
def _accept_bytes(c, B, k, logits_too):
    """Every logits row once, and row j of q where the token is drawn from a
    residual (one row a sampled sequence at most)."""
    sampled = {"sampling": B, "greedy": 0, "alternate": B // 2}[c["mode"]]
    return 4 * c["V"] * ((B * (k + 1) if logits_too else 0) + sampled) + 4 * B * (4 * k + 4)


def work(case):
    c, kind = case, case["kind"]
    nbytes = flops = 0
    if kind in ("step", "attend"):
        tokens = sum(p + c["rows"] for p in _prefixes(c))
        nbytes += c["layers"] * (4 * tokens * c["kv_heads"] * c["d"]
                                 + c["B"] * c["rows"] * c["heads"] * (4 * c["d"] + 4))
        flops += c["layers"] * 4 * tokens * c["rows"] * c["heads"] * c["d"]
    if kind in ("step", "accept"):
        k = _drafts(c)
        nbytes += _accept_bytes(c, c["B"], k, True)
        flops += 4 * c["B"] * (k + 1) * c["V"]
    if kind in ("draft", "head"):
        R = c["R"] if kind == "draft" else c["B"] * (c["k"] + 1)
        nbytes += 2 * c["V"] * c["hidden"] + 2 * R * c["hidden"] + 4 * R * c["V"] * (2 if kind == "draft" else 1)
        flops += 2 * R * c["V"] * c["hidden"]
        if kind == "head":
            nbytes += _accept_bytes(c, c["B"], c["k"], False)
    if kind == "compress":
        nbytes += 2 * c["d"] * (c["F"] * c["N"] + c["C"] + c["F"] * c["C"])
        flops += 4 * c["F"] * c["N"] * c["C"] * c["d"]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the error against 64 bits.  Attention and compressed
    features come out in bf16 (2.3e-3 off, most of it the outputs' own
    rounding, P's rounding to bf16 the rest); logits are fp32 sums of up to
    4096 bf16 products (4e-6) and the draft's probabilities show the logits'
    absolute error (1.3e-5); the acceptance ratios of given logits are 5e-8
    off.  Tokens and counts may differ only where a draw lies on a boundary."""
    if case["kind"] in ("step", "attend", "compress"):
        return {"rel": 1e-2, "max": 5e-2}
    if case["kind"] == "accept":
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-2}
    return {"rel": 5e-5, "max": 5e-4, "differ": 1e-2}


# --------------------------------------------------------------------------- #
# the same in 64 bits                                                         #
# --------------------------------------------------------------------------- #
def _exact_attention(c, x):
    f64, d, n, g = torch.float64, c["d"], c["rows"], c["heads"] // c["kv_heads"]
    lens = x["lens"].tolist()
    out = torch.empty(c["layers"], c["B"], n, c["heads"], d, dtype=f64, device=DEVICE)
    lse = torch.empty(c["layers"], c["B"], n, c["heads"], dtype=f64, device=DEVICE)
    for l, (q, k, v) in enumerate(x["layers"]):
        for b, T in enumerate(lens):
            page = x["table"][b, :-(-T // PAGE)].long()
            # [H_kv][T][d]
            kk, vv = (t[page].permute(1, 0, 2, 3).reshape(c["kv_heads"], -1, d)[:, :T].to(f64) for t in (k, v))
            # rows (i, j) of a KV head: draft row i, query head h * g + j
            qq = q[b].to(f64).view(n, c["kv_heads"], g, d).permute(1, 0, 2, 3).reshape(c["kv_heads"], n * g, d)
            s = (qq @ kk.transpose(1, 2)).view(c["kv_heads"], n, g, T) / math.sqrt(d)
            hidden = torch.arange(T, device=DEVICE)[None, :] > T - n + torch.arange(n, device=DEVICE)[:, None]
            s.masked_fill_(hidden[None, :, None, :], -math.inf)
            z = torch.logsumexp(s, dim=-1)
            o = torch.exp(s - z[..., None]).view(c["kv_heads"], n * g, T) @ vv
            out[l, b] = o.view(c["kv_heads"], n, g, d).permute(1, 0, 2, 3).reshape(n, c["heads"], d)
            lse[l, b] = z.permute(1, 0, 2).reshape(n, c["heads"])
    return out, lse


def _exact_ratio(c, x, logits):
    """min(1, p/q) of every draft; 1 on an argmax match, else 0, for greedy
    sequences."""
    B, k = x["draft_tokens"].shape
    ratio = torch.empty(B, k, dtype=torch.float64, device=DEVICE)
    for b, tau in enumerate(x["tau"].tolist()):
        at = x["draft_tokens"][b].long()
        rows = logits[b, :k].to(torch.float64)
        if tau > 0:
            p = torch.softmax(rows / tau, dim=-1).gather(1, at[:, None])[:, 0]
            ratio[b] = torch.clamp(p / x["draft_probs"][b].gather(1, at[:, None])[:, 0].to(torch.float64), max=1.0)
        else:
            ratio[b] = (rows.argmax(-1) == at).to(torch.float64)
    return ratio


def _exact_logits(hidden, weight):
    h = hidden.to(torch.float64)
    parts = [h @ w.to(torch.float64).t() for w in weight.split(16384)]
    return torch.cat(parts, dim=-1)


def exact(case, seed):
    c, kind = case, case["kind"]
    x = _inputs(c, seed)
    o = {}
    if kind in ("step", "attend"):
        o["attention"], o["lse"] = _exact_attention(c, x)
    if kind in ("step", "accept"):
        o.update(num_accepted=None, out_tokens=None, accept_ratio=_exact_ratio(c, x, x["logits"]))
    if kind == "draft":
        o["logits"] = _exact_logits(x["hidden"], x["weight"])
        one_hot = torch.nn.functional.one_hot(o["logits"].argmax(-1), c["V"]).to(torch.float64)
        o.update(probs=torch.where(x["tau"][:, None] > 0, torch.softmax(o["logits"], dim=-1), one_hot), tokens=None)
    if kind == "head":
        o["logits"] = _exact_logits(x["hidden"], x["weight"])
        o.update(num_accepted=None, out_tokens=None, accept_ratio=_exact_ratio(c, x, o["logits"]))
    if kind == "compress":
        f = x["features"].to(torch.float64)
        o["compressed"] = torch.softmax(x["queries"].to(torch.float64) @ f.transpose(1, 2), dim=-1) @ f
    return o
