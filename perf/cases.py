"""Performance cases of the sampling library: what a serving program asks of it, with inputs made on the GPU.

A case is one call of one entry point of the binding:

  op        "sample" (one token per row), "verify" (speculative verification), "topk" (standalone top-k) or
            "topk_static" (the same without a workspace, at most 8 rows)
  rows, vocab, dtype   the logit matrix; for "verify" `rows` requests of `draft` + 1 positions each
  mix       the requests' parameters (sample, verify):
              "mixed"    half greedy, half stochastic with temperature, top-k of 0 (off), 20, 50 or 1000, top-p and min-p
              "kinds"    greedy, top-k 50, top-p 0.9 and min-p 0.05 rows in turn
              "chat"     every row temperature 0.8, top-k 50, top-p 0.9
              "nucleus"  every row stochastic with top-p or min-p and no top-k
              "grammar"  a quarter greedy, else temperature, top-k 64, top-p 0.95
              "greedy"   every row greedy
              "drafts"   (verify) half greedy, half stochastic with top-k of 0, 20 or 50 and top-p
  history, bias   entries of each row's token history (all three penalties on) and of its bias list; 0: off
  mask      a grammar bitmask that allows 2% of the ids
  shape     how the logits are distributed: "mixture" (a third of the rows peaked, a third Zipf, a third flat),
            "spiked" (N(0, 1) with a few ids far above), "zipf" or "normal"
  k         (topk) entries wanted
  captured  the call is captured in a CUDA graph once, as a decode loop does, and a pass replays it; otherwise a pass
            makes the call itself
"""
import ctypes
import math

import torch

from paper_2607_20475_b200 import binding as sonic
from paper_2607_20475_b200 import workloads as wl

MAX_HISTORY = 1024


def _sample(rows, vocab, dtype, mix, shape, captured, history=0, bias=0, mask=False):
    return {"op": "sample", "rows": rows, "vocab": vocab, "dtype": dtype, "mix": mix, "shape": shape,
            "history": history, "bias": bias, "mask": mask, "captured": captured}


def _verify(rows, draft, vocab, dtype, captured, history=0, bias=0, mask=False):
    return {"op": "verify", "rows": rows, "draft": draft, "vocab": vocab, "dtype": dtype, "mix": "drafts",
            "shape": "spiked", "history": history, "bias": bias, "mask": mask, "captured": captured}


def _topk(rows, vocab, dtype, k, shape, captured, op="topk"):
    return {"op": op, "rows": rows, "vocab": vocab, "dtype": dtype, "k": k, "shape": shape, "captured": captured}


def listed():
    return [
        # One interactive request, called eagerly: host launches and the chain's latency.
        {"name": "one_row", **_sample(1, 131072, "bf16", "chat", "spiked", False)},
        # A handful of requests with one row of each kind, inside a captured decode step.
        {"name": "tiny_kinds", **_sample(4, 32768, "f32", "kinds", "spiked", True)},
        # The ordinary decode batch of a server: heterogeneous requests with penalties and biases.
        {"name": "decode_mixed", **_sample(64, 131072, "bf16", "mixed", "mixture", True, history=512, bias=16)},
        # The same from a program that does not capture, with a vocabulary and a batch that divide nothing.
        {"name": "ragged_mixed", **_sample(37, 50021, "f32", "mixed", "mixture", False, history=300, bias=5)},
        # Structured output: a grammar bitmask on every row, large vocabulary.
        {"name": "grammar", **_sample(128, 262144, "f32", "grammar", "mixture", False, history=512, bias=16, mask=True)},
        # Requests that ask for top-p or min-p only: the truncation needs the whole row.
        {"name": "nucleus", **_sample(32, 100003, "bf16", "nucleus", "mixture", False)},
        # A large batch of like requests (temperature, top-k 50, top-p 0.9), the default of a chat server.
        {"name": "chat_batch", **_sample(256, 262144, "bf16", "chat", "normal", True)},
        # Speculative decoding: the verification of four drafts for each of 32 requests.
        {"name": "verify", **_verify(32, 4, 131072, "f32", True)},
        # The same for a few requests with penalties, eager.
        {"name": "verify_small", **_verify(3, 2, 32003, "bf16", False, history=200, bias=4)},
        # Standalone top-k as a beam or candidate search uses it: the largest matrix, moderate k.
        {"name": "topk_64", **_topk(256, 262144, "f32", 64, "normal", False)},
        # Top-k for distillation targets: thousands of entries of every row, odd vocabulary.
        {"name": "topk_4096", **_topk(128, 200003, "f32", 4096, "zipf", False)},
        # A plug-in that may not allocate, a few rows.
        {"name": "topk_static", **_topk(8, 65536, "bf16", 50, "normal", False, op="topk_static")},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: sizes over the logarithm of their range, odd ones among them; rows * vocab stays below the listed case
    of the kind (rows without top-k cost the most per element, a plain top-k the least)."""
    op = rng.choice(("sample", "sample", "sample", "verify", "topk", "topk_static"))
    dtype = rng.choice(("bf16", "f32"))
    captured = rng.random() < 0.5
    vocab = _log_int(rng, 8192, 262144)
    if rng.random() < 0.4:
        vocab = min(262144, (vocab + 1023) // 1024 * 1024)
    history = rng.choice((0, _log_int(rng, 16, MAX_HISTORY)))
    bias = rng.choice((0, rng.randint(1, 32)))
    if op in ("topk", "topk_static"):
        k = _log_int(rng, 1, 4096)
        most = 8 if op == "topk_static" else 256 if k <= 256 else 96
        rows = _log_int(rng, 1, most)
        return _topk(rows, vocab, dtype, k, rng.choice(("spiked", "zipf", "normal")), captured, op)
    if op == "verify":
        draft = rng.randint(1, 7)
        rows = _log_int(rng, 1, max(1, min(64, 20_000_000 // (vocab * (draft + 1)))))
        return _verify(rows, draft, vocab, dtype, captured, history, bias, rng.random() < 0.2)
    mix = rng.choice(("mixed", "mixed", "kinds", "chat", "nucleus", "grammar", "greedy"))
    elements = {"mixed": 8_000_000, "kinds": 4_000_000, "nucleus": 3_200_000}.get(mix, 64_000_000)
    rows = _log_int(rng, 1, max(1, min(256, elements // vocab)))
    return _sample(rows, vocab, dtype, mix, rng.choice(("mixture", "spiked", "normal")), captured, history, bias,
                   mix == "grammar")


# ------------------------------------------------------------------------------------------------ inputs
def _spiked(g, rows, vocab, boost):
    x = torch.randn(rows, vocab, generator=g, device="cuda")
    ids = torch.randint(0, vocab, (rows, 4), generator=g, device="cuda")
    up = torch.rand(rows, 4, generator=g, device="cuda") < 0.6      # one to four ids far above the rest
    up[:, 0] = True
    return x.scatter_add_(1, ids, up * boost)


def _zipf(g, rows, vocab, s):
    order = torch.rand(rows, vocab, generator=g, device="cuda").argsort(1)
    logp = -s * torch.log(torch.arange(1, vocab + 1, device="cuda", dtype=torch.float32))
    return logp[order]


def _logits(g, rows, vocab, shape):
    if shape == "spiked":
        return _spiked(g, rows, vocab, 10.0)
    if shape == "zipf":
        return _zipf(g, rows, vocab, 1.0)
    if shape == "normal":
        return torch.randn(rows, vocab, generator=g, device="cuda")
    x = torch.empty(rows, vocab, device="cuda")
    for r, part in ((0, lambda n: _spiked(g, n, vocab, 10.0)), (1, lambda n: _zipf(g, n, vocab, 1.1)),
                    (2, lambda n: torch.randn(n, vocab, generator=g, device="cuda") * 0.5)):
        n = len(range(r, rows, 3))
        if n:
            x[r::3] = part(n)
    return x


def _padded(x, dtype):
    """The logit matrix as the library takes it: rows that start on 16-byte boundaries."""
    rows, vocab = x.shape
    t, vec = (torch.float32, 4) if dtype == "f32" else (torch.bfloat16, 8)
    out = torch.zeros(rows, -(-vocab // vec) * vec, dtype=t, device="cuda")
    out[:, :vocab] = x
    return out


def _params(g, rows, mix):
    """Per-request mode bits and parameters. Choices of a kind are dealt evenly and shuffled, so that another seed gives
    other requests but the same mixture."""
    def deal(values, n):
        v = [values[i % len(values)] for i in range(n)]
        return [v[i] for i in torch.randperm(n, generator=g).tolist()]

    p = {"mode": [0] * rows, "top_k": [0] * rows, "top_p": [1.0] * rows, "min_p": [0.0] * rows}
    tau = (0.5 + torch.rand(rows, generator=g)).tolist()
    kind = {"mixed": ["s", "g"], "drafts": ["s", "g"], "kinds": ["g", "k", "p", "m"], "chat": ["c"], "nucleus": ["n"],
            "grammar": ["g", "q", "q", "q"], "greedy": ["g"]}[mix]
    kind = [kind[r % len(kind)] for r in range(rows)]
    ks = deal((50, 0, 20, 1000) if mix == "mixed" else (50, 0, 20), rows)
    ps = deal((0.9, 1.0, 0.95), rows)
    ms = deal((0.0, 0.05), rows)
    for r, c in enumerate(kind):
        if c == "g":
            p["mode"][r] = wl.GREEDY
            continue
        k, top, low = {"s": (ks[r], ps[r], 0.0 if mix == "drafts" else ms[r]), "k": (50, 1.0, 0.0), "p": (0, 0.9, 0.0),
                       "m": (0, 1.0, 0.05), "c": (50, 0.9, 0.0), "q": (64, 0.95, 0.0),
                       "n": (0, 0.9 if r % 4 < 2 else 0.95 if r % 4 == 2 else 1.0, 0.05 if r % 4 == 3 else 0.0)}[c]
        tau[r] = 0.8 if c == "c" else tau[r]
        p["top_k"][r], p["top_p"][r], p["min_p"][r] = k, top, low
        p["mode"][r] = (wl.TEMPERATURE | (wl.TOP_K if k else 0) | (wl.TOP_P if top < 1.0 else 0)
                        | (wl.MIN_P if low > 0.0 else 0))
    p["temperature"] = tau
    return p


def _distinct(g, rows, vocab, n):
    """n distinct ids of every row, in no order."""
    u = torch.rand(rows, n, generator=g, device="cuda", dtype=torch.float64)
    ids = ((torch.arange(n, device="cuda") + u) * (vocab / n)).long().clamp_(max=vocab - 1)
    return ids.gather(1, torch.rand(rows, n, generator=g, device="cuda").argsort(1)).int()


def _bitmask(g, x):
    """Packed words that allow 2% of the ids of every row, the largest logit among them on even rows and not on odd ones."""
    rows, vocab = x.shape
    words = -(-vocab // 32)
    on = torch.zeros(rows, words * 32, dtype=torch.bool, device="cuda")
    on[:, :vocab] = torch.rand(rows, vocab, generator=g, device="cuda") < 0.02
    top = x.argmax(1, keepdim=True)
    on.scatter_(1, top, (torch.arange(rows, device="cuda") % 2 == 0).unsqueeze(1))
    bit = (torch.ones(32, dtype=torch.int32, device="cuda") << torch.arange(32, dtype=torch.int32, device="cuda"))
    return (on.view(rows, words, 32) * bit).sum(2, dtype=torch.int32)


def _draft(g, x, p, rows, draft, vocab):
    """Draft distributions [rows, draft, vocab] of a model that is near the target, cut as the request asks, and tokens
    drawn from them (their maxima for greedy requests)."""
    q = torch.empty(rows, draft, vocab, device="cuda")
    tokens = torch.empty(rows, draft, dtype=torch.int32, device="cuda")
    for b in range(rows):
        greedy = bool(p["mode"][b] & wl.GREEDY)
        z = x[b, :draft].float() + torch.randn(draft, vocab, generator=g, device="cuda") * 0.5
        z = z if greedy else z / p["temperature"][b]
        v, order = z.sort(1, descending=True)
        w = torch.softmax(v, 1, dtype=torch.float64)
        if not greedy:
            if p["top_k"][b]:
                w[:, p["top_k"][b]:] = 0.0
            if p["top_p"][b] < 1.0:
                before = w.cumsum(1) - w
                w[before >= p["top_p"][b] * w.sum(1, keepdim=True)] = 0.0
        q[b] = torch.zeros(draft, vocab, device="cuda").scatter_(1, order, (w / w.sum(1, keepdim=True)).float())
        tokens[b] = (q[b].argmax(1) if greedy else torch.multinomial(q[b], 1, generator=g)[:, 0]).int()
    return q, tokens


# ------------------------------------------------------------------------------------------------ the calls
def _set_params(s, a, p, g, case, logit_rows, x):
    rows, vocab = case["rows"], case["vocab"]
    if case["history"]:
        n = min(case["history"], vocab)
        s["hist_ids"] = _distinct(g, rows, vocab, n)
        s["hist_counts"] = 1 + (torch.rand(rows, n, generator=g, device="cuda") < 0.1).int()
        s["hist_len"] = torch.full((rows,), n, dtype=torch.int32, device="cuda")
        a.hist_stride = n
        for name, v in (("rep_penalty", 1.1), ("freq_penalty", 0.2), ("pres_penalty", 0.3)):
            s[name] = torch.full((rows,), v, dtype=torch.float32, device="cuda")
        p["mode"] = [m | wl.REPETITION | wl.FREQUENCY | wl.PRESENCE for m in p["mode"]]
    if case["bias"]:
        n = min(case["bias"], vocab)
        s["bias_ids"] = _distinct(g, rows, vocab, n)
        s["bias_vals"] = torch.rand(rows, n, generator=g, device="cuda") * 10.0 - 5.0
        s["bias_len"] = torch.full((rows,), n, dtype=torch.int32, device="cuda")
        a.bias_stride = n
        p["mode"] = [m | wl.BIAS for m in p["mode"]]
    if case["mask"]:
        s["bitmask"] = _bitmask(g, x)
        a.bitmask_stride = s["bitmask"].shape[1]
        p["mode"] = [m | wl.GRAMMAR for m in p["mode"]]
    for name, t in (("mode", torch.int32), ("temperature", torch.float32), ("top_k", torch.int32), ("top_p", torch.float32),
                    ("min_p", torch.float32)):
        s[name] = torch.tensor(p[name], dtype=t, device="cuda")
    s["seed"] = torch.randint(0, 1 << 62, (rows,), generator=g, device="cuda", dtype=torch.int64)
    s["offset"] = torch.randint(0, 4096, (rows,), generator=g, device="cuda", dtype=torch.int64)
    s["out_token"] = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
    s["out_prob"] = torch.zeros(rows, dtype=torch.float32, device="cuda")
    s["out_flags"] = torch.zeros(rows, dtype=torch.int32, device="cuda")
    s["out_support"] = torch.zeros(rows, dtype=torch.int32, device="cuda")
    for name in ("logits", "mode", "bitmask", "temperature", "top_k", "top_p", "min_p", "rep_penalty", "freq_penalty",
                 "pres_penalty", "hist_ids", "hist_counts", "hist_len", "bias_ids", "bias_vals", "bias_len", "seed", "offset",
                 "out_token", "out_prob", "out_flags", "out_support"):
        if name in s:
            setattr(a, name, s[name].data_ptr())
    a.struct_size = ctypes.sizeof(sonic.SampleArgs)
    a.B, a.V = rows, vocab
    a.dtype = wl.DTYPE_F32 if case["dtype"] == "f32" else wl.DTYPE_BF16
    a.row_stride = s["logits"].shape[1]
    s["ws"] = sonic.new_workspace(logit_rows, vocab)


def _call(s):
    op = s["op"]
    if op == "sample":
        sonic.sonic_sample(s["args"], s["ws"])
    elif op == "verify":
        sonic.sonic_verify(s["args"], s["ws"])
    elif op == "topk":
        sonic.sonic_topk(s["logits"], s["type"], s["rows"], s["vocab"], s["stride"], s["k"], s["vals"], s["idx"], s["ws"])
    else:
        sonic.sonic_topk_static(s["logits"], s["type"], s["rows"], s["vocab"], s["stride"], s["k"], s["vals"], s["idx"])


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    host = torch.Generator()
    host.manual_seed(seed)
    op, rows, vocab = case["op"], case["rows"], case["vocab"]
    s = {"op": op}
    if op in ("topk", "topk_static"):
        s["logits"] = _padded(_logits(g, rows, vocab, case["shape"]), case["dtype"])
        s.update(rows=rows, vocab=vocab, k=case["k"], stride=s["logits"].shape[1],
                 type=wl.DTYPE_F32 if case["dtype"] == "f32" else wl.DTYPE_BF16)
        s["vals"] = torch.zeros(rows, case["k"], dtype=torch.float32, device="cuda")
        s["idx"] = torch.full((rows, case["k"]), -7, dtype=torch.int32, device="cuda")
        if op == "topk":
            s["ws"] = sonic.new_workspace(rows, vocab)
        s["out"] = (s["vals"], s["idx"])
    else:
        p = _params(host, rows, case["mix"])
        per = case["draft"] + 1 if op == "verify" else 1
        x = _logits(g, rows * per, vocab, case["shape"])
        s["logits"] = _padded(x, case["dtype"])
        a = sonic.SampleArgs()
        _set_params(s, a, p, g, case, rows * per, x)
        if op == "sample":
            s["args"] = a
            s["out"] = (s["out_token"], s["out_prob"], s["out_support"])
        else:
            draft = case["draft"]
            s["q"], s["draft_tokens"] = _draft(g, s["logits"][:, :vocab].view(rows, per, -1), p, rows, draft, vocab)
            s["out_tokens"] = torch.full((rows, draft + 1), -7, dtype=torch.int32, device="cuda")
            s["out_accept"] = torch.zeros(rows, dtype=torch.int32, device="cuda")
            s["out_p"] = torch.zeros(rows, draft, dtype=torch.float32, device="cuda")
            v = s["args"] = sonic.VerifyArgs()
            v.struct_size = ctypes.sizeof(sonic.VerifyArgs)
            v.K = draft
            v.s = a
            v.draft_tokens, v.draft_probs = s["draft_tokens"].data_ptr(), s["q"].data_ptr()
            v.out_tokens, v.out_accept_len = s["out_tokens"].data_ptr(), s["out_accept"].data_ptr()
            v.out_p_draft = s["out_p"].data_ptr()
            s["out"] = (s["out_tokens"], s["out_accept"], s["out_p"])
    if case["captured"]:
        _call(s)                       # the first call of a process loads the kernels
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _call(s)
    return s


def run(state):
    # The per-row flags are not among the outputs: they say which kernels finished a row, beside what the token (-1) says.
    if "graph" in state:
        state["graph"].replay()
    else:
        _call(state)
    return state["out"]


def work(case):
    """Every logit, mask word and list entry read once, the outputs written once; of the draft distributions only the
    probability of each drafted token, since whole rows are needed for rejected drafts alone. One comparison per logit."""
    rows, vocab = case["rows"], case["vocab"]
    logit_rows = rows * (case["draft"] + 1) if case["op"] == "verify" else rows
    elements = logit_rows * vocab
    n = elements * (4 if case["dtype"] == "f32" else 2)
    if case["op"] in ("topk", "topk_static"):
        return {"bytes": n + rows * case["k"] * 8, "flops": elements}
    if case["mask"]:
        n += logit_rows * -(-vocab // 32) * 4
    n += rows * 8 * (min(case["history"], vocab) + min(case["bias"], vocab)) + rows * 48
    if case["op"] == "verify":
        n += rows * case["draft"] * 16 + rows * 8
    return {"bytes": n, "flops": elements}


def tolerance(case):
    if case["op"] in ("topk", "topk_static"):
        return "exact"                 # values are copied, ties go to the lowest index
    # Probabilities are quotients of sums of exponentials in 32 bits or more. A draw or a cut within rounding of its
    # threshold may fall on either side.
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
