"""Performance cases of the drafting library: the calls a serving program makes.

Each case is one call (one block, one reduction, one preparation step) through
the public entry points, on inputs made on the GPU from the seed alone. Kinds:

* ``draft``            dels_draft_block / dels_draft_block_weighted through ``Drafter``
* ``draft_sampled``    temperature-1 drafting through ``Drafter.sample``
* ``verify_sampled``   speculative-sampling verification of a sampled block
* ``combine``          dels_combine_argmax over independent rows
* ``verify``           greedy verification against target logits
* ``prior``            unigram prior of a corpus held on the device
* ``input_table``      the GRU input table, built once per set of weights

Weights are scaled by 1/sqrt(fan-in) with unit embeddings, so that the local
head's logits are of order one, as a trained head's are. Logit rows are
N(0, 3) with one likely token 0.5 to 8 above the rest of the row, as a
language model's rows have; a target row agrees with the drafter's likely
token three times out of four.
"""
from __future__ import annotations

import math

import torch

import paper_2607_07409_gb300 as dels

DEV = "cuda:0"
M32 = 0xFFFFFFFF
L2_BYTES = 126 << 20          # weights beyond this are streamed from memory again at every position
STD = 3.0
TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}


class Spec:
    """Shape of a local head, with the fields ``make_head`` reads."""

    def __init__(self, c):
        self.kind, self.wdtype = c["head"], c["wdtype"]
        self.d_model, self.d_hidden, self.d_rank = c["d_model"], c["d_hidden"], c["d_rank"]
        self.window, self.n_layers = c.get("window", 0), c.get("n_layers", 1)
        self.n_heads, self.max_pos = c.get("n_heads", 0), c.get("max_pos", 0)


def _draft(kind, head, wdtype, ldtype, B, n, V, d_model, d_hidden, d_rank, **kw):
    return dict(kind=kind, head=head, wdtype=wdtype, ldtype=ldtype, B=B, n=n, V=V, d_model=d_model,
                d_hidden=d_hidden, d_rank=d_rank, weight=0.5, **kw)


def listed():
    return [
        # The smallest call: one request, a toy float32 window-MLP head over 1024 tokens. Latency and launches.
        dict(_draft("draft", "mlp", "f32", "f32", 1, 8, 1024, 128, 128, 128, window=2, n_layers=1),
             name="draft_mlp_f32_tiny"),
        # Interactive serving: one request, two-layer window-MLP head of width 1024, full vocabulary, float32 logits.
        dict(_draft("draft", "mlp", "bf16", "f32", 1, 16, 151936, 1024, 1024, 1024, window=4, n_layers=2),
             name="draft_mlp_b1"),
        # A small batch with the transformer head: width 2560, 8 heads, feed-forward 10240.
        dict(_draft("draft", "xfmr", "bf16", "f32", 8, 16, 151936, 2560, 10240, 2560, n_heads=8, max_pos=16),
             name="draft_xfmr_b8"),
        # Batched serving, the default GRU head (embedding 4096, state 1024, rank 256) with its input table.
        dict(_draft("draft", "gru", "bf16", "bf16", 64, 16, 151936, 4096, 1024, 256, table=True),
             name="draft_gru_b64"),
        # The same head without the table (its 1.9 GB not to spare), an odd batch and block, per-position weights.
        dict(_draft("draft", "gru", "bf16", "f32", 27, 11, 50008, 4096, 1024, 256, table=False, per_position=True),
             name="draft_gru_plain_ragged"),
        # A float32 GRU head, as a head is checked before it is rounded to bf16: 8 requests, 32000 tokens.
        dict(_draft("draft", "gru", "f32", "f32", 8, 8, 32000, 1024, 512, 256, table=False), name="draft_gru_f32"),
        # Batched serving at temperature 1: drafting with Gumbel-max draws ...
        dict(_draft("draft_sampled", "gru", "bf16", "bf16", 64, 16, 151936, 4096, 1024, 256, table=True),
             name="draft_sampled_b64"),
        # ... and the lossless verification of that block.
        dict(_draft("verify_sampled", "gru", "bf16", "bf16", 64, 16, 151936, 4096, 1024, 256, table=True),
             name="verify_sampled_b64"),
        # Fusing two sets of precomputed logits for 64 blocks of 16 positions.
        dict(kind="combine", rows=1024, V=151936, ldtype="bf16", weight=0.5, short=True, prior=True,
             name="combine_bf16_1024"),
        # Greedy verification of 64 blocks of 16 drafted tokens.
        dict(kind="verify", B=64, n=16, V=151936, ldtype="bf16", name="verify_bf16_b64"),
        # The unigram prior of a chat corpus of 2^28 positions.
        dict(kind="prior", N=1 << 28, V=151936, name="prior_corpus"),
        # Loading a set of GRU weights: the input table of the full vocabulary.
        dict(kind="input_table", V=151936, d_model=4096, d_hidden=1024, name="input_table"),
    ]


# ------------------------------------------------------------------ drawing

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng):
    return rng.choice([32000, 50008, 128256, 151936, 8 * _log_int(rng, 1000, 18992)])


def draw(rng):
    kind = rng.choice(["draft", "draft", "draft", "draft", "draft_sampled", "verify_sampled", "combine", "combine",
                       "verify", "verify", "prior", "input_table"])
    ld = rng.choice(["f32", "bf16"])
    if kind in ("draft", "draft_sampled", "verify_sampled"):
        head = rng.choice(["gru", "gru", "mlp", "xfmr", "markov"])
        n = rng.randint(2, 20)
        if head != "xfmr" and rng.random() < 0.3:
            # float32 heads: few requests, smaller vocabularies and widths
            d = 16 * _log_int(rng, 4, 64)
            r = 16 * _log_int(rng, 4, 32)
            h = d if head == "mlp" else 16 * _log_int(rng, 4, 32)
            c = _draft(kind, head, "f32", ld, rng.randint(1, 16), min(n, 12), 8 * _log_int(rng, 128, 4000),
                       r if head == "markov" else d, h, h if head == "mlp" else r, window=rng.randint(1, 4),
                       n_layers=rng.randint(1, 2), table=False)
        else:
            B = _log_int(rng, 1, 128)
            V = _vocab(rng)
            if head == "gru":
                h = 16 * _log_int(rng, 16, 96)
                c = _draft(kind, head, "bf16", ld, B, n, V, 64 * _log_int(rng, 8, 64), h, 16 * _log_int(rng, 8, 32),
                           table=rng.random() < 0.6)
            elif head == "mlp":
                h = 64 * _log_int(rng, 4, 24)
                c = _draft(kind, head, "bf16", ld, B, n, V, 64 * _log_int(rng, 4, 24), h, h,
                           window=rng.randint(1, 4), n_layers=rng.randint(1, 2))
            elif head == "xfmr":
                heads = rng.choice([4, 8, 16])
                d = heads * 16 * rng.randint(4, 10)
                c = _draft(kind, head, "bf16", ld, B, n, V, d, 64 * _log_int(rng, 8, 128), d, n_heads=heads,
                           max_pos=rng.randint(20, 32))
            else:
                r = 16 * _log_int(rng, 8, 64)
                c = _draft(kind, head, "bf16", ld, B, n, V, r, r, r)
        c["weight"] = round(rng.uniform(0.1, 1.0), 3)
        c["per_position"] = rng.random() < 0.3
        return c
    if kind == "combine":
        V = rng.choice([32000, 151936, 32003, _log_int(rng, 1000, 151936)])
        rows = _log_int(rng, 1, min(8192, 2 ** 28 // V))
        return dict(kind=kind, rows=rows, V=V, ldtype=ld, weight=rng.choice([0.0, 0.5, 1.0]), short=rng.random() < 0.8,
                    prior=rng.random() < 0.8)
    if kind == "verify":
        n = rng.choice([4, 7, 8, 16, 32])
        V = rng.choice([32000, 151936, 50257, _log_int(rng, 1000, 151936)])
        B = _log_int(rng, 1, max(1, min(256, 2 ** 29 // (V * (n + 1)))))
        return dict(kind=kind, B=B, n=n, V=V, ldtype=ld)
    if kind == "prior":
        return dict(kind=kind, N=_log_int(rng, 1 << 14, 1 << 28) | 1, V=_log_int(rng, 1000, 200000))
    return dict(kind=kind, V=_log_int(rng, 4000, 151936), d_model=64 * _log_int(rng, 8, 64),
                d_hidden=16 * _log_int(rng, 16, 64))


# ------------------------------------------------------------------- inputs

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _normal(shape, std, g, dtype):
    x = torch.randn(*shape, generator=g, device=DEV)
    return x.mul_(std).to(TORCH[dtype])


def _weights(c, seed):
    g, V, dt = _gen(seed, 1), c["V"], c["wdtype"]
    D, H, R = c["d_model"], c["d_hidden"], c["d_rank"]

    def lin(out, fan):
        return _normal((out, fan), 1.0 / math.sqrt(fan), g, dt)

    w = {"emb": _normal((V, R if c["head"] == "markov" else D), 1.0, g, dt), "w_vocab": lin(V, R)}
    if c["head"] == "gru":
        w.update(w_ih=lin(3 * H, D), w_hh=lin(3 * H, H), w_rank=lin(R, H))
    elif c["head"] == "mlp":
        w["w1"] = lin(H, c["window"] * D)
        if c["n_layers"] == 2:
            w["w2"] = lin(H, H)
    elif c["head"] == "xfmr":
        w["pos"] = _normal((c["max_pos"], D), 1.0, g, dt)
        for k in ("wq", "wk", "wv", "wo"):
            w[k] = lin(D, D)
        w.update(w1=lin(H, D), w2=lin(D, H))
    return w


def _log_prior(V, seed):
    """log of a Zipf(1.1) unigram law over a shuffled vocabulary, add-one smoothed."""
    rank = torch.randperm(V, generator=_gen(seed, 2), device=DEV).double()
    q = (rank + 1.0).pow(-1.1)
    n = torch.floor(q / q.sum() * 1e7) + 1.0
    return torch.log(n / n.sum()).float().contiguous()


def _peak(rows, ids, g):
    """Sets one entry of each row 0.5 to 8 above the row's largest."""
    top = rows.amax(-1, keepdim=True)
    lift = torch.rand(top.shape, generator=g, device=DEV) * 7.5 + 0.5
    return rows.scatter_(-1, ids.unsqueeze(-1), top + lift)


def _rows(shape, V, dtype, g):
    """Logit rows [*shape, V] and the likely token of each."""
    ids = torch.randint(0, V, tuple(shape), generator=g, device=DEV)
    x = torch.empty(*shape, V, dtype=TORCH[dtype], device=DEV)
    flat, at, step = x.view(-1, V), ids.view(-1), max(1, (1 << 26) // V)
    for i in range(0, at.numel(), step):         # in pieces: float32 temporaries stay small
        k = min(at.numel(), i + step)
        r = torch.randn(k - i, V, generator=g, device=DEV).mul_(STD)
        flat[i:k] = _peak(r, at[i:k], g).to(x.dtype)
    return x, ids


def _target(long, ids, g):
    """Target rows [B, n + 1, V]: the drafter's rows plus N(0, 1), with its likely token kept
    three times out of four; the last row is a row of its own."""
    B, n, V = long.shape
    t = torch.empty(B, n + 1, V, dtype=long.dtype, device=DEV)
    other = torch.randint(0, V, (B, n + 1), generator=g, device=DEV)
    keep = torch.rand(B, n + 1, generator=g, device=DEV) < 0.75
    for b in range(B):
        r = torch.randn(n + 1, V, generator=g, device=DEV)
        r[:n] += long[b].float().clamp(max=4.5 * STD)
        r[n] *= STD
        like = torch.cat([ids[b], other[b, n:]])
        t[b] = _peak(r, torch.where(keep[b], like, other[b]), g).to(t.dtype)
    return t


def _fusion(c):
    """alpha, beta: one weight, or a pair for each position that falls along the block."""
    if not c.get("per_position"):
        return c["weight"], c["weight"]
    n = c["n"]
    return ([c["weight"] * (1.0 - 0.5 * j / n) for j in range(n)],
            [c["weight"] * (0.8 - 0.4 * j / n) for j in range(n)])


def _corpus(c, seed):
    """Ids from a Zipf(1.1) law over a shuffled vocabulary; spans of user text (mask 0) and of
    assistant text (mask 1), about three quarters masked in."""
    N, V, g = c["N"], c["V"], _gen(seed, 7)
    by_rank = torch.randperm(V, generator=g, device=DEV).to(torch.int32)
    cdf = torch.cumsum((torch.arange(V, device=DEV, dtype=torch.float64) + 1.0).pow(-1.1), 0)
    cdf = (cdf / cdf[-1]).float()
    tokens = torch.empty(N, dtype=torch.int32, device=DEV)
    for a in range(0, N, 1 << 26):
        u = torch.rand(min(N, a + (1 << 26)) - a, generator=g, device=DEV)
        tokens[a:a + u.numel()] = by_rank[torch.searchsorted(cdf, u).clamp_(max=V - 1)]
    spans = N // 128 + 2
    lens = torch.randint(8, 257, (spans,), generator=g, device=DEV)
    lens[1::2] = torch.randint(16, 769, (spans // 2,), generator=g, device=DEV)
    mask = torch.repeat_interleave(torch.arange(spans, device=DEV) & 1, lens)
    mask = mask.to(torch.uint8).repeat(N // mask.numel() + 1)[:N].contiguous()
    return tokens, mask


def _zeros(nbytes):
    return torch.zeros(nbytes, dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c, "seed": int(seed) & ((1 << 62) - 1)}
    if kind in ("draft", "draft_sampled", "verify_sampled"):
        s["weights"] = _weights(c, seed)
        spec = Spec(c)
        if c.get("table"):
            s["weights"]["input_table"] = dels.gru_input_table(spec, s["weights"], c["V"])
        s["prior"] = _log_prior(c["V"], seed)
        s["long"], ids = _rows((c["B"], c["n"]), c["V"], c["ldtype"], _gen(seed, 3))
        s["alpha"], s["beta"] = _fusion(c)
        s["drafter"] = dels.Drafter(spec, s["weights"], c["B"], c["n"], c["V"])
        s["step"] = 1 + s["seed"] % 1000
        if kind == "verify_sampled":
            B, n, V = c["B"], c["n"], c["V"]
            s["target"] = _target(s["long"], ids, _gen(seed, 4))
            s["code"] = dels.dtype_code(s["target"])
            tok, lp, _, s["state"] = s["drafter"].sample(s["long"], s["prior"], s["alpha"], s["beta"], s["seed"],
                                                         s["step"])
            s["draft"], s["draft_lp"] = tok, lp
            s["alphas"], s["betas"] = ([x] * n if isinstance(x, float) else x for x in (s["alpha"], s["beta"]))
            s["bytes"] = dels.dels_verify_sampled_workspace_bytes(s["drafter"].head, B, n, V, s["code"])
            s["ws"] = _zeros(s["bytes"])
            s["accept"], s["bonus"] = (torch.empty(B, dtype=torch.int32, device=DEV) for _ in range(2))
            s["gap"] = torch.empty(B, dtype=torch.float32, device=DEV)
    elif kind == "combine":
        rows, V = c["rows"], c["V"]
        g = _gen(seed, 3)
        s["long"] = _rows((rows,), V, c["ldtype"], g)[0]
        s["short"] = None
        if c["short"]:
            s["short"] = torch.empty_like(s["long"])
            for i in range(0, rows, 256):
                k = min(rows, i + 256)
                s["short"][i:k] = torch.randn(k - i, V, generator=g, device=DEV).mul_(STD)
        s["prior"] = _log_prior(V, seed) if c["prior"] else None
        s["code"] = dels.dtype_code(s["long"])
        s["bytes"] = dels.dels_combine_workspace_bytes(rows, V, s["code"])
        s["ws"] = _zeros(s["bytes"])
        s["token"] = torch.empty(rows, dtype=torch.int32, device=DEV)
        s["lp"], s["gap"] = (torch.empty(rows, dtype=torch.float32, device=DEV) for _ in range(2))
    elif kind == "verify":
        B, n, V, g = c["B"], c["n"], c["V"], _gen(seed, 3)
        s["target"], ids = _rows((B, n + 1), V, c["ldtype"], g)
        off = torch.rand(B, n, generator=g, device=DEV) < 0.25
        other = torch.randint(0, V, (B, n), generator=g, device=DEV)
        s["draft"] = torch.where(off, other, ids[:, :n]).to(torch.int32).contiguous()
        s["code"] = dels.dtype_code(s["target"])
        s["bytes"] = dels.dels_verify_workspace_bytes(B, n, V, s["code"])
        s["ws"] = _zeros(s["bytes"])
        s["accept"], s["bonus"] = (torch.empty(B, dtype=torch.int32, device=DEV) for _ in range(2))
        s["argmax"] = torch.empty(B, n + 1, dtype=torch.int32, device=DEV)
    elif kind == "prior":
        N, V = c["N"], c["V"]
        s["tokens"], s["mask"] = _corpus(c, seed)
        s["bytes"] = dels.dels_prior_workspace_bytes(V, N)
        s["ws"] = _zeros(s["bytes"])
        s["out"] = torch.empty(V, dtype=torch.float32, device=DEV)
        s["counts"] = torch.empty(V, dtype=torch.int64, device=DEV)
        s["tally"] = torch.empty(2, dtype=torch.int64, device=DEV)
    else:
        s["weights"], s["head"] = _table_head(c, seed)
        s["bytes"] = dels.dels_gru_input_table_bytes(s["head"], c["V"])
        s["table"] = torch.empty(c["V"], 3 * c["d_hidden"], dtype=torch.float32, device=DEV)
        s["ws"] = _zeros(256)
    return s


def _table_head(c, seed):
    full = dict(c, head="gru", wdtype="bf16", d_rank=16, window=0)
    w = _weights(full, seed)
    return w, dels.make_head(Spec(full), w)


def _ok(code):
    if code != 0:
        raise RuntimeError(dels.dels_status_string(code))


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "draft":
        return s["drafter"](s["long"], s["prior"], s["alpha"], s["beta"])
    if kind == "draft_sampled":
        return s["drafter"].sample(s["long"], s["prior"], s["alpha"], s["beta"], s["seed"], s["step"])[:3]
    if kind == "verify_sampled":
        _ok(dels.dels_verify_block_sampled(
            s["drafter"].head, s["draft"], s["draft_lp"], s["state"], s["long"], s["code"], s["prior"], s["alphas"],
            s["betas"], s["target"], s["code"], c["B"], c["n"], c["V"], s["seed"], s["step"], s["accept"], s["bonus"],
            s["gap"], s["ws"], s["bytes"]))
        return s["accept"], s["bonus"], s["gap"]
    if kind == "combine":
        _ok(dels.dels_combine_argmax(s["long"], s["short"], s["code"], s["prior"], c["weight"], c["weight"],
                                     c["rows"], c["V"], s["token"], s["lp"], s["gap"], s["ws"], s["bytes"]))
        return s["token"], s["lp"], s["gap"]
    if kind == "verify":
        _ok(dels.dels_verify_block(s["draft"], s["target"], s["code"], c["B"], c["n"], c["V"], s["accept"], s["bonus"],
                                   s["argmax"], s["ws"], s["bytes"]))
        return s["accept"], s["bonus"], s["argmax"]
    if kind == "prior":
        _ok(dels.dels_prior_estimate(s["tokens"], s["mask"], c["N"], c["V"], 1.0, s["out"], s["counts"], s["tally"],
                                     s["ws"], s["bytes"]))
        return s["out"], s["counts"], s["tally"]
    _ok(dels.dels_gru_build_input_table(s["head"], c["V"], s["table"], s["bytes"], s["ws"], 256))
    return s["table"]


# --------------------------------------------------------------------- work

def work(case):
    c, kind = case, case["kind"]
    V = c["V"]
    es = 2 if c.get("ldtype") == "bf16" else 4
    if kind in ("draft", "draft_sampled", "verify_sampled"):
        B, n, D, H, R = c["B"], c["n"], c["d_model"], c["d_hidden"], c["d_rank"]
        ws = 2 if c["wdtype"] == "bf16" else 4
        if kind == "verify_sampled":
            # the target rows, one drafter's row per request, the prior and the vocabulary matrix
            return {"bytes": B * (n + 2) * V * es + V * 4 + V * R * ws + B * n * (8 + R * ws),
                    "flops": 2 * B * V * R + 8 * B * (n + 1) * V}
        per = {"gru": R * H + 3 * H * H + (0 if c.get("table") else 3 * H * D),
               "mlp": c.get("window", 0) * D * H + (H * H if c.get("n_layers") == 2 else 0),
               "xfmr": 4 * D * D + 2 * D * H, "markov": 0}[c["head"]] + V * R
        # the next position's products wait for this position's token: a head that does not fit
        # in the L2 cache is read again at each position
        times = n - 1 if per * ws > L2_BYTES else min(1, n - 1)
        row = B * (n - 1) * (3 * H * 4 if c.get("table") else (R if c["head"] == "markov" else D) * ws)
        return {"bytes": B * n * V * es + V * 4 + times * per * ws + row + B * n * 12,
                "flops": (n - 1) * 2 * B * per + 8 * B * n * V}
    if kind == "combine":
        return {"bytes": c["rows"] * V * es * (2 if c["short"] else 1) + (V * 4 if c["prior"] else 0) + c["rows"] * 12,
                "flops": 8 * c["rows"] * V}
    if kind == "verify":
        return {"bytes": c["B"] * (c["n"] + 1) * (V * es + 4), "flops": c["B"] * (c["n"] + 1) * V}
    if kind == "prior":
        return {"bytes": 5 * c["N"] + 12 * V, "flops": c["N"]}
    D, H = c["d_model"], c["d_hidden"]
    return {"bytes": V * D * 2 + 3 * H * D * 2 + V * 3 * H * 4, "flops": 2 * V * D * 3 * H}


def tolerance(case):
    """About four times what the outputs differ from ``exact`` by, at the case where that is most."""
    kind = case["kind"]
    if kind == "verify":
        return "exact"                     # whole numbers from stored values
    if kind == "prior":
        # counts are exact, the logarithm is taken in float64 and stored as float32 (2e-8 seen)
        return {"rel": 1e-7, "max": 3e-7, "differ": 0.0}
    if kind == "input_table":
        return {"rel": 2e-5, "max": 2e-4}  # float32 sums of 4096 exact products (4e-6 seen)
    if kind == "combine" or case["wdtype"] == "f32":
        return {"rel": 5e-6, "max": 5e-5, "differ": 0.01}   # float32 sums (4e-7 to 7e-7 seen)
    # bf16 activations: one next to a rounding boundary lands on either side of it with the order
    # of a float32 sum, and moves single log-probabilities by up to 1e-3 (7e-5 seen over a block)
    return {"rel": 3e-4, "max": 1e-2, "differ": 0.01}


# ------------------------------------------------------ the same in 64 bits

def _bf16(x):
    return x.to(torch.bfloat16).double()


def _gelu(x):
    return 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))


def _rms(x):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + 1e-6)


def _mm(x, w, chunk=1 << 15):
    """x W^T in float64, over row blocks of W to bound memory."""
    return torch.cat([x @ w[i:i + chunk].double().t() for i in range(0, w.shape[0], chunk)], 1)


class _Head64:
    """The local head of Appendix A and its stand-ins, in float64; bf16 heads round the activations
    that feed a bf16 product (the transformer head's only on the way into the vocabulary)."""

    def __init__(self, c, w):
        self.c, self.w = c, w
        self.act = _bf16 if c["wdtype"] == "bf16" else (lambda x: x)
        self.hist, self.h = [], None

    def feature(self, tok):
        c, w, act = self.c, self.w, self.act
        self.hist.append(tok.long())
        e = w["emb"][self.hist[-1]].double()
        if c["head"] == "markov":
            return e
        if c["head"] == "gru":
            H = c["d_hidden"]
            h = torch.zeros(e.shape[0], H, dtype=torch.float64, device=DEV) if self.h is None else self.h
            gi, gh = _mm(e, w["w_ih"]), _mm(act(h), w["w_hh"])
            r, z = (torch.sigmoid(gi[:, k * H:(k + 1) * H] + gh[:, k * H:(k + 1) * H]) for k in (0, 1))
            self.h = (1 - z) * torch.tanh(gi[:, 2 * H:] + r * gh[:, 2 * H:]) + z * h
            x = _mm(act(self.h), w["w_rank"])
            return act(x * torch.sigmoid(x))
        if c["head"] == "mlp":
            parts = [w["emb"][self.hist[-1 - k]].double() if k < len(self.hist) else torch.zeros_like(e)
                     for k in range(c["window"])]
            x = act(_gelu(_mm(torch.cat(parts, 1), w["w1"])))
            return act(_gelu(_mm(x, w["w2"]))) if c["n_layers"] == 2 else x
        D, nh, B, m = c["d_model"], c["n_heads"], e.shape[0], len(self.hist)
        t = torch.stack([w["emb"][x].double() for x in self.hist], 1) + w["pos"][:m].double()
        a = _rms(t)
        flat = a.reshape(B * m, D)
        q = _mm(a[:, -1], w["wq"]).view(B, nh, 1, -1)
        k = _mm(flat, w["wk"]).view(B, m, nh, -1).transpose(1, 2)
        v = _mm(flat, w["wv"]).view(B, m, nh, -1).transpose(1, 2)
        p = torch.softmax((q @ k.transpose(2, 3)) / math.sqrt(D // nh), -1)
        u = t[:, -1] + _mm((p @ v).reshape(B, D), w["wo"])
        return act(_rms(u + _mm(_gelu(_mm(_rms(u), w["w1"])), w["w2"])))


def _philox(seed, step, b, j, stream, block):
    """Output words of Philox4x32-10 (Salmon et al. 2011), key = seed, counter (block, step, b + 2^16 j + 2^24 stream, 0)."""
    x0, x1 = block, torch.full_like(block, step)
    x2, x3 = (b + (j << 16) + (stream << 24)).expand_as(block), torch.zeros_like(block)
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p, q = x0 * 0xD2511F53, x2 * 0xCD9E8D57        # 64-bit products, the top bit as a sign
        x0, x1, x2, x3 = ((q >> 32) & M32) ^ x1 ^ k0, q & M32, ((p >> 32) & M32) ^ x3 ^ k1, p & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return torch.stack([x0, x1, x2, x3], -1)


def _uniforms(s, B, j, stream, V):
    """Uniforms [B, V] of block position(s) j (a number or one per request)."""
    b = torch.arange(B, device=DEV).view(B, 1)
    j = torch.as_tensor(j, device=DEV).view(-1, 1)
    blocks = torch.arange((V + 3) // 4, device=DEV).expand(B, -1)
    w = _philox(s["seed"], s["step"], b, j, stream, blocks).reshape(B, -1)[:, :V]
    return ((w >> 9).double() + 0.5) / 2.0 ** 23


def _gumbel(s, B, j, stream, V):
    return -torch.log(-torch.log(_uniforms(s, B, j, stream, V)))


def _top2(x):
    v, i = x.topk(2, -1)
    return i[:, 0], v[:, 0] - v[:, 1]


def _block64(s, sampled):
    """The drafted block in float64: tokens, log-probabilities, gaps, and the fused rows of each position."""
    c = s["case"]
    B, n, V = c["B"], c["n"], c["V"]
    head = _Head64(c, s["weights"])
    al, be = ([x] * n if isinstance(x, float) else x for x in (s["alpha"], s["beta"]))
    toks, lps, gaps, rows = [], [], [], []
    for j in range(n):
        l = s["long"][:, j].double()
        if j:
            l = l + al[j] * _mm(head.feature(toks[-1]), s["weights"]["w_vocab"]) - be[j] * s["prior"].double()
        x, gap = _top2(l + _gumbel(s, B, j, 0, V)) if sampled else _top2(l)
        toks.append(x.to(torch.int32))
        lps.append(torch.log_softmax(l, -1).gather(1, x.view(-1, 1)).squeeze(1))
        gaps.append(gap)
        rows.append(l)
    return torch.stack(toks, 1), torch.stack(lps, 1), torch.stack(gaps, 1), rows


def _inputs(c, seed):
    """The inputs that ``prepare`` makes, without the library."""
    s = {"case": c, "seed": int(seed) & ((1 << 62) - 1), "weights": _weights(c, seed),
         "prior": _log_prior(c["V"], seed)}
    s["step"] = 1 + s["seed"] % 1000
    s["long"], s["ids"] = _rows((c["B"], c["n"]), c["V"], c["ldtype"], _gen(seed, 3))
    s["alpha"], s["beta"] = _fusion(c)
    return s


def exact(case, seed):
    c, kind = case, case["kind"]
    V = c["V"]
    if kind in ("draft", "draft_sampled"):
        return _block64(_inputs(c, seed), kind == "draft_sampled")[:3]
    if kind == "verify_sampled":
        s = _inputs(c, seed)
        B, n = c["B"], c["n"]
        tok, lp, _, rows = _block64(s, True)
        target = _target(s["long"], s["ids"], _gen(seed, 4))
        acc = torch.full((B,), n, dtype=torch.int64, device=DEV)
        for j in reversed(range(n)):
            p = torch.log_softmax(target[:, j].double(), -1).gather(1, tok[:, j:j + 1].long()).squeeze(1)
            u = _uniforms(s, B, j, 1, 1).squeeze(1)
            acc = torch.where(u < torch.exp(p - lp[:, j]), acc, torch.full_like(acc, j))
        keys = _gumbel(s, B, acc, 2, V)
        for b in range(B):
            a = int(acc[b])
            t = target[b, a].double()
            if a < n:
                w = torch.softmax(t, 0) - torch.softmax(rows[a][b], 0)
                keys[b] += torch.log(w.clamp(min=0))
            else:
                keys[b] += t
        bonus, gap = _top2(keys)
        return acc.to(torch.int32), bonus.to(torch.int32), gap
    if kind == "combine":
        rows, g = c["rows"], _gen(seed, 3)
        long = _rows((rows,), V, c["ldtype"], g)[0]
        prior = _log_prior(V, seed).double() if c["prior"] else None
        out = []
        for i in range(0, rows, 256):
            k = min(rows, i + 256)
            l = long[i:k].double()
            if c["short"]:
                l += c["weight"] * torch.randn(k - i, V, generator=g, device=DEV).mul_(STD).to(long.dtype).double()
            if prior is not None:
                l -= c["weight"] * prior
            x, gap = _top2(l)
            out.append((x.to(torch.int32), torch.log_softmax(l, -1).gather(1, x.view(-1, 1)).squeeze(1), gap))
        return tuple(torch.cat(x) for x in zip(*out))
    if kind == "verify":
        B, n, g = c["B"], c["n"], _gen(seed, 3)
        target, ids = _rows((B, n + 1), V, c["ldtype"], g)
        off = torch.rand(B, n, generator=g, device=DEV) < 0.25
        other = torch.randint(0, V, (B, n), generator=g, device=DEV)
        draft = torch.where(off, other, ids[:, :n])
        at = torch.arange(V, device=DEV)
        t = torch.stack([torch.where(r == r.amax(-1, keepdim=True), at, V).amin(-1) for r in target])
        acc = (draft == t[:, :n]).long().cumprod(1).sum(1)
        return acc.to(torch.int32), t.gather(1, acc.view(-1, 1)).squeeze(1).to(torch.int32), t.to(torch.int32)
    if kind == "prior":
        tokens, mask = _corpus(c, seed)
        counts = torch.zeros(V, dtype=torch.int64, device=DEV)
        for a in range(0, c["N"], 1 << 26):
            counts += torch.bincount(tokens[a:a + (1 << 26)][mask[a:a + (1 << 26)] != 0].long(), minlength=V)
        p = (counts.double() + 1.0) / (counts.sum().double() + V)
        return torch.log(p), counts, torch.stack([counts.sum(), torch.zeros_like(counts[0])])
    full = dict(c, head="gru", wdtype="bf16", d_rank=16, window=0)
    w = _weights(full, seed)
    ih = w["w_ih"].double().t()
    out = torch.empty(V, 3 * c["d_hidden"], dtype=torch.float64, device=DEV)
    for i in range(0, V, 1 << 14):
        out[i:i + (1 << 14)] = w["emb"][i:i + (1 << 14)].double() @ ih
    return out
