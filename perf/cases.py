"""The calls whose speed matters to a program that adapts a model in-episode
with this library, with inputs drawn as the synthetic workloads draw them.

A case is a dict of plain values with a "kind":

  weights   Eq. 8 / Eq. 9 loss weights of one update text against the
            episode's token history (attt_ngram_weights);
  history   an episode boundary and a refill: reset, append of a long token
            history, then the weights of an update text against it;
  texts     the update-text filter over an episode: reset, then one
            attt_repetition per update text (Eq. 6 / Eq. 7);
  ce        Eq. 10 and its gradient through the frozen LM head
            (attt_weighted_ce_fwd_bwd);
  lora      adapter gradients of the projections that share one input
            (attt_lora_grad);
  proj      the adapted projection of a chained update, forward and input
            gradient (attt_lora_forward, attt_lora_input_grad);
  episode   a chained episode: reset, two updates of five agent steps each
            with two AdamW gradient steps and dx, then the drift diagnostic
            (Episode.agent_step, Episode.drift, Episode.read_adapter);
  batch     concurrent episodes: reset, then two batched updates with two
            gradient steps and dx (Batch.update, Batch.read_adapter).

Ranges (draw): update texts of 32 to 8,192 tokens, vocabularies of 8,192 to
152,064, hidden sizes of 512 to 5,120, ranks 4 to 64, histories of 1,000 to
1,048,576 tokens, n-grams of 2 to 5.
"""
import math

import numpy as np
import torch

from paper_2607_03441_gb300 import attt

DEV = "cuda"
W_MIN = 0.05


def listed():
    return [
        # the weights of one short agent text early in an episode: latency
        {"name": "weights_short", "kind": "weights", "L": 211, "hist": 9001, "n": 3, "V": 152064, "frac": 0.3},
        # a long history rebuilt at an episode boundary, weights of a long text
        {"name": "history_1m", "kind": "history", "L": 8192, "hist": 1048576, "n": 4, "V": 128256, "frac": 0.3},
        # the sequence filter over an episode of a dozen 1,536-word texts
        {"name": "texts_episode", "kind": "texts", "updates": 12, "words": 1536, "vocab": 50000},
        # Eq. 10 at toy sizes: five launches' worth of latency
        {"name": "ce_tiny", "kind": "ce", "L": 256, "d": 512, "V": 8192},
        # Eq. 10 of one short agent text through a 7B-class head: the head is read for few rows
        {"name": "ce_short", "kind": "ce", "L": 93, "d": 3584, "V": 152064},
        # Eq. 10 of the 7B-class update
        {"name": "ce_7b", "kind": "ce", "L": 2048, "d": 3584, "V": 152064},
        # Eq. 10 of the 32B-class update, the largest call
        {"name": "ce_32b", "kind": "ce", "L": 8192, "d": 5120, "V": 152064},
        # adapter gradients of q and v of the 7B-class update
        {"name": "lora_7b_qv", "kind": "lora", "L": 2048, "din": 3584, "douts": "3584,512", "r": 16},
        # adapter gradients of q, k and v of the 32B-class update
        {"name": "lora_32b_qkv", "kind": "lora", "L": 8192, "din": 5120, "douts": "5120,1024,1024", "r": 64},
        # the adapted projection of a chained 7B-class update, both directions
        {"name": "proj_7b", "kind": "proj", "L": 2048, "din": 3584, "dout": 3584, "r": 16},
        # a chained episode on agent texts of a few hundred tokens
        {"name": "episode_7b", "kind": "episode", "L": 403, "din": 3584, "d": 3584, "V": 152064, "r": 16, "n": 4},
        # concurrent episodes with texts of different lengths
        {"name": "batch_7b", "kind": "batch", "E": 6, "L": 300, "din": 3584, "d": 3584, "V": 152064, "r": 16, "n": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo=512, hi=5120):
    """A hidden size: any multiple of 8 (the library's requirement)."""
    return 8 * _log_int(rng, lo // 8, hi // 8)


def draw(rng):
    kind = rng.choice(["weights", "history", "texts", "ce", "ce", "ce", "lora", "lora", "proj", "episode", "batch"])
    n, V = rng.choice([2, 3, 4, 5]), _log_int(rng, 8192, 152064)
    if kind in ("weights", "history"):
        return {"kind": kind, "L": _log_int(rng, 32, 8192), "hist": _log_int(rng, 1000, 1048576), "n": n, "V": V,
                "frac": round(rng.uniform(0.05, 0.6), 2)}
    if kind == "texts":
        return {"kind": kind, "updates": rng.randint(2, 32), "words": _log_int(rng, 40, 6000), "vocab": 50000}
    if kind == "ce":
        return {"kind": kind, "L": _log_int(rng, 32, 8192), "d": _width(rng), "V": V}
    if kind == "lora":
        douts = [_width(rng) for _ in range(rng.randint(1, 4))]
        return {"kind": kind, "L": _log_int(rng, 32, 8192), "din": _width(rng), "douts": ",".join(map(str, douts)),
                "r": rng.choice([4, 8, 12, 16, 32, 64])}
    din, d, r = _width(rng), _width(rng), rng.choice([8, 16, 32, 64])
    if kind == "proj":
        return {"kind": kind, "L": _log_int(rng, 32, 8192), "din": din, "dout": d, "r": r}
    if kind == "episode":
        return {"kind": kind, "L": _log_int(rng, 40, 1024), "din": din, "d": d, "V": V, "r": r, "n": n}
    return {"kind": kind, "E": rng.randint(2, 12), "L": _log_int(rng, 40, 400), "din": din, "d": d, "V": V, "r": r,
            "n": n}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

class _Rng:
    """Seeded draws on the GPU (the LM head's 0.8 G values among them)."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))

    def normal(self, shape, std=1.0, dtype=torch.bfloat16):
        """fp32 normal samples rounded once, in slabs of rows."""
        out = torch.empty(shape, dtype=dtype, device=DEV)
        flat = out.view(-1)
        for a in range(0, flat.numel(), 1 << 26):
            b = min(flat.numel(), a + (1 << 26))
            flat[a:b] = torch.randn(b - a, generator=self.g, device=DEV) * std
        return out

    def uniform(self, n):
        return torch.rand(n, generator=self.g, device=DEV, dtype=torch.float64)

    def states(self, W, tgt):
        """Hidden states of a model that knows some of the text: N(0, 1) plus a
        share of the target's and of another token's head row, so that their
        logits lie up to 16 above the rest (probabilities from 0 to nearly 1)."""
        L, d = tgt.numel(), W.shape[1]
        h = self.normal((L, d), dtype=torch.float32)
        for t in (tgt.long(), self.zipf(L, W.shape[0]).long()):
            h += (self.uniform(L) * 16 / (0.02 ** 2 * d)).float()[:, None] * W[t].float()
        return h.to(torch.bfloat16)

    def zipf(self, n, V):
        """Token ids of truncated Zipf(1.1), low ids the frequent ones."""
        cdf = torch.arange(1, V + 1, device=DEV, dtype=torch.float64).pow_(-1.1).cumsum_(0)
        u = self.uniform(n) * cdf[-1]
        return torch.searchsorted(cdf, u).clamp_(max=V - 1).to(torch.int32)

    def text(self, n, V, hist, frac):
        """An update text: Zipf ids, about `frac` of them in 16-token spans copied from `hist`."""
        x = self.zipf(n, V)
        m = hist.numel()
        if m < 32:
            return x
        at = torch.arange(n, device=DEV)
        span = at // 16
        k = int(span[-1]) + 1
        take = self.uniform(k) < frac
        src = (self.uniform(k) * (m - 16)).long()
        return torch.where(take[span], hist[src[span] + at % 16], x).contiguous()

    def weights(self, n):
        """Eq. 9 weights as a history gives them: 1 for new text, small for repeated text."""
        f = torch.floor(self.uniform(n).clamp_(min=1e-6).pow_(-0.7) - 1)
        return torch.clamp(1 / (1 + f), min=W_MIN).to(torch.float32)


def _texts(case, seed):
    """Update texts as bytes: Zipf words, the share copied from the text before rising over the episode."""
    g = np.random.default_rng(int(seed))
    letters = np.frombuffer(b"abcdefghijklmnopqrstuvwxyz0123456789._/()-:", dtype=np.uint8)
    size = case["vocab"]
    lens = g.integers(1, 13, size)
    chars = letters[g.integers(0, len(letters), int(lens.sum()))].tobytes()
    ends = np.cumsum(lens)
    cdf = np.cumsum(np.arange(1, size + 1, dtype=np.float64) ** -1.1)
    out, prev = [], None
    for u in range(case["updates"]):
        ids = np.minimum(np.searchsorted(cdf, g.random(case["words"]) * cdf[-1]), size - 1)
        if prev is not None:
            take = g.random(len(ids)) < 0.05 + 0.9 * u / case["updates"]
            ids = np.where(take, prev, ids)
        prev = ids
        seps = np.array([b" ", b" ", b" ", b" ", b"\n", b"\t", b"  ", b"\r\n"], dtype=object)[g.integers(0, 8, len(ids))]
        out.append(b"".join(chars[ends[i] - lens[i]:ends[i]] + s for i, s in zip(ids, seps)))
    return out


def _lens(case, seed):
    """Lengths of the update's parts: agent steps of an update, or episodes of a batch."""
    g = np.random.default_rng([int(seed), 7])
    k = 5 if case["kind"] == "episode" else case["E"]
    total = case["L"] if case["kind"] == "episode" else case["L"] * k
    cuts = np.sort(g.choice(np.arange(1, total), size=k - 1, replace=False))
    return [int(v) for v in np.diff(np.concatenate([[0], cuts, [total]]))]


def _douts(case):
    return [int(v) for v in case["douts"].split(",")]


def _scale(case):
    return 16.0 / case["r"]


def _inputs(case, seed):
    """The tensors of a case, from the seed alone."""
    k, g = case["kind"], _Rng(seed)
    s = {}
    if k in ("weights", "history"):
        s["hist"] = g.zipf(case["hist"], case["V"])
        s["tok"] = g.text(case["L"], case["V"], s["hist"], case["frac"])
    elif k == "ce":
        s["W"] = g.normal((case["V"], case["d"]), 0.02)
        s["tgt"] = g.zipf(case["L"], case["V"])
        s["h"] = g.states(s["W"], s["tgt"])
        s["w"] = g.weights(case["L"])
    elif k == "lora":
        L, din, r = case["L"], case["din"], case["r"]
        s["x"] = g.normal((L, din))
        s["dys"] = [g.normal((L, o)) for o in _douts(case)]
        s["As"] = [g.normal((din, r), 0.02) for _ in _douts(case)]
        s["Bs"] = [g.normal((r, o), 0.01) for o in _douts(case)]
    elif k == "proj":
        L, din, o, r = case["L"], case["din"], case["dout"], case["r"]
        s["x"], s["dy"] = g.normal((L, din)), g.normal((L, o))
        s["W0"] = g.normal((din, o), din ** -0.5)
        s["A"], s["B"] = g.normal((din, r), 0.02), g.normal((r, o), 0.01)
    elif k in ("episode", "batch"):
        din, d, V, r = case["din"], case["d"], case["V"], case["r"]
        rows = sum(_lens(case, seed))
        s["W0"], s["Wlm"] = g.normal((din, d), din ** -0.5), g.normal((V, d), 0.02)
        s["A0"] = g.normal((din, r), 0.02, torch.float32)
        s["B0"] = g.normal((r, d), 0.01, torch.float32)
        first = g.zipf(rows, V)
        s["tok"] = [first, g.text(rows, V, first, 0.4)]
        s["x"] = [g.normal((rows, din)) for _ in range(2)]
    return s


def _lr(case):
    return 5e-4


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"], k = case, case["kind"]
    empty = lambda *shape, dtype=torch.float32: torch.empty(*shape, dtype=dtype, device=DEV)  # noqa: E731
    ws = lambda n: empty(n, dtype=torch.uint8)  # noqa: E731
    if k in ("weights", "history"):
        s["H"] = attt.attt_history_create(case["n"], case["hist"])
        s["out"] = empty(case["L"])
        if k == "weights":
            attt.attt_history_insert(s["H"], s["hist"])
    elif k == "texts":
        texts = _texts(case, seed)
        s["texts"] = [torch.from_numpy(np.frombuffer(t, dtype=np.uint8).copy()).to(DEV) for t in texts]
        s["sets"] = attt.attt_wordsets_create(case["updates"], sum(len(t) for t in texts))
        s["rho_nu"] = [empty(2) for _ in texts]
        s["keep"] = [empty(1, dtype=torch.int32) for _ in texts]
    elif k == "ce":
        L, d, V = case["L"], case["d"], case["V"]
        s["loss"], s["dh"], s["lse"] = empty(1), empty(L, d), empty(L)
        s["ws"] = ws(attt.attt_ce_workspace_bytes(L, d, V))
    elif k == "lora":
        L, din, r = case["L"], case["din"], case["r"]
        s["dAs"] = [empty(din, r) for _ in _douts(case)]
        s["dBs"] = [empty(r, o) for o in _douts(case)]
        s["ws"] = ws(attt.attt_lora_workspace_bytes(L, din, _douts(case), r))
    elif k == "proj":
        L, din, o, r = case["L"], case["din"], case["dout"], case["r"]
        s["h"], s["dx"] = empty(L, o, dtype=torch.bfloat16), empty(L, din)
        s["ws"] = ws(max(attt.attt_lora_forward_workspace_bytes(L, din, o, r),
                         attt.attt_lora_input_grad_workspace_bytes(L, din, o, r)))
    else:
        lens = _lens(case, seed)
        rows = sum(lens)
        common = dict(n=case["n"], scale=_scale(case), lr=_lr(case), w_min=W_MIN, grad_steps=2)
        s["lens"] = lens
        s["dx"] = [empty(2, rows, case["din"]) for _ in range(2)]
        if k == "episode":
            s["ep"] = attt.Episode(s["W0"], s["Wlm"], s["A0"], s["B0"], max_history=65536, max_update=rows, cadence=5,
                                   optimizer="adamw", **common)
            s["losses"] = [empty(2) for _ in range(2)]
            s["kl"], s["kl_mean"] = empty(rows), empty(1)
            cuts = np.concatenate([[0], np.cumsum(lens)])
            s["steps"] = [[(t[a:b], x[a:b]) for a, b in zip(cuts[:-1], cuts[1:])] for t, x in zip(s["tok"], s["x"])]
        else:
            s["bt"] = attt.Batch(s["W0"], s["Wlm"], s["A0"], s["B0"], episodes=case["E"], max_history=65536,
                                 max_update=max(lens), **common)
            s["losses"] = [empty(case["E"], 2) for _ in range(2)]
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "weights":
        return attt.attt_ngram_weights(s["H"], s["tok"], W_MIN, out=s["out"])
    if k == "history":
        attt.attt_history_reset(s["H"])
        attt.attt_history_insert(s["H"], s["hist"])
        return attt.attt_ngram_weights(s["H"], s["tok"], W_MIN, out=s["out"])
    if k == "texts":
        attt.attt_wordsets_reset(s["sets"])
        for t, o, keep in zip(s["texts"], s["rho_nu"], s["keep"]):
            attt.attt_repetition(s["sets"], t, 0.5, out=o, keep=keep)
        # (rho, nu) of the texts, then the filter's decisions; a long episode
        # is joined so that it stays a handful of outputs
        return torch.stack(s["rho_nu"]), torch.cat(s["keep"])
    if k == "ce":
        loss, dh, lse = attt.attt_weighted_ce_fwd_bwd(s["h"], s["W"], s["tgt"], s["w"], loss=s["loss"], dh=s["dh"],
                                                      lse=s["lse"], workspace=s["ws"])
        return {"loss": loss, "dh": dh, "lse": lse}
    if k == "lora":
        dAs, dBs = attt.attt_lora_grad(s["x"], s["dys"], s["As"], s["Bs"], _scale(case), dAs=s["dAs"], dBs=s["dBs"],
                                       workspace=s["ws"])
        return {"dA": dAs, "dB": dBs}
    if k == "proj":
        h = attt.attt_lora_forward(s["x"], s["W0"], s["A"], s["B"], _scale(case), h=s["h"], workspace=s["ws"])
        dx = attt.attt_lora_input_grad(s["dy"], s["W0"], s["A"], s["B"], _scale(case), dx=s["dx"], workspace=s["ws"])
        return {"h": h, "dx": dx}
    if k == "episode":
        ep = s["ep"]
        ep.reset()
        for steps, losses, dx in zip(s["steps"], s["losses"], s["dx"]):
            for t, x in steps:
                ep.agent_step(t, x, losses=losses, dx=dx)
        kl, kl_mean = ep.drift(s["x"][1], kl=s["kl"], kl_mean=s["kl_mean"])
        A, B = ep.read_adapter()
        return {"losses": s["losses"], "dx": s["dx"], "kl": kl, "kl_mean": kl_mean, "A": A, "B": B}
    bt = s["bt"]
    bt.reset()
    for t, x, losses, dx in zip(s["tok"], s["x"], s["losses"], s["dx"]):
        bt.update(t, x, s["lens"], losses=losses, dx=dx)
    adapters = [bt.read_adapter(e) for e in range(case["E"])]
    return {"losses": s["losses"], "dx": s["dx"], "A": [a for a, _ in adapters], "B": [b for _, b in adapters]}


# --------------------------------------------------------------------------
# work and tolerance
# --------------------------------------------------------------------------

def work(case):
    k = case["kind"]
    if k == "weights":
        # the text in, one 8-byte table slot per window, the weights out
        return {"bytes": (4 + 8 + 4) * case["L"], "flops": 0}
    if k == "history":
        # tokens in, the stream and one 8-byte slot per n-gram out; then the weights
        return {"bytes": (4 + 4 + 8) * case["hist"] + 16 * case["L"], "flops": 0}
    if k == "texts":
        # the bytes in (about 7.7 per word), their copy out, one 16-byte slot per word
        return {"bytes": case["updates"] * case["words"] * (2 * 7.7 + 16), "flops": 0}
    if k == "ce":
        L, d, V = case["L"], case["d"], case["V"]
        return {"bytes": 2 * L * d + 2 * V * d + 8 * L + 4 * L * d + 4 * L, "flops": 4 * L * V * d}
    if k == "lora":
        L, din, r, o = case["L"], case["din"], case["r"], _douts(case)
        adapters = r * (din * len(o) + sum(o))
        return {"bytes": 2 * L * (din + sum(o)) + 6 * adapters, "flops": 4 * L * r * (din * len(o) + sum(o))}
    if k == "proj":
        L, din, o, r = case["L"], case["din"], case["dout"], case["r"]
        return {"bytes": 2 * L * (din + o) * 2 + 2 * L * din + 2 * din * o + 2 * r * (din + o),
                "flops": 4 * L * din * o + 4 * L * r * (din + o)}
    din, d, V, r = case["din"], case["d"], case["V"], case["r"]
    E = case.get("E", 1)
    rows = case["L"] * E
    # two updates of two gradient steps: forward, Eq. 10, adapter gradients, dx
    step = 4 * rows * V * d + 4 * rows * din * d + 8 * rows * r * (din + d)
    drift = 4 * rows * V * d + 4 * rows * din * d if k == "episode" else 0
    return {"bytes": 2 * V * d + 2 * din * d + 2 * 2 * rows * din + 4 * 4 * rows * din + 8 * E * r * (din + d),
            "flops": 4 * step + drift}


def tolerance(case):
    k = case["kind"]
    if k in ("weights", "history", "texts"):
        return "exact"
    if k == "ce":
        return {"rel": 1e-2}  # bf16 softmax block in the dh contraction
    if k == "lora":
        return {"rel": 1e-2}  # u and v rounded to bf16
    if k == "proj":
        return {"rel": 1e-2}  # h in bf16
    return {"rel": 2e-2}


# --------------------------------------------------------------------------
# 64-bit references
# --------------------------------------------------------------------------

_EXACT_FLOPS = 6e12  # about five seconds of 64-bit matrix products


def _counts(hist, tok, n):
    """count(tok[s .. s+n), hist) for every window, by joining equal n-grams."""
    def grams(t):
        return np.stack([t[i:len(t) - n + 1 + i] for i in range(n)], axis=1)
    if len(tok) < n:
        return np.zeros(0, dtype=np.int64)
    q = grams(tok)
    if len(hist) < n:
        return np.zeros(len(q), dtype=np.int64)
    both = np.ascontiguousarray(np.concatenate([grams(hist), q])).astype(np.uint64)
    key = both[:, 0].copy()
    for i in range(1, n):  # ids of the distinct prefixes, so that the join stays exact
        _, key = np.unique(key * np.uint64(1 << 24) + both[:, i], return_inverse=True)
        key = key.astype(np.uint64)
    _, key = np.unique(key, return_inverse=True)
    m = len(both) - len(q)
    return np.bincount(key[:m], minlength=int(key.max()) + 1)[key[m:]]


def _weights64(hist, tok, n):
    c = _counts(hist, tok, n)
    f = np.zeros(len(tok), dtype=np.int64)
    for i in range(n):
        if len(c):
            f[i:i + len(c)] = np.maximum(f[i:i + len(c)], c)
    return np.maximum(W_MIN, 1.0 / (1.0 + f))


def _ce64(h, W, tgt, w, row_scale):
    """(nll rows, dh, lse) with h and the result in 64 bits, over slabs of the vocabulary."""
    L, V, slab = h.shape[0], W.shape[0], 16384
    z = torch.empty(L, V, dtype=torch.float64, device=DEV)
    for v in range(0, V, slab):
        z[:, v:v + slab] = h @ W[v:v + slab].double().t()
    lse = torch.logsumexp(z, dim=1)
    t = tgt.long()
    nll = lse - z.gather(1, t[:, None])[:, 0]
    z.sub_(lse[:, None]).exp_()
    dh = -W[t].double()
    for v in range(0, V, slab):
        dh += z[:, v:v + slab] @ W[v:v + slab].double()
    return nll, dh * (w * row_scale)[:, None], lse


def _adamw64(p, g, m, v, t, lr, b1=0.9, b2=0.999, eps=1e-8, wd=0.01):
    p.mul_(1 - lr * wd)
    m.mul_(b1).add_(g, alpha=1 - b1)
    v.mul_(b2).addcmul_(g, g, value=1 - b2)
    p.sub_(lr / (1 - b1 ** t) * m / ((v / (1 - b2 ** t)).sqrt() + eps))


def _episodes64(case, seed, adamw):
    """The episodes of an "episode" (one) or "batch" case."""
    s = _inputs(case, seed)
    lens, scale, lr = _lens(case, seed), _scale(case), _lr(case)
    if case["kind"] == "episode":
        lens = [sum(lens)]
    E, cuts = len(lens), np.concatenate([[0], np.cumsum(lens)])
    W0 = s["W0"].double()
    A = [s["A0"].double() for _ in lens]
    B = [s["B0"].double() for _ in lens]
    mom = [[torch.zeros_like(a), torch.zeros_like(a), torch.zeros_like(b), torch.zeros_like(b)] for a, b in zip(A, B)]
    past = [np.zeros(0, dtype=np.int32) for _ in lens]
    losses = [torch.zeros(E, 2, dtype=torch.float64) for _ in range(2)]
    dxs = [torch.empty(2, int(cuts[-1]), case["din"], dtype=torch.float64, device=DEV) for _ in range(2)]
    for u in range(2):
        for e in range(E):
            a, b = int(cuts[e]), int(cuts[e + 1])
            tok, x = s["tok"][u][a:b], s["x"][u][a:b].double()
            w = torch.from_numpy(_weights64(past[e], tok.cpu().numpy(), case["n"])).to(DEV)
            for g in range(2):
                h = x @ W0 + scale * (x @ A[e]) @ B[e]
                nll, dh, _ = _ce64(h, s["Wlm"], tok, w, 1.0 / (b - a))
                losses[u][e, g] = float((w * nll).mean())
                dxs[u][g, a:b] = dh @ W0.t() + scale * (dh @ B[e].t()) @ A[e].t()
                dA, dB = scale * x.t() @ (dh @ B[e].t()), scale * (x @ A[e]).t() @ dh
                if adamw:
                    t = 2 * u + g + 1
                    _adamw64(A[e], dA, mom[e][0], mom[e][1], t, lr)
                    _adamw64(B[e], dB, mom[e][2], mom[e][3], t, lr)
                else:
                    A[e], B[e] = A[e] - lr * dA, B[e] - lr * dB
            past[e] = np.concatenate([past[e], tok.cpu().numpy()])
    return s, W0, A, B, losses, dxs


def exact(case, seed):
    k = case["kind"]
    if k in ("weights", "history"):
        s = _inputs(case, seed)
        return _weights64(s["hist"].cpu().numpy(), s["tok"].cpu().numpy(), case["n"])
    if k == "texts":
        seen, rows, keep = [], [], []
        for t in _texts(case, seed):
            words = set(t.split())
            rho = max((len(words & o) / len(words | o) for o in seen if words | o), default=0.0)
            rows.append([rho, 1.0 - rho])
            keep.append(0 if 1.0 - rho < 0.5 else 1)
            seen.append(words)
        return np.array(rows), np.array(keep, dtype=np.int32)
    if work(case)["flops"] > _EXACT_FLOPS:
        return None
    if k == "ce":
        s = _inputs(case, seed)
        L = case["L"]
        w = s["w"].double()
        nll, dh, lse = _ce64(s["h"].double(), s["W"], s["tgt"], w, 1.0 / L)
        return {"loss": (w * nll).mean().reshape(1), "dh": dh, "lse": lse}
    if k == "lora":
        s, scale = _inputs(case, seed), _scale(case)
        x = s["x"].double()
        out = {"dA": [], "dB": []}
        for dy, A, B in zip(s["dys"], s["As"], s["Bs"]):
            dy, A, B = dy.double(), A.double(), B.double()
            out["dA"].append(scale * x.t() @ (dy @ B.t()))
            out["dB"].append(scale * (x @ A).t() @ dy)
        return out
    if k == "proj":
        s, scale = _inputs(case, seed), _scale(case)
        x, dy, W0, A, B = (s[q].double() for q in ("x", "dy", "W0", "A", "B"))
        return {"h": x @ W0 + scale * (x @ A) @ B, "dx": dy @ W0.t() + scale * (dy @ B.t()) @ A.t()}
    s, W0, A, B, losses, dxs = _episodes64(case, seed, k == "episode")
    if k == "batch":
        return {"losses": losses, "dx": dxs, "A": A, "B": B}
    x = s["x"][1].double()
    hq = x @ W0
    hp = hq + _scale(case) * (x @ A[0]) @ B[0]
    Wd = s["Wlm"].double()
    lp, lq = torch.log_softmax(hp @ Wd.t(), dim=1), torch.log_softmax(hq @ Wd.t(), dim=1)
    kl = (lp.exp() * (lp - lq)).sum(dim=1)
    return {"losses": [v[0] for v in losses], "dx": dxs, "kl": kl, "kl_mean": kl.mean().reshape(1), "A": A[0],
            "B": B[0]}
