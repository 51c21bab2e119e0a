"""Performance cases of one refine step, through the calls a user's program makes.

listed() names the cases; draw() gives further ones of the same ranges. Every
case is one of eight operations:

  attn    dlm_bidir_attn: full attention of a batch of drafts (bf16 or fp32)
  masked  dlm_attn_masked: block-causal drafting or block-local refinement
  vocab   dlm_vocab_confidence: reduction of a step's logits, from the one row
          of a single position and the 64 rows of a local window to whole batches
  step    dlm_refine_step: reduction and update of a whole batch in one launch
  update  dlm_refine_update / dlm_refine_update_ranked on given predictions
  prob    dlm_token_prob: probability of each position's current token
  lmhead  dlm_lmhead_confidence: output projection fused with the reduction
  loop    a recorded pass (attention, then dlm_refine_step in place) repeated
          on the GPU until no confident edit remains: the whole call

Shapes are those of the package's workloads (32/4 and 16/2 heads, head_dim 128,
V = 151552, sequences of 512 to 2048, a 2048-wide output projection), of its
tests (odd vocabularies, head_dim 64, MHA, ragged lengths) and generic ones
between them.
"""
import math

import torch

from paper_2608_02625_gb300 import binding as B

_DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
_V = 151552            # the workloads' vocabulary
_TAU, _REMASK = 0.8, 0.1


def _attn(name, B_, L, Hq, Hkv, D, dtype, lo, hi, resp, **kw):
    return dict(name=name, op="attn", B=B_, L=L, Hq=Hq, Hkv=Hkv, D=D, dtype=dtype, lo=lo, hi=hi, resp=resp, **kw)


def listed():
    return [
        # One sequence of 128 prompt + 384 response positions: the smallest
        # attention call a refiner serving a single request makes per layer.
        _attn("attn_1x512", 1, 512, 32, 4, 128, "bf16", 128, 128, 384, packed=False),
        # The batched refine step: 32 drafts of ragged lengths, padded to 512.
        _attn("attn_32x512", 32, 512, 32, 4, 128, "bf16", 64, 256, 384, packed=False),
        # Long drafts (512 + 1536); q, k, v are views of one packed projection.
        _attn("attn_8x2048", 8, 2048, 32, 4, 128, "bf16", 512, 512, 1536, packed=True),
        # fp32 attention of one sequence: checking a model at full precision.
        _attn("attn_f32_1x512", 1, 512, 32, 4, 128, "f32", 128, 128, 384, packed=False),
        # Block-causal attention in blocks of 64: the drafter's own pattern.
        dict(name="causal_32x512", op="masked", B=32, L=512, Hq=32, Hkv=4, D=128, dtype="bf16", lo=64, hi=256,
             resp=384, packed=False, mode=1, block=64),
        # The 64 rows of one local refinement window.
        dict(name="vocab_64", op="vocab", N=64, V=_V, dtype="bf16", pad=False),
        # One sequence under an odd vocabulary, rows packed without padding
        # (every second row starts off a 16-byte, even off a 4-byte boundary).
        dict(name="vocab_odd_512", op="vocab", N=512, V=151553, dtype="bf16", pad=False),
        # The whole batch's reduction and update: the largest stream of a step.
        dict(name="step_32x512", op="step", B=32, L=512, V=_V, dtype="bf16", lo=64, hi=256, resp=384),
        # The update of eight long drafts, on predictions already made.
        dict(name="update_8x2048", op="update", B=8, L=2048, V=_V, lo=512, hi=512, resp=1536, ranked=False),
        # Output projection of one local window: bound by reading the weight.
        dict(name="lmhead_64", op="lmhead", N=64, V=_V, d=2048),
        # Output projection of a batch of responses: bound by the tensor cores.
        dict(name="lmhead_4096", op="lmhead", N=4096, V=_V, d=2048),
        # One request from draft to refined response, as a serving loop runs it.
        dict(name="loop_1x512", op="loop", B=1, L=512, Hq=32, Hkv=4, D=128, V=_V, dtype="bf16", lo=128, hi=128,
             resp=384, passes=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lens(rng, L):
    hi = rng.randint(0, L // 2)
    return dict(lo=rng.randint(0, hi), hi=hi, resp=rng.randint(max(1, L // 4), L))


def draw(rng):
    op = rng.choice(["attn", "attn", "attn", "masked", "masked", "vocab", "vocab", "vocab", "step", "update",
                     "prob", "lmhead", "lmhead", "loop"])
    if op in ("attn", "masked"):
        Hq, Hkv = rng.choice([(32, 4), (16, 2), (8, 2), (8, 8), (12, 4), (4, 1)])
        D = rng.choice([128, 128, 64])
        dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
        L = _log(rng, 16, 2560 if dtype == "bf16" else 600)
        # no more than the listed cases' (query, key) pairs times heads and width
        most = 8 * 2048 ** 2 * 32 * 128 if dtype == "bf16" else 512 ** 2 * 32 * 128
        B_ = _log(rng, 1, max(1, min(128, most // (L * L * Hq * D))))
        c = dict(op=op, B=B_, L=L, Hq=Hq, Hkv=Hkv, D=D, dtype=dtype, packed=rng.random() < 0.3, **_lens(rng, L))
        if op == "masked":
            c.update(mode=rng.choice([1, 2]), block=rng.choice([7, 32, 64, 64, 64, 100, 128]))
        return c
    V = rng.choice([_V, _V, _log(rng, 1000, 151553), _log(rng, 1000, 151553)])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    if op in ("vocab", "prob"):
        most = 10 ** 8 if dtype == "bf16" else 5 * 10 ** 7
        return dict(op=op, N=_log(rng, 1, min(16384, most // V)), V=V, dtype=dtype, pad=rng.random() < 0.3)
    if op == "step":
        L = _log(rng, 32, 1024)
        return dict(op=op, B=_log(rng, 1, max(1, min(64, 10 ** 8 // (L * V)))), L=L, V=V, dtype=dtype, **_lens(rng, L))
    if op == "update":
        L = _log(rng, 16, 8192)
        return dict(op=op, B=_log(rng, 1, 128), L=L, V=V, ranked=rng.random() < 0.4, **_lens(rng, L))
    if op == "lmhead":
        d = rng.choice([512, 1024, 2048, 2048, 4096])
        return dict(op=op, N=_log(rng, 1, 4096 * 2048 // max(d, 2048)), V=V, d=d)
    L = _log(rng, 64, 640)
    Hq, Hkv = rng.choice([(32, 4), (16, 2)])
    return dict(op=op, B=_log(rng, 1, 4), L=L, Hq=Hq, Hkv=Hkv, D=128, V=min(V, 60000), dtype="bf16", passes=4,
                **_lens(rng, L))


# ---------------------------------------------------------------- inputs

def _bounds(c):
    """Prompt and sequence lengths (p_b, n_b): prompts spread over [lo, hi], n_b = min(L, p_b + resp)."""
    out = []
    for b in range(c["B"]):
        p = c["lo"] + (c["hi"] - c["lo"]) * ((37 * b + 11) % c["B"]) // max(1, c["B"] - 1)
        out.append((p, min(c["L"], p + c["resp"])))
    return out


def _lengths(c, dev):
    b = _bounds(c)
    return (torch.tensor([p for p, _ in b], dtype=torch.int32, device=dev),
            torch.tensor([n for _, n in b], dtype=torch.int32, device=dev))


def _qkv(c, g, dev):
    Bn, L, Hq, Hkv, D = (c[k] for k in ("B", "L", "Hq", "Hkv", "D"))
    dt = _DTYPES[c["dtype"]]
    if c.get("packed"):
        x = torch.empty(Bn, L, Hq + 2 * Hkv, D, dtype=dt, device=dev).normal_(generator=g)
        return x[:, :, :Hq], x[:, :, Hq:Hq + Hkv], x[:, :, Hq + Hkv:]
    return tuple(torch.empty(Bn, L, H, D, dtype=dt, device=dev).normal_(generator=g) for H in (Hq, Hkv, Hkv))


def _logits(N, V, dtype, pad, g, dev):
    """N(0, 3) logits; a tenth of the rows peaked by about 8 above their maximum, some above and some below the
    edit threshold. pad: rows start on 16-byte boundaries, else they follow each other."""
    stride = (V + 7) // 8 * 8 if pad else V
    x = torch.empty(N, stride, dtype=_DTYPES[dtype], device=dev).normal_(0.0, 3.0, generator=g)[:, :V]
    rows = torch.nonzero(torch.rand(N, device=dev, generator=g) < 0.1).flatten()
    at = torch.randint(0, V, (len(rows),), device=dev, generator=g)
    x[rows, at] = (4.25 * 3 + 4 + 8 * torch.rand(len(rows), device=dev, generator=g)).to(x.dtype)
    return x


def _state(c, g, dev):
    """Draft tokens and mask (a quarter of the positions masked)."""
    tok = torch.randint(0, c["V"], (c["B"], c["L"]), dtype=torch.int32, device=dev, generator=g)
    msk = (torch.rand(c["B"], c["L"], device=dev, generator=g) < 0.25).to(torch.uint8)
    return torch.where(msk == 1, c["V"], tok), msk


def _params(c, s):
    return B.RefineParams(_TAU, -1, _REMASK, c["V"], s["p"], s["n"])


def _rows(N, dev):
    return [torch.empty(N, dtype=t, device=dev) for t in (torch.int32, torch.float32, torch.float32)]


def prepare(case, seed):
    c, dev = case, torch.device("cuda", torch.cuda.current_device())
    g = torch.Generator(device=dev).manual_seed(seed)
    s = {"case": c}
    op = c["op"]
    if "B" in c:
        s["p"], s["n"] = _lengths(c, dev)
    if op in ("attn", "masked", "loop"):
        s["q"], s["k"], s["v"] = _qkv(c, g, dev)
        s["out"] = torch.empty(c["B"], c["L"], c["Hq"], c["D"], dtype=_DTYPES[c["dtype"]], device=dev)
    if op in ("vocab", "prob"):
        s["x"] = _logits(c["N"], c["V"], c["dtype"], c["pad"], g, dev)
        s["rows"] = _rows(c["N"], dev)
    if op == "prob":
        s["tok"] = torch.randint(0, c["V"], (c["N"],), dtype=torch.int32, device=dev, generator=g)
        s["lse"] = torch.cat([torch.logsumexp(x.float(), 1) for x in s["x"].split(256)])
    if op in ("step", "loop"):
        s["x"] = _logits(c["B"] * c["L"], c["V"], c["dtype"], False, g, dev).view(c["B"], c["L"], c["V"])
        s["rows"] = [t.view(c["B"], c["L"]) for t in _rows(c["B"] * c["L"], dev)]
        s["ws"] = torch.zeros(B.dlm_refine_step_workspace_bytes(c["B"]), dtype=torch.uint8, device=dev)
    if op in ("step", "loop", "update"):
        s["tok"], s["msk"] = _state(c, g, dev)
        s["params"] = _params(c, s)
        s["new"] = [torch.empty_like(s["tok"]), torch.empty_like(s["msk"]),
                    torch.empty(c["B"], dtype=torch.int32, device=dev)]
    if op == "update":
        # half of the positions predict their own token; confidences from near 0 to 1
        am = torch.randint(0, c["V"], s["tok"].shape, dtype=torch.int32, device=dev, generator=g)
        keep = torch.rand(s["tok"].shape, device=dev, generator=g) < 0.5
        s["am"] = torch.where(keep & (s["msk"] == 0), s["tok"], am)
        s["cf"] = torch.rand(s["tok"].shape, device=dev, generator=g).square()
        s["tp"] = s["cf"] * torch.rand(s["tok"].shape, device=dev, generator=g) if c["ranked"] else None
    if op == "lmhead":
        s["h"] = torch.empty(c["N"], c["d"], dtype=torch.bfloat16, device=dev).normal_(generator=g)
        s["w"] = torch.empty(c["V"], c["d"], dtype=torch.bfloat16, device=dev).normal_(0.0, c["d"] ** -0.5, generator=g)
        s["rows"] = _rows(c["N"], dev)
        s["ws"] = torch.empty(B.dlm_lmhead_workspace_bytes(c["N"]), dtype=torch.uint8, device=dev)
    if op == "loop":
        # The serving program records its pass once and refines each new draft with one launch.
        s["steps"] = torch.zeros(1, dtype=torch.int32, device=dev)
        tok, msk, ne = s["new"]
        side = torch.cuda.Stream(dev)
        side.wait_stream(torch.cuda.current_stream(dev))
        with torch.cuda.stream(side):
            B.dlm_loop_begin(s["steps"])
            B.dlm_bidir_attn(s["q"], s["k"], s["v"], s["n"], s["out"])
            B.dlm_refine_step(s["x"], tok, msk, s["params"], *s["rows"], tok, msk, ne, s["ws"])
            s["loop"] = B.dlm_loop_end(ne, c["passes"], s["steps"])
    return s


# ---------------------------------------------------------------- one pass

def run(state):
    s = state
    op = s["case"]["op"]
    if op == "attn":
        return B.dlm_bidir_attn(s["q"], s["k"], s["v"], s["n"], s["out"])
    if op == "masked":
        return B.dlm_attn_masked(s["q"], s["k"], s["v"], s["n"], s["p"], s["case"]["mode"], s["case"]["block"], s["out"])
    if op == "vocab":
        return B.dlm_vocab_confidence(s["x"], *s["rows"])
    if op == "prob":
        return B.dlm_token_prob(s["x"], s["tok"], s["lse"], s["rows"][1])
    if op == "step":
        return B.dlm_refine_step(s["x"], s["tok"], s["msk"], s["params"], *s["rows"], *s["new"], s["ws"])
    if op == "update":
        if s["tp"] is None:
            return B.dlm_refine_update(s["tok"], s["msk"], s["am"], s["cf"], s["params"], *s["new"])
        return B.dlm_refine_update_ranked(s["tok"], s["msk"], s["am"], s["cf"], s["tp"], s["params"], *s["new"])
    if op == "lmhead":
        return B.dlm_lmhead_confidence(s["h"], s["w"], *s["rows"], s["ws"])
    s["new"][0].copy_(s["tok"])  # the new draft, refined in place
    s["new"][1].copy_(s["msk"])
    s["loop"].launch()
    return (s["out"], *s["rows"], *s["new"], s["steps"])


# ---------------------------------------------------------------- work and accuracy

def _pairs(c):
    """(query, key) pairs of the batch under the case's mask."""
    total = 0
    for p, n in _bounds(c):
        if c["op"] != "masked":
            total += n * n
            continue
        total += p * p
        for start in range(p, n, c["block"]):
            end = min(n, start + c["block"])
            total += (end - start) * (end if c["mode"] == 1 else p + end - start)
    return total


def work(case):
    c, esz = case, {"bf16": 2, "f32": 4}.get(case.get("dtype"), 4)
    op = c["op"]
    attn_bytes = attn_flops = 0
    if op in ("attn", "masked", "loop"):
        tokens = sum(n for _, n in _bounds(c))
        attn_bytes = esz * c["D"] * (tokens * (c["Hq"] + 2 * c["Hkv"]) + c["B"] * c["L"] * c["Hq"])
        attn_flops = 4 * c["D"] * c["Hq"] * _pairs(c)
    if op in ("attn", "masked"):
        return {"bytes": attn_bytes, "flops": attn_flops}
    if op == "prob":
        return {"bytes": c["N"] * (esz + 12), "flops": c["N"]}
    if op == "lmhead":
        return {"bytes": 2 * c["d"] * (c["N"] + c["V"]) + 12 * c["N"], "flops": 2 * c["N"] * c["V"] * c["d"]}
    rows = c["N"] if op == "vocab" else c["B"] * c["L"]
    update = rows * (18 + (4 if c.get("ranked") else 0)) + 4 * c.get("B", 0)
    if op == "update":
        return {"bytes": update, "flops": rows}
    logits = {"bytes": rows * (esz * c["V"] + 12), "flops": 3 * rows * c["V"]}
    if op == "vocab":
        return logits
    passes = 2 if op == "loop" else 1  # the second pass finds nothing left to edit
    return {"bytes": passes * (logits["bytes"] + update + attn_bytes),
            "flops": passes * (logits["flops"] + attn_flops)}


def tolerance(case):
    """About four times what was measured against exact(): 16-bit outputs and
    softmax weights in bf16 attention, 32-bit sums elsewhere. Whole values are
    decided by comparing numbers, so a rounding can swap two positions whose
    confidences, or two tokens whose logits, are within it (bf16 logits tie
    exactly, and exact ties are ordered): `differ` allows those."""
    c = case
    op = c["op"]
    if op == "update":
        return "exact"
    if op in ("attn", "masked"):
        return {"rel": 1.2e-2, "max": 6e-2} if c["dtype"] == "bf16" else {"rel": 2e-6, "max": 2e-5}
    if op == "lmhead":
        return {"rel": 3.5e-5, "max": 3.5e-4, "differ": 2e-3}
    if op == "loop":
        return {"rel": 1.2e-2, "max": 6e-2, "differ": 4e-3}
    return {"rel": 4e-6, "max": 4e-5, "differ": 4e-3 if op == "step" else 0.0}


def _allowed(c, p, n, dev):
    """[n, n] mask of the keys each query of a sequence attends to."""
    i = torch.arange(n, device=dev)
    if c["op"] != "masked":
        return torch.ones(n, n, dtype=torch.bool, device=dev)
    block = torch.where(i < p, -1, (i - p).div(c["block"], rounding_mode="floor"))
    q, k = block[:, None], block[None, :]
    return k <= q if c["mode"] == 1 else (k == -1) | (k == q)


def _exact_attn(c, s):
    out = torch.zeros(s["out"].shape, dtype=torch.float64, device=s["out"].device)
    rep = c["Hq"] // c["Hkv"]
    for b, (p, n) in enumerate(_bounds(c)):
        q, k, v = (s[t][b, :n].double().transpose(0, 1) for t in ("q", "k", "v"))
        allowed = _allowed(c, p, n, q.device)
        for h in range(c["Hkv"]):
            x = q[h * rep:(h + 1) * rep] @ k[h].T / math.sqrt(c["D"])
            w = torch.softmax(x.masked_fill(~allowed, -math.inf), -1)
            out[b, :n, h * rep:(h + 1) * rep] = (w @ v[h]).transpose(0, 1)
    return out


def _exact_rows(chunks):
    """argmax (lowest index), confidence and log-sum-exp of float64 rows."""
    parts = []
    for x in chunks:
        m = x.amax(1, keepdim=True)
        at = torch.arange(x.shape[1], device=x.device)
        lse = torch.logsumexp(x, 1)
        parts.append((torch.where(x == m, at, x.shape[1]).amin(1).int(), torch.exp(m[:, 0] - lse), lse))
    return [torch.cat(t) for t in zip(*parts)]


def exact(case, seed):
    c, s = case, prepare(case, seed)
    op = c["op"]
    if op == "update":
        return None
    if op in ("attn", "masked"):
        return _exact_attn(c, s)
    if op == "lmhead":
        w = s["w"].double()
        return tuple(_exact_rows(h.double() @ w.T for h in s["h"].split(512)))
    if op == "prob":
        return torch.exp(s["x"].gather(1, s["tok"].long()[:, None])[:, 0].double() - s["lse"].double())
    x = s["x"].view(-1, c["V"])
    rows = _exact_rows(t.double() for t in x.split(max(1, 2 * 10 ** 8 // c["V"])))
    if op == "vocab":
        return tuple(rows)
    rows = [t.view(c["B"], c["L"]) for t in rows]
    # what the update decides depends on the order of the confidences
    if op == "step":
        return (*rows, None, None, None)
    return (_exact_attn(c, s), *rows, None, None, None, None)
