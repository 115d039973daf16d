"""Performance cases: the attention work of a model with LongGen layers, called as its programs call it.

Four programs use the library.  A trainer runs forward + backward of one layer per call, on lists prepared once
where the pattern is static and prepared anew for every packed sample where documents prune it; a prefill runs
the forward of a prompt; a server appends one token per sequence and decodes over its caches; and a server with a
cache of fixed size takes a prompt chunk by chunk.  The listed cases stand for them at the library's benchmark
configurations (Llama-2 7B / 70B attention shapes, 512 to 131072 tokens) and at ragged sizes between; draw()
spreads over the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_01485_b200 import binding as lg
from paper_2410_01485_b200 import synth

FULL, WINDOW, STRIDED = synth.MODE_FULL_CAUSAL, synth.MODE_SINK_WINDOW, synth.MODE_STRIDED_LOCAL


def _attn(kind, B, Hq, Hkv, L, D, block, mode, sink=0, window=0, stride=0, local=0, exact=False, layout="bhld",
          doc_mean=0):
    return {"kind": kind, "B": B, "Hq": Hq, "Hkv": Hkv, "L": L, "D": D, "block": block, "mode": mode, "sink": sink,
            "window": window, "stride": stride, "local": local, "exact": exact, "layout": layout,
            "doc_mean": doc_mean}


def _serve(kind, B, Hq, Hkv, D, sink, window, n_min, n_max, block_tokens=0, T=0):
    return {"kind": kind, "B": B, "Hq": Hq, "Hkv": Hkv, "D": D, "sink": sink, "window": window, "n_min": n_min,
            "n_max": n_max, "block_tokens": block_tokens, "T": T}


def listed():
    cases = [
        # a unit-test-sized layer (the smallest benchmark configuration): launches and host calls decide
        ("train_tiny", _attn("train", 1, 2, 2, 512, 64, 64, WINDOW, sink=64, window=128)),
        # a small model's sparse layer on a ragged batch, token-exact window, activations as a model's
        # projections leave them ([B, L, H, D])
        ("train_ragged_d64", _attn("train", 3, 16, 4, 6001, 64, 64, WINDOW, sink=64, window=1024, exact=True,
                                   layout="blhd")),
        # one of the model's full-attention layers at an ordinary context length
        ("train_full_16k", _attn("train", 1, 32, 32, 16384, 128, 64, FULL)),
        # the strided pattern of the 70B-shaped configuration with grouped queries, at 64K
        ("train_strided_64k", _attn("train", 1, 64, 8, 65536, 128, 64, STRIDED, stride=16, local=4)),
        # the length-extension step the library's headline number is quoted on: 128K tokens, sink + window
        ("train_window_128k", _attn("train", 1, 32, 32, 131072, 128, 128, WINDOW, sink=128, window=4096)),
        # a sample packed from documents: every sample has its own boundaries, so its lists are part of the step
        ("train_documents_32k", _attn("documents", 1, 32, 32, 32768, 128, 64, WINDOW, sink=64, window=2048,
                                      doc_mean=4000)),
        # prefill of a long prompt through a sparse layer
        ("prefill_window_32k", _attn("prefill", 1, 32, 32, 32768, 128, 64, WINDOW, sink=64, window=4032)),
        # prefill of an odd-length prompt through a full layer with grouped queries
        ("prefill_full_10k", _attn("prefill", 1, 64, 8, 10007, 128, 128, FULL)),
        # one serving step (append + decode) of a batch over its sink + window rings
        ("decode_ring_b16", _serve("decode", 16, 64, 8, 128, 128, 4096, 131072, 131072)),
        # the same for a single user: latency
        ("decode_ring_b1", _serve("decode", 1, 64, 8, 128, 128, 4096, 131072, 131072)),
        # one serving step of a full layer: linear caches, every sequence at its own length
        ("decode_linear_b4", _serve("decode", 4, 32, 32, 128, 0, 32768, 9000, 32768)),
        # a chunk of a long prompt against the rings
        ("chunk_1500", _serve("chunk", 2, 64, 8, 128, 128, 4096, 20000, 20000, T=1500)),
    ]
    return [dict(c, name=n) for n, c in cases]


# ------------------------------------------------------------------------------- drawn cases

_MAX_FLOPS = 3.0e13          # of the largest listed case
_MAX_STATE = 40e9            # bytes a state may hold (three of them fit the card)


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _heads(rng):
    hkv = rng.choice((2, 4, 8, 16, 32))
    return min(64, hkv * rng.choice((1, 1, 2, 4, 8))), hkv


def _draw_attn(rng, kind):
    L = _log_int(rng, 500, 131072)
    if rng.random() < 0.5:
        L = max(512, (L + 128) // 256 * 256)               # half of the lengths are round, half ragged
    D = rng.choice((128, 128, 128, 64))
    block = rng.choice((64, 64, 128))
    mode = rng.choice((WINDOW, WINDOW, FULL) if kind == "documents" else (WINDOW, WINDOW, STRIDED, FULL))
    sink = window = stride = local = 0
    exact = False
    if mode == WINDOW:
        sink = block * rng.choice((0, 1, 1, 2))
        window = block * max(1, _log_int(rng, 128, 4096) // block)
        exact = rng.random() < 0.25
    elif mode == STRIDED:
        stride, local = rng.choice((8, 16, 32, 64)), rng.choice((1, 2, 4))
    Hq, Hkv = _heads(rng)
    B = 1 if kind == "documents" and rng.random() < 0.7 else rng.choice((1, 1, 1, 2, 4))
    doc_mean = _log_int(rng, 300, 8192) if kind == "documents" else 0
    c = _attn(kind, B, Hq, Hkv, L, D, block, mode, sink, window, stride, local, exact,
              rng.choice(("bhld", "bhld", "blhd")), doc_mean)
    while work(c)["flops"] > _MAX_FLOPS or _state_bytes(c) > _MAX_STATE:
        if c["B"] > 1:
            c["B"] //= 2
        elif c["Hkv"] > 2:
            c["Hq"], c["Hkv"] = c["Hq"] // 2, c["Hkv"] // 2
        else:
            c["L"] //= 2
    return c


def _draw_serve(rng, kind):
    Hq, Hkv = _heads(rng)
    D = rng.choice((128, 128, 128, 64))
    if kind == "chunk":
        sink, window = 64 * rng.choice((0, 1, 2)), 64 * (_log_int(rng, 512, 4096) // 64)
        n = rng.choice((0, _log_int(rng, 100, 4000), _log_int(rng, 4000, 130000)))
        c = _serve(kind, rng.choice((1, 1, 2, 4)), Hq, Hkv, D, sink, window, n, n, rng.choice((0, 0, 64)),
                   T=_log_int(rng, 16, 8192))
    elif rng.random() < 0.6:
        sink, window = 64 * rng.choice((1, 1, 2)), 64 * (_log_int(rng, 512, 4096) // 64)
        n_max = _log_int(rng, 600, 131072)
        c = _serve(kind, _log_int(rng, 1, 64), Hq, Hkv, D, sink, window, rng.choice((n_max, 1 + n_max // 4)), n_max,
                   rng.choice((0, 0, 64)))
    else:
        cap = _log_int(rng, 512, 65536)
        c = _serve(kind, _log_int(rng, 1, 32), Hq, Hkv, D, 0, cap, rng.choice((cap, 1 + cap // 4)), cap)
    while work(c)["bytes"] > 4e9:
        c["B"] = max(1, c["B"] // 2)
    return c


def draw(rng):
    kind = rng.choice(("train", "train", "train", "documents", "prefill", "prefill", "decode", "decode", "decode",
                       "chunk"))
    return _draw_serve(rng, kind) if kind in ("decode", "chunk") else _draw_attn(rng, kind)


# ----------------------------------------------------------------------------------- the work

def _doc_starts(c, seed):
    return torch.stack([synth.make_doc_start(c["L"], seed=seed * 64 + b, mean_len=c["doc_mean"])
                        for b in range(c["B"])])


def _visible_pairs(c):
    """(query, key) pairs of the batch that one head may see.  Documents: those of one fixed seed."""
    i = np.arange(c["L"], dtype=np.int64)
    bs, qb = c["block"], np.arange(c["L"], dtype=np.int64) // c["block"]
    if c["mode"] == STRIDED:
        first = np.maximum(0, qb - c["local"] + 1)                     # oldest local block
        return c["B"] * int((i - first * bs + 1 + (first + c["stride"] - 1) // c["stride"] * bs).sum())
    if c["mode"] == FULL:
        w0 = np.zeros_like(i)
    elif c["exact"]:
        w0 = np.maximum(0, i - c["window"] + 1)
    else:
        w0 = np.maximum(0, (qb - c["window"] // bs + 1) * bs)
    sink = np.minimum(w0, c["sink"])                                    # sink keys outside the window
    if not c["doc_mean"]:
        return c["B"] * int((i - w0 + 1 + sink).sum())
    total = 0
    for ds in _doc_starts(c, 0).numpy().astype(np.int64):
        total += int((i - np.maximum(w0, ds) + 1 + np.maximum(0, sink - ds)).sum())
    return total


def _chunk_pairs(c):
    pos = c["n_min"] + np.arange(c["T"], dtype=np.int64)
    if c["block_tokens"]:
        bs = c["block_tokens"]
        w0 = np.maximum(0, (pos // bs - c["window"] // bs + 1) * bs)
    else:
        w0 = np.maximum(0, pos - c["window"] + 1)
    return c["B"] * int((pos - w0 + 1 + np.minimum(w0, c["sink"])).sum())


def _lengths(c):
    """Tokens in each sequence's cache after the append: spread evenly over the case's range."""
    B = c["B"]
    return [c["n_max"] - (c["n_max"] - c["n_min"]) * b // max(1, B - 1) if B > 1 else c["n_max"] for b in range(B)]


def work(case):
    c, D = case, case["D"]
    if c["kind"] == "decode":
        slots = sum(min(n, c["sink"] + c["window"]) for n in _lengths(c))
        rows = c["B"] * c["Hq"]
        return {"bytes": slots * c["Hkv"] * D * 4 + c["B"] * c["Hkv"] * D * 8 + rows * (D * 4 + 4),
                "flops": 4.0 * slots * c["Hq"] * D}
    if c["kind"] == "chunk":
        kept = min(c["n_min"], c["sink"] + c["window"])
        q = c["B"] * c["Hq"] * c["T"]
        return {"bytes": q * (4 * D + 4) + 4 * c["B"] * c["Hkv"] * (kept + c["T"]) * D,
                "flops": 4.0 * D * c["Hq"] * _chunk_pairs(c)}
    q, kv = c["B"] * c["Hq"] * c["L"], c["B"] * c["Hkv"] * c["L"]
    if c["kind"] == "prefill":
        return {"bytes": q * (4 * D + 4) + kv * 4 * D, "flops": 4.0 * D * c["Hq"] * _visible_pairs(c)}
    # q, dO in, O, LSE, dQ out; K, V in, dK, dV out
    return {"bytes": q * (8 * D + 4) + kv * 8 * D, "flops": 14.0 * D * c["Hq"] * _visible_pairs(c)}


def _state_bytes(c):
    per_row = 2 * c["D"] * (4 * c["Hq"] + 4 * c["Hkv"])
    kept = 2.3 * c["Hq"] * _visible_pairs(c) if c["kind"] != "prefill" else 0     # dS the backward may keep
    return c["B"] * c["L"] * per_row + kept + 4.0 * (c["L"] / c["block"]) ** 2 * 5


def tolerance(case):
    # Measured against the same definition in fp64 (bf16 operands, fp32 sums), over all kinds of case: O, dQ, dK, dV
    # 2.0e-3 to 2.6e-3 (bf16 results alone: 1.7e-3), the largest single difference 0.1 of the tensor's root mean
    # square (a bf16 rounding of the early rows' large gradients).  Four times that.
    return {"rel": 1.0e-2, "max": 0.4}


# ------------------------------------------------------------------------------ one pass

def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32).to(torch.bfloat16)


def _tensor(c, H, gen=None):
    """[B, H, L, D] in the case's memory layout, N(0,1) from `gen` or uninitialised."""
    B, L, D = c["B"], c["L"], c["D"]
    shape = (B, H, L, D) if c["layout"] == "bhld" else (B, L, H, D)
    t = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    if gen is not None:
        flat = t.view(-1)
        for s in range(0, flat.numel(), 1 << 27):
            flat[s:s + (1 << 27)] = _randn(gen, min(1 << 27, flat.numel() - s))
    return t if c["layout"] == "bhld" else t.transpose(1, 2)


def _inputs(c, seed):
    """The tensors a program has in hand before the call."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, Hq, Hkv, D, T = c["B"], c["Hq"], c["Hkv"], c["D"], c.get("T", 0)
    if c["kind"] in ("decode", "chunk"):
        cap, step = c["sink"] + c["window"], (1,) if c["kind"] == "decode" else (T,)
        s = {"k_cache": _randn(gen, B, Hkv, cap, D), "v_cache": _randn(gen, B, Hkv, cap, D)}
        s.update(q=_randn(gen, B, Hq, *(step if c["kind"] == "chunk" else ()), D), k=_randn(gen, B, Hkv, *step, D),
                 v=_randn(gen, B, Hkv, *step, D))
        return s
    s = {"q": _tensor(c, Hq, gen), "k": _tensor(c, Hkv, gen), "v": _tensor(c, Hkv, gen)}
    if c["kind"] != "prefill":
        s["do"] = _tensor(c, Hq, gen)
    if c["doc_mean"]:
        s["docs"] = _doc_starts(c, seed).cuda()
    return s


def prepare(case, seed):
    c = case
    s = dict(_inputs(c, seed), kind=c["kind"])
    if c["kind"] in ("decode", "chunk"):
        return _prepare_serve(c, s)
    want_bwd = c["kind"] != "prefill"
    s.update(o=_tensor(c, c["Hq"]), lse=torch.empty(c["B"], c["Hq"], c["L"], dtype=torch.float32, device="cuda"))
    if want_bwd:
        s.update(dq=_tensor(c, c["Hq"]), dk=_tensor(c, c["Hkv"]), dv=_tensor(c, c["Hkv"]))
    docs = s.get("docs")
    p = lg.attn_params(c["B"], c["Hq"], c["Hkv"], c["L"], c["D"], c["block"], c["mode"], c["sink"], c["window"],
                       c["stride"], c["local"], window_exact=c["exact"], doc_start=docs)
    s["p"], s["ws"] = p, lg.attn_workspace(p, want_bwd)
    if docs is None:
        lg.lg_sparse_attn_prepare(p, s["ws"], want_bwd)      # the pattern is static: once per program
    s["per_sample_lists"] = docs is not None and c["B"] == 1    # (several sequences: the calls build their own)
    return s


def _prepare_serve(c, s):
    B, Hq, Hkv, D = c["B"], c["Hq"], c["Hkv"], c["D"]
    s["p"] = p = lg.decode_params(B, Hq, Hkv, D, c["sink"], c["window"], block_tokens=c["block_tokens"])
    if c["kind"] == "chunk":
        T = c["T"]
        s.update(o=torch.empty(B, Hq, T, D, dtype=torch.bfloat16, device="cuda"),
                 lse=torch.empty(B, Hq, T, dtype=torch.float32, device="cuda"), n=c["n_min"],
                 ws=lg.chunk_prefill_workspace(p, T, c["n_min"]))
        return s
    n = torch.tensor(_lengths(c), dtype=torch.int64).cuda()
    s.update(n=n, n_before=n - 1, o=torch.empty(B, Hq, D, dtype=torch.bfloat16, device="cuda"),
             lse=torch.empty(B, Hq, dtype=torch.float32, device="cuda"), ws=lg.decode_workspace(p))
    # a serving loop's decode: fixed buffers, arguments marshalled once
    s["decode"] = lg.decode_call(p, s["q"], s["k_cache"], s["v_cache"], n, s["o"], s["lse"], s["ws"])
    return s


def run(s):
    p = s["p"]
    if s["kind"] == "decode":
        lg.lg_kv_ring_append(p, s["k_cache"], s["v_cache"], s["k"], s["v"], s["n_before"])
        s["decode"]()
        return s["o"], s["lse"], s["k_cache"], s["v_cache"]
    if s["kind"] == "chunk":
        return lg.lg_chunk_prefill(p, s["q"], s["k"], s["v"], s["k_cache"], s["v_cache"], s["n"], o=s["o"],
                                   lse=s["lse"], workspace=s["ws"])
    if s["per_sample_lists"]:
        lg.lg_sparse_attn_prepare(p, s["ws"], True)
    out = lg.lg_sparse_attn_fwd(p, s["q"], s["k"], s["v"], o=s["o"], lse=s["lse"], workspace=s["ws"])
    if s["kind"] == "prefill":
        return out
    return out + lg.lg_sparse_attn_bwd(p, s["q"], s["k"], s["v"], s["o"], s["lse"], s["do"], dq=s["dq"], dk=s["dk"],
                                       dv=s["dv"], workspace=s["ws"])


# ------------------------------------------------------- the same outputs in 64 bits

_MAX_EXACT_FLOPS = 1.5e14    # masked pairs counted: about ten seconds of 64-bit products


def _attend(q, k, v, see, do=None):
    """Rows of masked softmax attention for one head, and what they add to the gradients."""
    scale = q.shape[-1] ** -0.5
    x = (q @ k.T).mul_(scale).masked_fill_(~see, -math.inf)
    lse = torch.logsumexp(x, 1)
    p = x.sub_(lse[:, None]).exp_()
    o = p @ v
    if do is None:
        return o, lse
    ds = (do @ v.T).sub_((do * o).sum(1, keepdim=True)).mul_(p).mul_(scale)
    return o, lse, ds @ k, ds.T @ q, p.T @ do


def _seen(c, i, j, doc=None):
    """Which keys j the queries at positions i see, as the pattern of a training or prefill call says."""
    bs = c["block"]
    see = j[None, :] <= i[:, None]
    if c["mode"] == WINDOW:
        near = (i[:, None] - j[None, :] < c["window"] if c["exact"] else
                (i // bs)[:, None] - (j // bs)[None, :] < c["window"] // bs)
        see &= near | (j < c["sink"])[None, :]
    elif c["mode"] == STRIDED:
        see &= ((i // bs)[:, None] - (j // bs)[None, :] < c["local"]) | (j // bs % c["stride"] == 0)[None, :]
    return see if doc is None else see & (j[None, :] >= doc[:, None])


def _exact_attn(c, s):
    B, Hq, Hkv, L, D, bs, G = c["B"], c["Hq"], c["Hkv"], c["L"], c["D"], c["block"], c["Hq"] // c["Hkv"]
    grads = "do" in s
    f64 = dict(dtype=torch.float64, device="cuda")
    o, lse = torch.empty(B, Hq, L, D, **f64), torch.empty(B, Hq, L, **f64)
    dq, dk, dv = (torch.zeros(B, H, L, D, **f64) for H in ((Hq, Hkv, Hkv) if grads else (0, 0, 0)))
    pos = torch.arange(L, device="cuda")
    rows = 1024 if L <= 65536 else 512
    for r0 in range(0, L, rows):
        r1 = min(L, r0 + rows)
        i = pos[r0:r1]
        j = pos[:r1]
        near = r0 - c["window"] - bs if c["mode"] == WINDOW else r0 // bs * bs - c["local"] * bs
        if c["mode"] == WINDOW:
            j = j[(j >= near) | (j < c["sink"])]
        elif c["mode"] == STRIDED:
            j = j[(j >= near) | (j // bs % c["stride"] == 0)]
        for b in range(B):
            see = _seen(c, i, j, s["docs"][b, r0:r1] if "docs" in s else None)
            for h in range(Hq):
                kv = (b, h // G, j)
                got = _attend(s["q"][b, h, r0:r1].double(), s["k"][kv].double(), s["v"][kv].double(), see,
                              s["do"][b, h, r0:r1].double() if grads else None)
                o[b, h, r0:r1], lse[b, h, r0:r1] = got[:2]
                if grads:
                    dq[b, h, r0:r1] = got[2]
                    dk[kv] += got[3]
                    dv[kv] += got[4]
    return (o, lse, dq, dk, dv) if grads else (o, lse)


def _slots(c, n):
    """The ring slots that hold something after n tokens, and the position of the token in each, oldest first."""
    sink, window = c["sink"], c["window"]
    j = torch.cat([torch.arange(min(n, sink)), torch.arange(max(sink, n - window), max(n, sink))]).cuda()
    return torch.where(j < sink, j, sink + (j - sink) % window), j


def _kept(c, i, j):
    """Which cached positions j a query at position i of a serving call attends."""
    bs = c["block_tokens"]
    near = i // bs - j // bs < c["window"] // bs if bs else i - j < c["window"]
    return (j <= i) & (near | (j < c["sink"]))


def _exact_serve(c, s):
    B, Hq, G, T = c["B"], c["Hq"], c["Hq"] // c["Hkv"], max(1, c["T"])
    o, lse = torch.empty(s["q"].shape, dtype=torch.float64, device="cuda"), []
    for b, n in enumerate(_lengths(c)):
        if c["kind"] == "decode":
            at = n - 1 if n <= c["sink"] else c["sink"] + (n - 1 - c["sink"]) % c["window"]
            s["k_cache"][b, :, at], s["v_cache"][b, :, at] = s["k"][b, :, 0], s["v"][b, :, 0]
        slot, j = _slots(c, n)
        i = torch.arange(n, n + T, device="cuda") if c["kind"] == "chunk" else torch.tensor([n - 1], device="cuda")
        every = torch.cat([j, i]) if c["kind"] == "chunk" else j
        see = _kept(c, i[:, None], every[None, :])
        for h in range(Hq):
            k, v = (s[x][b, h // G, slot].double() for x in ("k_cache", "v_cache"))
            if c["kind"] == "chunk":
                k, v = torch.cat([k, s["k"][b, h // G].double()]), torch.cat([v, s["v"][b, h // G].double()])
            got, l = _attend(s["q"][b, h].double().view(T, -1), k, v, see)
            o[b, h] = got.view(o[b, h].shape)
            lse.append(l)
    lse = torch.stack(lse).view(*s["q"].shape[:-1])
    return (o, lse) if c["kind"] == "chunk" else (o, lse, s["k_cache"].double(), s["v_cache"].double())


def exact(case, seed):
    if work(case)["flops"] > _MAX_EXACT_FLOPS:
        return None
    return (_exact_serve if case["kind"] in ("decode", "chunk") else _exact_attn)(case, _inputs(case, seed))
