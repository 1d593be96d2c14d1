"""Performance cases of the ReCo hot path, measured through the public entry points.

Each case is one call (or one short chain of calls) that a serving loop makes: the scoring
of a cache at a step boundary, the selection with its compaction, one decode step, a run of
tokens through a captured graph, the answer probe, and the Tiny workload's whole step.
Shapes come from the workloads of this package (their heads, windows, vocabularies and
lengths) and from the ranges the tests cover: 1 to 16 query heads per KV head, head
dimensions 64 and 128, float32 and bf16 caches, a few tokens to tens of thousands per unit.

`listed` names the fixed cases, `draw` gives more of the same ranges, `prepare` builds a
case's inputs from a seed, `run` makes one pass, `exact` computes the same outputs with
plain torch in float64, `work` counts what a pass cannot do without and `tolerance` states
how far another correct implementation may be.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_04771_gb300 import reco
from paper_2608_04771_gb300 import workloads as W
from paper_2608_04771_gb300.driver import HotPath

DEV = "cuda"
GB = 1e9


def _heads(layers, batch, h_q, h_kv, d, dtype):
    return {"layers": layers, "batch": batch, "h_q": h_q, "h_kv": h_kv, "d": d, "dtype": dtype}


def listed():
    return [
        # The Tiny workload's whole step (float32): score, select, compact, one decode, the
        # penalty and the answer probe, a dozen launches on almost no data.
        {"name": "tiny_step_f32", "kind": "tiny", "L": 512, "w": 16, "pool": 7, "vocab": 1024, "ids": 8, "answer": 8},
        # Eq. 2 in two passes over a 7B-class prompt cache: window queries that were never
        # decoded (after a prefill), every sequence compressed.
        {"name": "score_7b", "kind": "score", **_heads(28, 8, 28, 4, 128, "bf16"), "lo": 15000, "hi": 16384, "w": 32,
         "pool": 7, "scored": 8},
        # Eq. 2 in one pass with the decode's normalisers, 32B-class heads and window (320
        # window rows), eight of its layers at full length.
        {"name": "score_lse_32b", "kind": "score_lse", **_heads(8, 4, 40, 8, 128, "bf16"), "lo": 30000, "hi": 32768,
         "w": 64, "pool": 7, "scored": 4},
        # Eq. 2 in two passes over a float32 cache with the 1.5B-class heads.
        {"name": "score_f32", "kind": "score", **_heads(8, 4, 12, 2, 128, "f32"), "lo": 3000, "hi": 4096, "w": 32,
         "pool": 7, "scored": 4},
        # A step boundary of the step-loop trace: two of sixteen sequences score their short
        # caches from the decode's rings and select; the others are masked out.
        {"name": "boundary_trace", "kind": "boundary", **_heads(28, 16, 28, 4, 128, "bf16"), "lo": 90, "hi": 240,
         "w": 32, "pool": 7, "scored": 2, "ratio": 0.25},
        # Top-m selection and in-place compaction of the 7B-class cache (16 of its layers).
        {"name": "compress_7b", "kind": "compress", **_heads(16, 8, 28, 4, 128, "bf16"), "lo": 15000, "hi": 16384,
         "w": 32, "pool": 7, "scored": 8, "ratio": 0.25},
        # Sixteen tokens of the step-loop trace, each one captured graph: input copy, decode
        # with the window rings over caches of 40 to 200 rows, penalty and draw.
        {"name": "token_trace", "kind": "token", **_heads(28, 16, 28, 4, 128, "bf16"), "lo": 40, "hi": 200, "w": 32,
         "vocab": 152064, "ids": 16, "tokens": 16},
        # One decode step of the 1.5B-class stack after compression: few units of about a
        # thousand rows, fewer units than warps.
        {"name": "decode_1.5b", "kind": "decode", **_heads(28, 4, 12, 2, 128, "bf16"), "lo": 800, "hi": 1500,
         "out": "bf16", "ragged": False},
        # One decode step of the 7B-class stack after compression.
        {"name": "decode_7b", "kind": "decode", **_heads(28, 8, 28, 4, 128, "bf16"), "lo": 3800, "hi": 4700,
         "out": "bf16", "ragged": False},
        # One decode step with 16 query heads per KV head, the most the decode takes.
        {"name": "decode_16heads", "kind": "decode", **_heads(28, 4, 64, 4, 128, "bf16"), "lo": 2000, "hi": 4100,
         "out": "bf16", "ragged": False},
        # One decode step over a float32 cache with the 1.5B-class heads.
        {"name": "decode_f32", "kind": "decode", **_heads(28, 4, 12, 2, 128, "f32"), "lo": 800, "hi": 1500,
         "out": "f32", "ragged": False},
        # The answer probe of the 7B-class workload: 8 answers of 32 tokens over the vocabulary.
        {"name": "ppl_7b", "kind": "ppl", "batch": 8, "answer": 32, "vocab": 152064, "ragged": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges: any kind, type, head shape and length."""
    kind = rng.choice(["score", "score", "score_lse", "boundary", "compress", "token", "decode", "decode", "decode",
                       "sample", "ppl", "tiny"])
    if kind == "tiny":
        w = rng.randint(5, 32)
        return {"kind": kind, "L": _log_int(rng, 128, 2048), "w": w, "pool": rng.choice([1, 3, 5, 7]),
                "vocab": _log_int(rng, 500, 20000), "ids": rng.randint(2, 16), "answer": rng.randint(2, 16)}
    if kind == "sample":
        return {"kind": kind, "batch": _log_int(rng, 1, 64), "vocab": _log_int(rng, 2000, 200000),
                "ids": rng.randint(1, 64)}
    if kind == "ppl":
        return {"kind": kind, "batch": rng.randint(1, 16), "answer": rng.randint(2, 48),
                "vocab": _log_int(rng, 2000, 200000), "ragged": rng.random() < 0.5}
    dtype = "f32" if kind in ("score", "score_lse", "compress", "decode") and rng.random() < 0.25 else "bf16"
    d = 64 if rng.random() < 0.25 else 128
    h_kv = rng.choice([1, 2, 3, 4, 8])
    G = rng.randint(1, 16) if kind == "decode" else rng.randint(1, 8)
    case = {"kind": kind, **_heads(rng.randint(1, 28), rng.randint(1, 16), G * h_kv, h_kv, d, dtype)}
    units = case["layers"] * case["batch"] * h_kv
    row = d * (4 if dtype == "f32" else 2)
    # lengths: spread over their logarithm, at most about 1.5 GB of K and V together
    most = int(min(32768, max(64, 1.5 * GB / (units * row * 2))))
    hi = _log_int(rng, 64, most)
    case["lo"], case["hi"] = max(40, hi // rng.randint(1, 4)), max(48, hi)
    if kind == "decode":
        case["out"] = "f32" if dtype == "f32" or rng.random() < 0.3 else "bf16"
        case["ragged"] = rng.random() < 0.5
        return case
    if kind == "token":
        case["lo"], case["hi"] = min(case["lo"], 800), min(case["hi"], 1200)
        case.update({"w": 32, "vocab": _log_int(rng, 2000, 152064), "ids": rng.randint(2, 32), "tokens": 16})
        return case
    w = rng.randint(8, min(64, 390 // G))
    case.update({"w": w, "pool": rng.choice([1, 3, 5, 7, 7]), "scored": rng.randint(1, case["batch"])})
    case["lo"], case["hi"] = max(case["lo"], w + 1), max(case["hi"], w + 2)
    if kind in ("boundary", "compress"):
        case["ratio"] = round(rng.uniform(0.2, 0.9), 3)
    if dtype == "f32" and kind != "compress":  # float32 scoring is bound by arithmetic: keep it ordinary
        flops = 4.0 * units * G * w * d * case["hi"]
        case["layers"] = max(1, min(case["layers"], int(case["layers"] * 1e11 / flops)))
    return case


# ---------------------------------------------------------------- inputs
class State:
    pass


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _np(seed, stream):
    return np.random.Generator(np.random.PCG64([int(seed), stream]))


def _dt(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _randn(g, shape, dtype, scale=1.0):
    x = torch.randn(shape, generator=g, device=DEV, dtype=dtype)
    return x if scale == 1.0 else x.mul_(scale)


def _lens(case, seed):
    """[layers, B, h_kv] lengths: one per sequence, as the keep counts leave them, or (ragged) one
    per unit."""
    rng = _np(seed, 1)
    Ly, B, H = case["layers"], case["batch"], case["h_kv"]
    if case.get("ragged"):
        n = rng.integers(case["lo"], case["hi"] + 1, (Ly, B, H))
    else:
        n = np.broadcast_to(rng.integers(case["lo"], case["hi"] + 1, (1, B, 1)), (Ly, B, H))
    return np.ascontiguousarray(n, dtype=np.int32)


def _keep(case, seed, lens):
    """[B] keep counts: `scored` sequences keep a ratio around the case's, the others everything."""
    rng = _np(seed, 2)
    keep = lens[0, :, 0].copy()
    for b in rng.permutation(case["batch"])[:case["scored"]]:
        r = float(np.clip(case.get("ratio", 0.25) + rng.uniform(-0.05, 0.05), 0.1, 0.95))
        keep[b] = reco.reco_keep_count(r, int(keep[b]), case["w"])
    return keep.astype(np.int32)


def _to(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _scale(case):
    return 1.0 / math.sqrt(case["d"])


def _score_state(case, seed):
    s = State()
    g = _gen(seed)
    lens = _lens(case, seed)
    cap = case["hi"] + 64
    shape = (case["layers"], case["batch"], case["h_kv"], cap, case["d"])
    s.K = _randn(g, shape, _dt(case))
    s.V = torch.empty_like(s.K)  # scoring does not read the values
    s.q_win = _randn(g, (case["layers"], case["batch"], case["h_q"], case["w"], case["d"]), _dt(case))
    s.lens = _to(lens)
    s.keep = _to(_keep(case, seed, lens)) if case["scored"] < case["batch"] or case["kind"] == "boundary" else None
    s.kv = reco.make_kv(s.K, s.V, case["h_q"])
    s.scores = torch.zeros(shape[:4], dtype=torch.float32, device=DEV)
    s.ws = reco.workspace(reco.RECO_OP_SCORE, s.kv, case["w"], DEV)
    if case["kind"] != "score":  # the decode's log-sum-exps of the window tokens
        s.row_lse = torch.empty((case["w"], case["layers"], case["batch"], case["h_q"]), dtype=torch.float32,
                                device=DEV)
        for b, h, lse, _ in _window_rows(case, s, torch.float32):
            G = case["h_q"] // case["h_kv"]
            s.row_lse[:, :, b, h * G:(h + 1) * G] = lse.view(case["layers"], G, case["w"]).permute(2, 0, 1)
    if case["kind"] == "boundary":
        s.kept = torch.zeros(shape[:4], dtype=torch.int32, device=DEV)
        s.ws_select = reco.workspace(reco.RECO_OP_SELECT, s.kv, case["w"], DEV)
    return s


def _compress_state(case, seed):
    s = State()
    g = _gen(seed)
    lens = _lens(case, seed)
    shape = (case["layers"], case["batch"], case["h_kv"], case["hi"] + 64, case["d"])
    s.K, s.V = _randn(g, shape, _dt(case)), _randn(g, shape, _dt(case))
    s.lens0 = _to(lens)
    s.lens = s.lens0.clone()
    s.keep = _to(_keep(case, seed, lens))
    # scores as Eq. 2 leaves them: positive, skewed, max-pooled (runs of equal values)
    raw = torch.exp(0.5 * torch.randn(shape[:4], generator=g, device=DEV)) * (case["w"] / case["hi"])
    p = case["pool"]
    s.scores = torch.nn.functional.max_pool1d(raw.view(1, -1, shape[3]), p, 1, p // 2).view(shape[:4]).contiguous()
    s.kv = reco.make_kv(s.K, s.V, case["h_q"])
    s.kept = torch.zeros(shape[:4], dtype=torch.int32, device=DEV)
    s.ws = reco.workspace(reco.RECO_OP_SELECT, s.kv, case["w"], DEV)
    return s


def _decode_state(case, seed):
    s = State()
    g = _gen(seed)
    Ly, B, d = case["layers"], case["batch"], case["d"]
    shape = (Ly, B, case["h_kv"], case["hi"] + 64, d)
    s.K, s.V = _randn(g, shape, _dt(case)), _randn(g, shape, _dt(case))
    s.q = _randn(g, (Ly, B, case["h_q"], d), _dt(case))
    s.kn, s.vn = _randn(g, (Ly, B, case["h_kv"], d), _dt(case)), _randn(g, (Ly, B, case["h_kv"], d), _dt(case))
    s.lens0 = _to(_lens(case, seed))
    s.lens = s.lens0.clone()
    s.out = torch.empty(s.q.shape, dtype=torch.float32 if case["out"] == "f32" else torch.bfloat16, device=DEV)
    s.lse = torch.empty((Ly, B, case["h_q"]), dtype=torch.float32, device=DEV)
    s.kv = reco.make_kv(s.K, s.V, case["h_q"])
    s.ws = reco.workspace(reco.RECO_OP_DECODE, s.kv, 0, DEV)
    return s


def _vocab_inputs(case, seed, B, g):
    rng = _np(seed, 3)
    s = State()
    s.ids = _to(rng.choice(case["vocab"], case["ids"], replace=False).astype(np.int32))
    s.rewards = _to(rng.beta(2.0, 2.0, B).astype(np.float32))
    return s


def _token_state(case, seed):
    """The trace's per-token graph: the token's packed inputs copied from a pool of w rows at the
    ring slot, the decode with the lse and query rings, the penalty and the draw."""
    g = _gen(seed)
    Ly, B, Hq, H, d, w, V = (case[k] for k in ("layers", "batch", "h_q", "h_kv", "d", "w", "vocab"))
    s = _vocab_inputs(case, seed, B, g)
    shape = (Ly, B, H, case["hi"] + 64, d)
    s.K, s.V = _randn(g, shape, _dt(case)), _randn(g, shape, _dt(case))
    s.lens0 = _to(_lens(case, seed))
    s.lens = s.lens0.clone()
    parts = [((Ly, B, Hq, d), torch.bfloat16), ((Ly, B, H, d), torch.bfloat16), ((Ly, B, H, d), torch.bfloat16),
             ((B, V), torch.float32), ((B,), torch.float32)]
    size = [(math.prod(sh) * (2 if dt == torch.bfloat16 else 4) + 255) // 256 * 256 for sh, dt in parts]
    s.pool = torch.zeros((w, sum(size)), dtype=torch.uint8, device=DEV)
    s.static = torch.zeros(sum(size), dtype=torch.uint8, device=DEV)

    def view(buf, k):
        off, (sh, dt) = sum(size[:k]), parts[k]
        n = math.prod(sh) * (2 if dt == torch.bfloat16 else 4)
        return buf[off:off + n].view(dt).view(sh)

    for t in range(w):
        for k in range(3):
            view(s.pool[t], k).normal_(generator=g)
        view(s.pool[t], 3).normal_(std=2.0, generator=g)
        view(s.pool[t], 4).uniform_(generator=g)
    s.pool_view = lambda t, k: view(s.pool[t], k)
    s.q, s.kn, s.vn, s.logits, s.draws = (view(s.static, k) for k in range(5))
    s.out = torch.empty(s.q.shape, dtype=torch.bfloat16, device=DEV)
    s.tok = torch.zeros(B, dtype=torch.int32, device=DEV)
    s.ring = torch.zeros((2 * w, Ly, B, Hq), dtype=torch.float32, device=DEV)
    s.q_ring = torch.zeros((Ly, B, Hq, w, d), dtype=torch.bfloat16, device=DEV)
    s.slot = torch.zeros(1, dtype=torch.long, device=DEV)
    s.kv = reco.make_kv(s.K, s.V, Hq)
    s.ws = reco.workspace(reco.RECO_OP_DECODE, s.kv, 0, DEV)
    s.ws_sample = reco.sample_workspace(B, V, DEV)
    lse = torch.empty((Ly, B, Hq), dtype=torch.float32, device=DEV)
    # one call outside the capture, without an append (cache and lengths stay as they are)
    reco.reco_decode_attn(s.kv, s.q, None, None, s.lens, _scale(case), s.out, lse, s.ws)
    torch.cuda.synchronize()
    s.graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s.graph, capture_error_mode="relaxed"):
        reco.reco_copy_row(s.pool, s.slot, s.static)
        reco.reco_decode_attn_ring(s.kv, s.q, s.kn, s.vn, s.lens, _scale(case), s.out, s.ring, s.slot, s.ws,
                                   q_ring=s.q_ring)
        reco.reco_penalty_sample(s.logits, s.ids, s.rewards, s.draws, s.tok, s.ws_sample)
    return s


def _sample_state(case, seed):
    g = _gen(seed)
    B, V = case["batch"], case["vocab"]
    s = _vocab_inputs(case, seed, B, g)
    s.fresh = _randn(g, (B, V), torch.float32, 2.0)
    s.logits = s.fresh.clone()
    s.draws = torch.rand(B, generator=g, device=DEV)
    s.tok = torch.zeros(B, dtype=torch.int32, device=DEV)
    s.beta = torch.empty(B, dtype=torch.float32, device=DEV)
    s.ws = reco.sample_workspace(B, V, DEV)
    return s


def _ppl_state(case, seed):
    s = State()
    g, rng = _gen(seed), _np(seed, 4)
    B, n, V = case["batch"], case["answer"], case["vocab"]
    s.logits = _randn(g, (B, n, V), torch.float32, 2.0)
    s.tokens = _to(rng.integers(0, V, (B, n)).astype(np.int32))
    boost = torch.zeros((B, 1, 1), device=DEV)
    boost[0::2] = 20.0  # every other answer is confident
    s.logits.scatter_add_(2, s.tokens.long().unsqueeze(-1), boost.expand(-1, n, 1))
    s.n_valid = _to(rng.integers(1, n + 1, B).astype(np.int32)) if case["ragged"] else None
    s.ppl = torch.empty(B, dtype=torch.float32, device=DEV)
    s.stop = torch.empty(B, dtype=torch.uint8, device=DEV)
    s.ws = reco.workspace(reco.RECO_OP_PPL, None, B * n, DEV)
    return s


def _tiny_workload(case, seed):
    return W.WORKLOADS["tiny"].reduced(L=case["L"], w=case["w"], pool=case["pool"], vocab=case["vocab"],
                                       n_ids=case["ids"], n_answer=case["answer"], seed=int(seed) % 1_000_000)


def _tiny_state(case, seed):
    s = State()
    s.hp = HotPath(_tiny_workload(case, seed), DEV, out_dtype=torch.float32)
    s.logits0 = s.hp.logits.clone()
    return s


def prepare(case, seed):
    kind = case["kind"]
    make = {"tiny": _tiny_state, "compress": _compress_state, "decode": _decode_state, "token": _token_state,
            "sample": _sample_state, "ppl": _ppl_state}.get(kind, _score_state)
    s = make(case, seed)
    s.case = case
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "score":
        reco.reco_score_cache(s.kv, s.q_win, s.lens, c["w"], c["pool"], _scale(c), s.scores, s.ws, keep=s.keep)
        return {"scores": s.scores}
    if kind == "score_lse":
        reco.reco_score_cache_lse(s.kv, s.q_win, s.lens, s.row_lse, c["w"], c["pool"], _scale(c), s.scores, s.ws,
                                  keep=s.keep)
        return {"scores": s.scores}
    if kind == "boundary":
        reco.reco_score_cache_lse(s.kv, s.q_win, s.lens, s.row_lse, c["w"], c["pool"], _scale(c), s.scores, s.ws,
                                  keep=s.keep)
        reco.reco_select_topm(s.kv, s.scores, s.lens, s.keep, c["w"], s.kept, s.ws_select)
        return {"scores": s.scores, "kept": s.kept}
    if kind == "compress":  # the lengths before the boundary, then the boundary
        s.lens.copy_(s.lens0)
        reco.reco_select_compact(s.kv, s.scores, s.lens, s.keep, c["w"], s.kept, s.ws)
        return {"K": s.K, "V": s.V, "kept": s.kept, "lens": s.lens}
    if kind == "decode":  # every pass appends the same token at the same length
        s.lens.copy_(s.lens0)
        reco.reco_decode_attn(s.kv, s.q, s.kn, s.vn, s.lens, _scale(c), s.out, s.lse, s.ws)
        return {"out": s.out, "lse": s.lse, "lens": s.lens, "K": s.K, "V": s.V}
    if kind == "token":
        s.lens.copy_(s.lens0)
        s.slot.zero_()
        for _ in range(c["tokens"]):
            s.graph.replay()
        return {"out": s.out, "ring": s.ring, "q_ring": s.q_ring, "logits": s.logits, "tokens": s.tok, "lens": s.lens,
                "slot": s.slot, "K": s.K, "V": s.V}
    if kind == "sample":
        s.logits.copy_(s.fresh)  # the model's logits of the token
        reco.reco_penalty_sample(s.logits, s.ids, s.rewards, s.draws, s.tok, s.ws, beta_out=s.beta)
        return {"logits": s.logits, "tokens": s.tok, "beta": s.beta}
    if kind == "ppl":
        reco.reco_answer_ppl(s.logits, s.tokens, s.n_valid, 1.1, s.ppl, s.stop, s.ws)
        return {"ppl": s.ppl, "stop": s.stop}
    hp = s.hp
    hp.reset()
    hp.logits.copy_(s.logits0)
    hp.step()
    return {"scores": hp.scores, "kept": hp.kept, "K": hp.K, "V": hp.V, "lens": hp.lens, "out": hp.out, "lse": hp.lse,
            "logits": hp.logits, "beta": hp.beta, "ppl": hp.ppl, "stop": hp.stop}


# ---------------------------------------------------------------- the same in float64
def _window_rows(case, s, dtype, chunk_bytes=2e9):
    """For each sequence and KV head: (b, h, log normalisers [layers, G*w], candidate probabilities
    summed over the window rows / G [layers, Lmax]) of Eq. 2, in `dtype`."""
    Ly, w, G = case["layers"], case["w"], case["h_q"] // case["h_kv"]
    size = 8 if dtype == torch.float64 else 4
    for b in range(case["batch"]):
        for h in range(case["h_kv"]):
            L = s.lens[:, b, h].long()
            top = int(L.max())
            step = max(1, int(chunk_bytes / (G * w * top * size)))
            lse, raw = [], []
            for l0 in range(0, Ly, step):
                ls = slice(l0, min(Ly, l0 + step))
                q = s.q_win[ls, b, h * G:(h + 1) * G].to(dtype).reshape(-1, G * w, case["d"])
                x = torch.matmul(q, s.K[ls, b, h, :top].to(dtype).transpose(1, 2)) * _scale(case)
                j = torch.arange(top, device=DEV).view(1, 1, top)
                t = torch.arange(w, device=DEV).repeat(G).view(1, -1, 1)
                x.masked_fill_(j > L[ls].view(-1, 1, 1) - w + t, -math.inf)
                z = torch.logsumexp(x, 2)
                lse.append(z)
                if dtype == torch.float64:
                    raw.append(torch.exp_(x.sub_(z.unsqueeze(2))).sum(1) / G)
                del x
            yield b, h, torch.cat(lse), (torch.cat(raw) if raw else None)


def _scores64(case, s, keep):
    out = torch.zeros(s.K.shape[:4], dtype=torch.float64, device=DEV)
    p = case["pool"]
    for b, h, _, raw in _window_rows(case, s, torch.float64):
        nc = s.lens[:, b, h].long().view(-1, 1) - case["w"]
        ok = torch.arange(raw.shape[1], device=DEV).view(1, -1) < nc
        raw = raw.masked_fill(~ok, -math.inf)
        pooled = torch.nn.functional.max_pool1d(raw.unsqueeze(0), p, 1, p // 2).squeeze(0)
        if keep is not None:
            ok = ok & (keep[b] < s.lens[:, b, h]).view(-1, 1)
        out[:, b, h, :raw.shape[1]] = torch.where(ok, pooled, 0.0)
    return out


def _attend64(q, K, V, L, scale):
    """q [layers, n, d], K and V [layers, top, d], L [layers, n] visible keys -> out, lse (float64)."""
    x = torch.matmul(q.double(), K.double().transpose(1, 2)) * scale
    j = torch.arange(K.shape[1], device=DEV).view(1, 1, -1)
    x.masked_fill_(j >= L.unsqueeze(2), -math.inf)
    lse = torch.logsumexp(x, 2)
    return torch.matmul(torch.exp(x - lse.unsqueeze(2)), V.double()), lse


def _decode64(case, K, V, q, kn, vn, lens):
    """One appended token per unit: out [layers, B, h_q, d], lse [layers, B, h_q]."""
    Ly, B, H, G = case["layers"], case["batch"], case["h_kv"], case["h_q"] // case["h_kv"]
    out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    lse = torch.zeros(q.shape[:3], dtype=torch.float64, device=DEV)
    rows = torch.arange(Ly, device=DEV)
    for b in range(B):
        for h in range(H):
            L = lens[:, b, h].long()
            top = int(L.max()) + 1
            k, v = K[:, b, h, :top].clone(), V[:, b, h, :top].clone()
            k[rows, L], v[rows, L] = kn[:, b, h], vn[:, b, h]
            hs = slice(h * G, (h + 1) * G)
            out[:, b, hs], lse[:, b, hs] = _attend64(q[:, b, hs], k, v, (L + 1).view(-1, 1).expand(-1, G), _scale(case))
    return out, lse


def _token64(case, s):
    Ly, B, Hq, H, w, N = (case[k] for k in ("layers", "batch", "h_q", "h_kv", "w", "tokens"))
    G, d = Hq // H, case["d"]
    q = torch.stack([s.pool_view(t, 0) for t in range(N)], 3)  # [layers, B, Hq, N, d]
    kn = torch.stack([s.pool_view(t, 1) for t in range(N)], 3)
    vn = torch.stack([s.pool_view(t, 2) for t in range(N)], 3)
    out = torch.zeros((Ly, B, Hq, d), dtype=torch.float64, device=DEV)
    ring = torch.zeros(s.ring.shape, dtype=torch.float64, device=DEV)
    at = torch.arange(N, device=DEV)
    for b in range(B):
        for h in range(H):
            L = s.lens0[:, b, h].long()
            top = int(L.max()) + N
            k, v = s.K[:, b, h, :top].clone(), s.V[:, b, h, :top].clone()
            rows = torch.arange(Ly, device=DEV).view(-1, 1)
            k[rows, L.view(-1, 1) + at], v[rows, L.view(-1, 1) + at] = kn[:, b, h], vn[:, b, h]
            hs = slice(h * G, (h + 1) * G)
            seen = (L.view(-1, 1) + 1 + at.view(1, -1)).unsqueeze(1).expand(-1, G, -1).reshape(Ly, G * N)
            o, z = _attend64(q[:, b, hs].reshape(Ly, G * N, d), k, v, seen, _scale(case))
            out[:, b, hs] = o.view(Ly, G, N, d)[:, :, -1]
            z = z.view(Ly, G, N).permute(2, 0, 1)
            ring[:N, :, b, hs], ring[w:w + N, :, b, hs] = z, z
    z, _ = _penalised64(s.pool_view(N - 1, 3), s.ids, s.rewards)
    return {"out": out, "ring": ring, "logits": z}


def _penalised64(logits, ids, rewards, tau_l=0.4, tau_h=0.8, beta=4.0):
    lo, hi = torch.tensor(tau_l, device=DEV), torch.tensor(tau_h, device=DEV)
    b = torch.where(rewards <= lo, 0.0, torch.where(rewards >= hi, beta, beta / 2)).double()
    z = logits.double().clone()
    z[:, ids.long()] -= b.view(-1, 1)
    return z, b


def _ppl64(logits, tokens, n_valid):
    z = logits.double()
    lp = z.gather(2, tokens.long().unsqueeze(-1)).squeeze(-1) - torch.logsumexp(z, 2)
    n = torch.full((z.shape[0],), z.shape[1], device=DEV) if n_valid is None else n_valid.long()
    on = torch.arange(z.shape[1], device=DEV).view(1, -1) < n.view(-1, 1)
    return torch.exp(-(lp * on).sum(1) / n)


def _tiny64(case, s):
    hp, wl = s.hp, s.hp.wl
    c = {**case, **_heads(wl.layers, wl.batch, wl.h_q, wl.h_kv, wl.d, "f32")}
    t = State()
    t.K, t.q_win, t.lens = hp.K0, hp.q_win, hp.lens0
    scores = _scores64(c, t, None)
    Ly, B, H = wl.layers, wl.batch, wl.h_kv
    K, V = hp.K0.clone(), hp.V0.clone()
    m, nc = int(hp.keep_host[0]), wl.L - wl.w  # one sequence
    order = torch.sort(scores[..., :nc].float(), dim=-1, descending=True, stable=True).indices[..., :m - wl.w]
    window = torch.arange(nc, wl.L, device=DEV).expand(Ly, B, H, wl.w)
    kept = torch.cat([torch.sort(order, dim=-1).values, window], -1).unsqueeze(-1).expand(-1, -1, -1, -1, wl.d)
    K[..., :m, :], V[..., :m, :] = hp.K0.gather(3, kept), hp.V0.gather(3, kept)
    out, lse = _decode64(c, K, V, hp.dq[0], hp.dk[0], hp.dv[0], torch.full_like(hp.lens0, m))
    z, beta = _penalised64(s.logits0, hp.ids, hp.rewards)
    return {"scores": scores, "out": out.unsqueeze(0), "lse": lse.unsqueeze(0), "logits": z, "beta": beta,
            "ppl": _ppl64(hp.ans_logits, hp.ans_tokens, None)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "compress":  # moves rows, computes no numbers
        return None
    s = prepare(case, seed)
    if kind == "decode":
        out, lse = _decode64(case, s.K, s.V, s.q, s.kn, s.vn, s.lens0)
        return {"out": out, "lse": lse}
    if kind == "token":
        return _token64(case, s)
    if kind == "sample":
        z, beta = _penalised64(s.fresh, s.ids, s.rewards)
        return {"logits": z, "beta": beta}
    if kind == "ppl":
        return {"ppl": _ppl64(s.logits, s.tokens, s.n_valid)}
    if kind == "tiny":
        return _tiny64(case, s)
    return {"scores": _scores64(case, s, s.keep)}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind in ("sample", "ppl"):
        n = case["batch"] * case["vocab"] * (case["answer"] if kind == "ppl" else 1)
        return {"bytes": 4.0 * n * (0.5 * (1 + 1 / case["answer"]) if case.get("ragged") else 1), "flops": 0.0}
    if kind == "tiny":
        L, w, m = case["L"], case["w"], max(case["w"], case["L"] // 4)
        units, G, d = 2, 4, 64
        by = units * (L * d * 4 + 4 * m * d * 4 + 2 * m * d * 4 + 2 * L * 4) + 4 * case["answer"] * case["vocab"]
        return {"bytes": float(by), "flops": 2.0 * units * G * d * (w * L + 2 * m)}
    Ly, B, H, d = case["layers"], case["batch"], case["h_kv"], case["d"]
    G, es = case["h_q"] // H, 4 if case["dtype"] == "f32" else 2
    mean = 0.5 * (case["lo"] + case["hi"])
    units = Ly * B * H
    if kind in ("decode", "token"):
        n = case.get("tokens", 1)
        rows = mean + 0.5 * (n + 1)
        one = units * (2 * rows * d * es + G * d * es + 4 * d * es + G * d * (4 if case.get("out") == "f32" else 2))
        if kind == "token":
            one += 4.0 * B * case["vocab"]
        return {"bytes": n * one, "flops": n * 4.0 * units * G * rows * d}
    units *= case["scored"] / B
    if kind == "compress":
        m = mean * min(1.0, case["ratio"])
        return {"bytes": units * (4 * mean + 4 * m + 4 * m * d * es), "flops": 0.0}
    by = units * (mean * d * es + G * case["w"] * d * es + 4 * mean)
    return {"bytes": by, "flops": 2.0 * units * G * case["w"] * mean * d}


def tolerance(case):
    kind = case["kind"]
    if kind in ("compress",):
        return "exact"
    if kind in ("decode", "token") and case.get("out", "bf16") == "bf16":
        # outputs rounded to bf16 (about 1.7e-3 off); a draw beside a boundary of the distribution
        # may take the next token
        return {"rel": 7e-3, "max": 3e-2, "differ": 5e-3 if kind == "token" else 0.0}
    if kind == "decode" and case["dtype"] == "bf16":  # float32 outputs, probabilities as two bf16 parts
        return {"rel": 5e-5, "max": 1e-3}
    # float32 sums; scores within rounding of the m-th may trade places
    return {"rel": 1e-5, "max": 2e-4, "differ": 5e-3}
