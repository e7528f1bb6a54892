"""The work that programs using this output head have it do, as timed cases.

A case is one call of a public entry point on inputs made from a seed:

  head    one decode step's output head: ``Head.topk`` / ``topk_sparse`` /
          ``topk_sample`` / ``topk_host`` on a bf16 or e4m3 head;
  many    the exact top-k of many hidden states (``Head.topk_many``), the
          ground truth of a Recall@k evaluation;
  recall  the hit counts of that evaluation (``recall_hits``);
  sample  top-k sampling alone (``sample_topk``).

Weights and queries follow ``paper_2608_27460_gb300.synth`` (rows s_i g_i with
g ~ N(0, 0.02^2) and log-normal s; queries three planted rows plus unit
noise), drawn on the GPU from the case's seed.
"""
import math

import numpy as np
import torch

import paper_2608_27460_gb300 as vie

TEMPERATURE, TOP_P, MIN_P = 0.8, 0.9, 0.05


def _head(name, V, d, batch, k, call, storage="bf16", dup=0.0):
    return {"name": name, "kind": "head", "V": V, "d": d, "batch": batch, "k": k, "call": call,
            "storage": storage, "dup": dup}


def listed():
    return [
        # second-stage sampling on logits a caller already holds: the smallest call, one launch
        {"name": "sample_b32_k50", "kind": "sample", "V": 151936, "batch": 32, "k": 50},
        # a small model's decode step, odd vocabulary: launch latency beside 26 MB of weights
        _head("small_20011x640_b1", 20011, 640, 1, 50, "sparse"),
        # one decode step of a single stream, sparse logits handed to logit processors
        _head("qwen3-0.6b_b1", 151936, 1024, 1, 50, "sparse"),
        # the same step end to end for a caller with page-locked host buffers
        _head("gemma3-1b_b1_host", 262144, 1152, 1, 50, "host"),
        # a decode step with its token drawn on the device
        _head("gemma3-270m_b1_sample", 262144, 640, 1, 50, "sample"),
        # a small decode batch on a vocabulary with 5 % duplicate rows (ties)
        _head("gemma3-1b-ties_b4", 262144, 1152, 4, 50, "sparse", dup=0.05),
        # a serving batch
        _head("llama3.2-3b_b64", 128256, 3072, 64, 50, "topk"),
        # quantised rows: single stream, and a batch
        _head("qwen3-0.6b_e4m3_b1", 151936, 1024, 1, 50, "topk", "e4m3"),
        _head("llama3.2-3b_e4m3_b16", 128256, 3072, 16, 50, "topk", "e4m3"),
        # wide candidate lists for rescoring; vocabulary, width and batch all odd sizes
        _head("wide_100003x1000_b5_k300", 100003, 1000, 5, 300, "topk"),
        # Recall@k bookkeeping of 20 000 states against an approximate search's candidates
        {"name": "recall_n20000_k50_m500", "kind": "recall", "V": 151936, "n": 20000, "k": 50, "m": 500},
        # the exact top-2 of 20 000 states, the paper's Recall@2 ground truth
        {"name": "many_qwen3-0.6b_n20000_k2", "kind": "many", "V": 151936, "d": 1024, "n": 20000, "k": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["head"] * 6 + ["many", "recall", "sample"])
    V = _log(rng, 16000, 262144)
    if kind == "sample":
        return {"kind": kind, "V": V, "batch": _log(rng, 1, 1024), "k": _log(rng, 1, 1024)}
    if kind == "recall":
        return {"kind": kind, "V": V, "n": _log(rng, 1000, 40000), "k": _log(rng, 1, 1024),
                "m": _log(rng, 1, 4096)}
    d = _log(rng, 256, 3072)
    if rng.random() < 0.6:
        d = (d + 63) // 64 * 64  # most models' widths; the others are odd sizes
    if kind == "many":
        n = _log(rng, 1024, 20000)
        n = max(1000, min(n, int(0.4 * 151936 * 1024 * 20000 / (V * d))))  # no dearer than the listed one
        return {"kind": kind, "V": V, "d": d, "n": n, "k": rng.choice([1, 2, 5, 10, 50])}
    storage = rng.choice(["bf16", "bf16", "e4m3"])
    call = rng.choice(["topk", "sparse", "sample", "host"])
    batch = rng.choice([1, 1, _log(rng, 2, 64), _log(rng, 2, 64)])
    if call in ("sparse", "host"):
        batch = min(batch, 8)
    k = rng.choice([1, 50, 50, _log(rng, 2, 128), _log(rng, 65, 1024)])
    case = _head("", V, d, batch, k, call, storage, rng.choice([0.0, 0.0, 0.05]))
    del case["name"]
    return case


# ---- inputs -----------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _weights(case, g):
    """bf16 W [V, d] on the GPU."""
    V, d = case["V"], case["d"]
    W = torch.empty((V, d), dtype=torch.bfloat16, device="cuda")
    for r0 in range(0, V, 32768):
        n = min(32768, V - r0)
        s = torch.exp(0.3 * torch.randn((n, 1), generator=g, device="cuda"))
        W[r0:r0 + n] = (0.02 * s) * torch.randn((n, d), generator=g, device="cuda")
    n_dup = int(case.get("dup", 0.0) * V)
    if n_dup:
        perm = torch.randperm(V, generator=g, device="cuda")
        src = perm[n_dup:][torch.randint(0, V - n_dup, (n_dup,), generator=g, device="cuda")]
        W[perm[:n_dup]] = W[src]
    return W


def _queries(W, n, g):
    """fp32 hidden states [n, d]: three planted rows each, plus unit noise."""
    V, d = W.shape
    h = torch.randn((n, d), generator=g, device="cuda")
    for _ in range(3):
        rows = torch.randint(0, V, (n,), generator=g, device="cuda")
        c = 20.0 + 2.0 * torch.randn((n, 1), generator=g, device="cuda")
        h += c * W[rows].float()
    return h


def _candidates(case, g):
    """Sorted candidates as a head returns them: int32 / fp32 [batch, k]."""
    b, k, V = case["batch"], case["k"], case["V"]
    z = 3.0 * torch.randn((b, k), generator=g, device="cuda")
    idx = (torch.arange(k, device="cuda") * (V // k) + torch.randint(0, V // k, (b, k), generator=g, device="cuda"))
    return idx.int(), torch.sort(z, dim=1, descending=True).values.contiguous()


def _recall_lists(case, g):
    """Exact lists of distinct rows, and candidates holding most of them among
    others, shuffled, with a few empty slots (what an approximate search returns)."""
    n, k, m, V = case["n"], case["k"], case["m"], case["V"]
    step = V // k
    exact = (torch.arange(k, device="cuda") * step + torch.randint(0, step, (n, k), generator=g, device="cuda")).int()
    approx = torch.randint(0, V, (n, m), generator=g, device="cuda", dtype=torch.int32)
    take = min(k, m)
    keep = torch.rand((n, take), generator=g, device="cuda") < 0.9
    approx[:, :take] = torch.where(keep, exact[:, :take], approx[:, :take])
    approx = approx[:, torch.randperm(m, generator=g, device="cuda")].contiguous()
    approx[torch.rand((n, m), generator=g, device="cuda") < 0.01] = -1
    return exact.contiguous(), approx


def _inputs(case, seed):
    g = _generator(seed)
    if case["kind"] == "sample":
        return _candidates(case, g)
    if case["kind"] == "recall":
        return _recall_lists(case, g)
    W = _weights(case, g)
    return W, _queries(W, case["n"] if case["kind"] == "many" else case["batch"], g)


def prepare(case, seed):
    s = dict(case, seed=int(seed))
    if case["kind"] == "sample":
        s["idx"], s["logits"] = _inputs(case, seed)
        b = case["batch"]
        s["tok"] = torch.empty((b,), dtype=torch.int32, device="cuda")
        s["prob"] = torch.empty((b,), dtype=torch.float32, device="cuda")
        return s
    if case["kind"] == "recall":
        s["exact"], s["approx"] = _inputs(case, seed)
        s["hits"] = torch.empty((case["n"],), dtype=torch.int32, device="cuda")
        return s
    W, h = _inputs(case, seed)
    s["head"] = vie.Head(W, storage=case.get("storage", "bf16"))
    del W
    host = case.get("call") == "host"
    n, k = h.shape[0], case["k"]
    where = {"pin_memory": True} if host else {"device": "cuda"}
    s["idx"] = torch.empty((n, k), dtype=torch.int32, **where)
    s["logits"] = torch.empty((n, k), dtype=torch.float32, **where)
    if case.get("call") in ("sparse", "host"):
        s["sparse"] = torch.empty((n, case["V"]), dtype=torch.float32, device="cuda")
    s["h"] = h.cpu().pin_memory() if host else h
    return s


def run(s):
    if s["kind"] == "sample":
        return vie.sample_topk(s["idx"], s["logits"], TEMPERATURE, TOP_P, MIN_P, seed=s["seed"], step=1,
                               out_token=s["tok"], out_prob=s["prob"])
    if s["kind"] == "recall":
        return vie.recall_hits(s["exact"], s["approx"], out_hits=s["hits"])
    head, h, k = s["head"], s["h"], s["k"]
    if s["kind"] == "many":
        return head.topk_many(h, k, out_idx=s["idx"], out_logits=s["logits"])
    if s["call"] == "sparse":
        return head.topk_sparse(h, k, out_idx=s["idx"], out_logits=s["logits"], out_sparse=s["sparse"])
    if s["call"] == "sample":
        return head.topk_sample(h, k, TEMPERATURE, TOP_P, MIN_P, seed=s["seed"], step=1)
    if s["call"] == "host":
        head.topk_host(h, k, out_idx=s["idx"], out_logits=s["logits"], out_sparse=s["sparse"])
        return s["idx"], s["logits"], s["sparse"]
    return head.topk(h, k, out_idx=s["idx"], out_logits=s["logits"])


# ---- what a pass cannot do without, and how exact it is ---------------------

def work(case):
    if case["kind"] == "sample":
        b, k = case["batch"], case["k"]
        return {"bytes": b * k * 8 + b * 8, "flops": 0}
    if case["kind"] == "recall":
        n, k, m = case["n"], case["k"], case["m"]
        return {"bytes": 4 * n * (k + m + 1), "flops": 0}
    V, d, k = case["V"], case["d"], case["k"]
    n = case["n"] if case["kind"] == "many" else case["batch"]
    w = V * d + 4 * V if case.get("storage") == "e4m3" else 2 * V * d
    out = n * k * 8
    if case.get("call") in ("sparse", "host"):
        out += 4 * n * V
    if case.get("call") == "sample":
        out += 8 * n
    return {"bytes": w + 4 * n * d + out, "flops": 2 * V * d * n}


def tolerance(case):
    if case["kind"] == "recall":
        return "exact"  # integer counts
    if case["kind"] == "sample":
        # fp32 softmax and prefix sums of k terms; a draw on a boundary may go either way
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    # 32-bit sums of d products: logits about 1e-6 off; neighbours whose logits
    # are closer than that may swap places, the more of them the longer the list
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}


# ---- the same in 64 bits ----------------------------------------------------

def _philox_uniform(seed, step, queries):
    """Top 24 bits of the first word of Philox4x32-10 (Salmon et al., SC 2011)
    at counter (step lo, step hi, query, 0), key (seed lo, seed hi), as [0, 1)."""
    mask = 0xFFFFFFFF
    u = np.empty(queries)
    for q in range(queries):
        c = [step & mask, step >> 32 & mask, q, 0]
        key = [seed & mask, seed >> 32 & mask]
        for r in range(10):
            if r:
                key = [(key[0] + 0x9E3779B9) & mask, (key[1] + 0xBB67AE85) & mask]
            p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
            c = [p1 >> 32 ^ c[1] ^ key[0], p1 & mask, p0 >> 32 ^ c[3] ^ key[1], p0 & mask]
        u[q] = (c[0] >> 8) / 16777216.0
    return u


def _draw(idx, z, seed):
    """Tokens and their probabilities drawn from sorted fp64 logits z [b, k]."""
    idx, z = idx.cpu().numpy(), z.double().cpu().numpy()
    b, k = z.shape
    e = np.exp((z - z[:, :1]) / TEMPERATURE)
    p = e / e.sum(1, keepdims=True)
    C = np.cumsum(p, 1)
    u = _philox_uniform(seed, 1, b)
    tok, prob = np.empty(b, np.int32), np.empty(b)
    for q in range(b):
        n_p = min(int(np.searchsorted(C[q], TOP_P)) + 1, k)
        n = max(1, min(n_p, int(np.sum(p[q] >= MIN_P * p[q, 0]))))
        j = min(int(np.searchsorted(C[q, :n], u[q] * C[q, n - 1], side="right")), n - 1)
        tok[q], prob[q] = idx[q, j], p[q, j] / C[q, n - 1]
    return torch.from_numpy(tok), torch.from_numpy(prob)


def _dequantised(W):
    """The e4m3 rows with one fp32 scale each, as fp64 [V, d]."""
    w = W.float()
    amax = w.abs().amax(dim=1, keepdim=True)
    top = torch.full_like(amax, 448.0)  # a tensor: torch multiplies by 1 / x for a plain number
    scale = torch.where(amax > 0, amax / top, torch.ones_like(amax))
    q = (w / scale).clamp(-448.0, 448.0).to(torch.float8_e4m3fn)
    return q.double(), scale.double()


def _exact_topk(W, h, k, storage):
    """Top-k by (logit, smaller row first) of the fp64 logits of every query."""
    if storage == "e4m3":
        Wd, scale = _dequantised(W)
    else:
        Wd, scale = W.double(), None
    idx, val = [], []
    for q0 in range(0, h.shape[0], 1024):
        z = h[q0:q0 + 1024].double() @ Wd.t()
        if scale is not None:
            z *= scale.t()
        v, i = torch.topk(z, k, dim=1)
        order = torch.argsort(i, dim=1)  # equal logits (duplicate rows): smaller row first
        v, i = v.gather(1, order), i.gather(1, order)
        order = torch.sort(v, dim=1, descending=True, stable=True).indices
        idx.append(i.gather(1, order).int())
        val.append(v.gather(1, order))
    return torch.cat(idx), torch.cat(val)


def exact(case, seed):
    if case["kind"] == "recall":
        return None  # integer counts, compared bit for bit
    if case["kind"] == "sample":
        idx, z = _inputs(case, seed)
        return _draw(idx, z, int(seed))
    W, h = _inputs(case, seed)
    idx, val = _exact_topk(W, h, case["k"], case.get("storage", "bf16"))
    if case.get("call") in ("sparse", "host"):
        sparse = torch.full((h.shape[0], case["V"]), -math.inf, dtype=torch.float64, device="cuda")
        sparse.scatter_(1, idx.long(), val)
        return idx, val, sparse
    if case.get("call") == "sample":
        tok, prob = _draw(idx, val, int(seed))
        return idx, val, tok, prob
    return idx, val
