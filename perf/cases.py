"""Cases that time the library through its public entry points.

Each listed case is one call that a program using this library makes, on
inputs of the sizes and distributions of the repository's own workloads
(``synth.py``, ``bench.py``, the tests): the paper's edge matrix, all-pairs
top-k lists (raw, normalised and substitution-matrix scoring), queries, explicit
pairs, batches of dictionaries, and the stages of the learned proposal.
``draw`` gives further cases of the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_01654_gb300 import nw, synth

ALPHABET = 40
PAPER = "1 -1 -1"  # match, mismatch, gap


def listed():
    return [
        # the paper's first experiment at its small end: every int8 edge of 2,000 words (launch-bound)
        {"name": "matrix_2000", "kind": "matrix", "n": 2000},
        # the flagship: exact top-10 graph and histogram of a 600,000-word dictionary
        {"name": "topk_600000", "kind": "topk", "n": 600000, "k": 10, "hist": True, "scoring": PAPER},
        # Section 5's normalised ranking on an ordinary dictionary of odd size
        {"name": "topk_norm_30011", "kind": "topk_norm", "n": 30011, "k": 10, "scoring": PAPER},
        # per-phoneme similarity coefficients (a full substitution matrix), top-10 and histogram
        {"name": "topk_sim_40009", "kind": "topk_sim", "n": 40009, "k": 10},
        # one interactive lookup: a single query word against a dictionary, host buffers (latency)
        {"name": "query_1", "kind": "query", "n": 100000, "nq": 1, "k": 10, "device": False},
        # a full serving batch against the flagship dictionary, device buffers
        {"name": "query_4096", "kind": "query", "n": 600000, "nq": 4096, "k": 10, "device": True},
        # a list of explicit pairs scored on the device (training labels, spot checks), another scoring
        {"name": "pairs_1000003", "kind": "pairs", "n": 100000, "m": 1000003, "scoring": "2 -1 -2"},
        # independent dictionaries of uneven size, alphabet and scoring, each with its queries, in one graph
        {"name": "batch_16", "kind": "batch", "dicts": 16, "size_lo": 500, "size_hi": 8000, "k": 10, "shape": 3},
        # embeddings of a dictionary (forward pass of the character CNN)
        {"name": "embed_200003", "kind": "embed", "n": 200003},
        # loss and gradient of one training batch (forward and backward pass)
        {"name": "grad_8192", "kind": "grad", "n": 50000, "m": 8192},
        # the candidate stage alone: each row's 256 largest exact integer products among 100,000 rows
        {"name": "dot_topk_100003", "kind": "dot", "n": 100003, "C": 256},
        # the whole proposal: embed, quantise, 512 candidates a word, exact rescoring, top-10
        {"name": "proposal_100000", "kind": "proposal", "n": 100000, "C": 512, "k": 10},
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matrix", "topk", "topk", "topk_norm", "topk_sim", "query", "query", "pairs", "batch", "embed",
                       "grad", "dot", "proposal"])
    k = rng.choice([1, 5, 10, 10, 25])
    if kind == "matrix":
        return {"kind": kind, "n": _logu(rng, 100, 20000)}
    if kind == "topk":
        return {"kind": kind, "n": _logu(rng, 300, 200000), "k": k, "hist": rng.random() < 0.75,
                "scoring": rng.choice([PAPER, PAPER, "0 -1 -1", "2 -1 -2", "1 -2 -1"])}
    if kind == "topk_norm":
        return {"kind": kind, "n": _logu(rng, 300, 100000), "k": k, "scoring": PAPER}
    if kind == "topk_sim":
        return {"kind": kind, "n": _logu(rng, 300, 100000), "k": k}
    if kind == "query":
        return {"kind": kind, "n": _logu(rng, 5000, 600000), "nq": _logu(rng, 1, 4096), "k": k,
                "device": rng.random() < 0.5}
    if kind == "pairs":
        return {"kind": kind, "n": _logu(rng, 1000, 300000), "m": _logu(rng, 1000, 4000000),
                "scoring": rng.choice([PAPER, "2 -1 -2", "0 -1 -1"])}
    if kind == "batch":
        hi = _logu(rng, 1000, 12000)
        return {"kind": kind, "dicts": rng.randint(3, 24), "size_lo": max(2, hi // rng.randint(2, 20)), "size_hi": hi,
                "k": k, "shape": rng.randint(1, 10 ** 6)}
    if kind == "embed":
        return {"kind": kind, "n": _logu(rng, 1000, 300000)}
    if kind == "grad":
        return {"kind": kind, "n": _logu(rng, 1000, 100000), "m": _logu(rng, 64, 16384)}
    if kind == "dot":
        return {"kind": kind, "n": _logu(rng, 1000, 150000), "C": rng.choice([32, 100, 256, 384, 512])}
    return {"kind": kind, "n": _logu(rng, 2000, 150000), "C": rng.choice([64, 128, 256, 512]), "k": min(k, 10)}


# ---------------------------------------------------------------------------
# inputs

def _dictionary_words(n, seed):
    """A frequency-sorted dictionary: lengths round(N(8, 3)) on [1, 25], Zipf(1.1) codes."""
    return synth.make_words(n, ALPHABET, 1.1, 8.0, 3.0, 1, 25, seed=seed)


def _scoring(text):
    return tuple(int(v) for v in text.split())


def _lengths_law(mu=8.0, sigma=3.0, lo=1, hi=25):
    p = synth.rounded_normal_probs(mu, sigma, lo, hi)
    return np.arange(lo, hi + 1, dtype=np.float64), p


def _similarity_table():
    """A phoneme-like table: 3 for equal codes, 1 for neighbouring ones, else -2."""
    c = np.arange(ALPHABET)
    d = np.abs(c[:, None] - c[None, :])
    return np.where(d == 0, 3, np.where(d <= 1, 1, -2)).astype(np.int32)


def _cuda(a):
    return torch.from_numpy(a).cuda()


def _csr_cuda(w):
    return _cuda(w.codes), _cuda(w.offsets.view(np.int32))


def _lists(n, k):
    return (torch.empty((n, k), dtype=torch.int32, device="cuda"),
            torch.empty((n, k), dtype=torch.int16, device="cuda"))


CH, EMB, OUT = 128, 32, 64


def _param_blocks(p):
    """The flat parameter vector as named blocks (the layout of include/nw_proposal.h)."""
    shapes = [("emb", (ALPHABET, EMB)), ("W1", (CH, 3, EMB)), ("b1", (CH,)), ("W2", (CH, 3, CH)), ("b2", (CH,)),
              ("W3", (CH, 3, CH)), ("b3", (CH,)), ("Wl", (OUT, CH)), ("bl", (OUT,))]
    out, at = {}, 0
    for name, sh in shapes:
        size = int(np.prod(sh))
        out[name] = p[at:at + size].reshape(sh)
        at += size
    assert at == p.shape[0]
    return out


def _network(words, seed):
    """Parameters standing in for a trained network: random features, and an output layer that centres the
    pooled features and keeps their principal directions, fitted on a sample of the words in float64."""
    r = np.random.default_rng([seed, 77])
    size = ALPHABET * EMB + CH * 3 * EMB + CH + 2 * (CH * 3 * CH + CH) + OUT * CH + OUT
    p = np.zeros(size, np.float32)
    b = _param_blocks(p)
    b["emb"][:] = r.uniform(-1.7, 1.7, b["emb"].shape)
    for name, fan in (("W1", 3 * EMB), ("W2", 3 * CH), ("W3", 3 * CH)):
        b[name][:] = r.uniform(-1, 1, b[name].shape) * math.sqrt(6.0 / fan)
    for name in ("b1", "b2", "b3"):
        b[name][:] = r.uniform(-0.2, 0.2, CH)
    m = min(words.n, 1500)
    pooled = _pooled({k: torch.from_numpy(v.astype(np.float64)) for k, v in b.items()},
                     torch.from_numpy(words.codes[:int(words.offsets[m])].astype(np.int64)),
                     torch.from_numpy(words.offsets[:m + 1].astype(np.int64))).numpy()
    mean = pooled.mean(0)
    w, v = np.linalg.eigh(np.cov((pooled - mean).T))
    order = np.argsort(-w)[:OUT - 1]
    v = v[:, order] * np.sign(v[np.argmax(np.abs(v[:, order]), axis=0), np.arange(OUT - 1)])
    b["Wl"][:OUT - 1] = (v / np.sqrt(np.sqrt(np.maximum(w[order], 1e-4)))).T
    b["Wl"][OUT - 1] = r.uniform(-0.02, 0.02, CH)
    b["bl"][:] = -(b["Wl"].astype(np.float64) @ mean)
    return p


def _pooled(b, codes, offsets):
    """Mean-pooled features of words in CSR form, in the blocks' precision (float64): three width-3
    convolutions with ReLU, zero outside the word."""
    P = codes.shape[0]
    lens = offsets[1:] - offsets[:-1]
    word = torch.repeat_interleave(torch.arange(lens.shape[0], device=codes.device), lens)
    at = torch.arange(P, device=codes.device)
    prev = torch.where(at == offsets[word], P, at - 1)
    nxt = torch.where(at + 1 == offsets[word + 1], P, at + 1)
    x = b["emb"][codes]
    for W, bias in (("W1", "b1"), ("W2", "b2"), ("W3", "b3")):
        x = torch.cat([x, torch.zeros_like(x[:1])])
        y = b[bias] + x[prev] @ b[W][:, 0].T + x[:-1] @ b[W][:, 1].T + x[nxt] @ b[W][:, 2].T
        x = torch.relu(y)
    pooled = torch.zeros((lens.shape[0], CH), dtype=x.dtype, device=x.device).index_add(0, word, x)
    return pooled / torch.clamp(lens, min=1).to(x.dtype)[:, None]


def _embed64(b, codes, offsets):
    return _pooled(b, codes, offsets) @ b["Wl"].T + b["bl"]


def _grad_inputs(case, seed):
    w = _dictionary_words(case["n"], seed)
    r = np.random.default_rng([seed, 5])
    i = r.integers(0, w.n, case["m"])
    j = (i + r.integers(1, w.n, case["m"])) % w.n
    target = np.clip(r.normal(-0.2, 0.35, case["m"]), -1, 1).astype(np.float32)
    return w, i.astype(np.uint32), j.astype(np.uint32), target


def _batch_inputs(case, seed):
    """Uneven dictionaries with their query sets; `shape` fixes sizes, alphabets and scorings, the seed the words."""
    shapes = synth.uniform01(case["shape"], synth.STREAM_MISC, 6 * case["dicts"]).reshape(-1, 6)
    lo, hi = math.log(case["size_lo"]), math.log(case["size_hi"])
    out = []
    for d, u in enumerate(shapes):
        n, alpha = int(math.exp(lo + u[0] * (hi - lo))), 40 + int(u[1] * 81)
        sc = (1 + int(u[2] * 3), -1 - int(u[3] * 3), -1 - int(u[4] * 4))
        nq = int(math.exp(u[5] * math.log(1000)))
        w = synth.make_uniform_length_words(n, alpha, 1.0, 1, 40, seed=1000 * seed + d, length_stream=1, code_stream=2)
        q = synth.make_uniform_length_words(nq, alpha, 1.0, 1, 40, seed=1000 * seed + d)
        out.append((w.codes, w.offsets, alpha, sc, (q.codes, q.offsets)))
    return out


def prepare(case, seed):
    kind = case["kind"]
    ctx = nw.Context(0)
    st = {"kind": kind, "ctx": ctx}
    if kind == "matrix":
        w = synth.make_words(case["n"], ALPHABET, 1.0, 7.0, 2.5, 2, 16, seed=seed)
        st["d"] = ctx.load_dictionary(*_csr_cuda(w), ALPHABET, _scoring(PAPER))
        st["out"] = torch.empty(w.n * (w.n - 1) // 2, dtype=torch.int8, device="cuda")
    elif kind in ("topk", "topk_norm", "topk_sim"):
        w = _dictionary_words(case["n"], seed)
        if kind == "topk_sim":
            st["d"] = ctx.load_dictionary_sim(*_csr_cuda(w), ALPHABET, _similarity_table(), -2)
        else:
            st["d"] = ctx.load_dictionary(*_csr_cuda(w), ALPHABET, _scoring(case["scoring"]))
        st["k"] = case["k"]
        st["idx"], st["score"] = _lists(w.n, case["k"])
        # the normalised ranking is asked for lists alone, the others for the histogram as well
        st["hist"] = (torch.empty(256, dtype=torch.int64, device="cuda")  # at least info()["nbins"]
                      if case.get("hist", kind == "topk_sim") else None)
    elif kind == "query":
        w = _dictionary_words(case["n"], seed)
        q = synth.serving_queries(case["nq"], seed=seed + 1)
        st["d"] = ctx.load_dictionary(*_csr_cuda(w), ALPHABET, _scoring(PAPER))
        st["k"] = case["k"]
        if case["device"]:
            st["q"] = _csr_cuda(q)
            st["idx"], st["score"] = _lists(q.n, case["k"])
        else:
            st["q"] = (q.codes, q.offsets)
            st["idx"] = np.empty((q.n, case["k"]), np.uint32)
            st["score"] = np.empty((q.n, case["k"]), np.int16)
    elif kind == "pairs":
        w = _dictionary_words(case["n"], seed)
        st["d"] = ctx.load_dictionary(*_csr_cuda(w), ALPHABET, _scoring(case["scoring"]))
        g = torch.Generator(device="cuda").manual_seed(seed)
        st["i"] = torch.randint(0, w.n, (case["m"],), generator=g, device="cuda", dtype=torch.int32)
        st["j"] = torch.randint(0, w.n, (case["m"],), generator=g, device="cuda", dtype=torch.int32)
        st["out"] = torch.empty(case["m"], dtype=torch.int16, device="cuda")
    elif kind == "batch":
        dicts = _batch_inputs(case, seed)
        st["batch"] = nw.Batch(ctx, dicts, k=case["k"])
        st["outs"] = [_lists(d[1].size - 1, case["k"]) for d in dicts]
        st["qouts"] = [_lists(d[4][1].size - 1, case["k"]) for d in dicts]
    elif kind in ("embed", "proposal"):
        w = _dictionary_words(case["n"], seed)
        st["d"] = ctx.load_dictionary(*_csr_cuda(w), ALPHABET, _scoring(PAPER))
        st["model"] = nw.Model(ctx, ALPHABET, seed=seed)
        st["model"].set_params(_network(w, seed))
        if kind == "embed":
            st["out"] = torch.empty((w.n, OUT), dtype=torch.float32, device="cuda")
        else:
            st["C"], st["k"] = case["C"], case["k"]
            st["idx"], st["score"] = _lists(w.n, case["k"])
    elif kind == "grad":
        w, st["i"], st["j"], st["target"] = _grad_inputs(case, seed)
        st["d"] = ctx.load_dictionary(*_csr_cuda(w), ALPHABET, _scoring(PAPER))
        st["model"] = nw.Model(ctx, ALPHABET, seed=seed)
        st["model"].set_params(_network(w, seed))
    elif kind == "dot":
        # quantised embeddings in clusters of similar words with a spread of sizes, biases against the larger ones
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["n"]
        centres = torch.randn((max(2, n // 50), OUT - 1), generator=g, device="cuda") * 18
        centres *= torch.linspace(2.2, 0.4, OUT - 1, device="cuda")
        pick = torch.randint(0, centres.shape[0], (n,), generator=g, device="cuda")
        x = centres[pick] + 7 * torch.randn((n, OUT - 1), generator=g, device="cuda")
        q = torch.zeros((n, OUT), dtype=torch.int8, device="cuda")
        q[:, :OUT - 1] = torch.clamp(torch.round(x), -127, 127).to(torch.int8)
        st["q"] = q
        st["bias"] = (-0.4 * (q.float() ** 2).sum(1)).to(torch.int32)
        st["C"] = case["C"]
    torch.cuda.synchronize()
    return st


def run(state):
    kind = state["kind"]
    if kind == "matrix":
        return state["d"].all_pairs_matrix(out=state["out"])
    if kind in ("topk", "topk_norm", "topk_sim"):
        idx, score, hist, lo = state["d"].all_pairs_topk(state["k"], state["idx"], state["score"],
                                                         hist=state["hist"] if state["hist"] is not None else False,
                                                         normalised=kind == "topk_norm")
        return (idx, score, lo) if hist is None else (idx, score, hist, lo)
    if kind == "query":
        return state["d"].query(*state["q"], state["k"], state["idx"], state["score"])
    if kind == "pairs":
        return state["d"].score_pairs(state["i"], state["j"], out=state["out"])
    if kind == "batch":
        outs, qouts = state["batch"].run_queries(state["outs"], state["qouts"])
        return [t for pair in outs + qouts for t in pair]
    if kind == "embed":
        return state["model"].embed(state["d"], out=state["out"])
    if kind == "grad":
        return state["model"].loss_grad(state["d"], state["i"], state["j"], state["target"])
    if kind == "dot":
        return nw.dot_topk(state["ctx"], state["q"], state["C"], bias=state["bias"], locality=True)
    idx, score, _ = state["model"].proposal_topk(state["d"], state["C"], state["k"], state["idx"], state["score"])
    return idx, score


# ---------------------------------------------------------------------------
# the work of one pass, and its values in 64 bits

def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: three per cell of Algorithm 1 (an addition and
    two maxima), two per multiply-add of a product.  Sizes are the expected ones of the length distributions."""
    kind = case["kind"]
    k = case.get("k", 0)
    x, p = _lengths_law(7.0, 2.5, 2, 16) if kind == "matrix" else _lengths_law()
    mean = float((x * p).sum())
    ux = 20.5 if kind == "batch" else 15.5  # mean length of uniform lengths (batches: 1..40, queries: 1..30)
    conv = 2.0 * CH * (3 * EMB + 2 * 3 * CH)  # forward operations of one word position
    if kind == "matrix":
        e = case["n"] * (case["n"] - 1) / 2
        return {"bytes": case["n"] * (mean + 4) + e, "flops": 3 * e * mean * mean}
    if kind in ("topk", "topk_norm", "topk_sim"):
        n = case["n"]
        return {"bytes": n * (mean + 4) + 6 * n * k, "flops": 3 * n * (n - 1) / 2 * mean * mean}
    if kind == "query":
        n, nq = case["n"], case["nq"]
        return {"bytes": n * (mean + 4) + nq * (ux + 4 + 6 * k), "flops": 3.0 * n * nq * mean * ux}
    if kind == "pairs":
        return {"bytes": case["n"] * (mean + 4) + 10 * case["m"], "flops": 3 * case["m"] * mean * mean}
    if kind == "batch":
        u = synth.uniform01(case["shape"], synth.STREAM_MISC, 6 * case["dicts"]).reshape(-1, 6)
        n = np.exp(math.log(case["size_lo"]) + u[:, 0] * math.log(case["size_hi"] / case["size_lo"]))
        nq = np.exp(u[:, 5] * math.log(1000))
        return {"bytes": float(((n + nq) * (ux + 4 + 6 * k)).sum()),
                "flops": float((3 * (n * n / 2 + n * nq) * ux * ux).sum())}
    if kind == "embed":
        n = case["n"]
        return {"bytes": n * (mean + 4 + 4 * OUT), "flops": n * (mean * conv + 2.0 * CH * OUT)}
    if kind == "grad":
        m = 2 * case["m"]
        return {"bytes": m * (mean + 4) + 8 * case["m"] + 8 * 120000, "flops": 3 * m * (mean * conv + 2.0 * CH * OUT)}
    n, C = case["n"], case["C"]
    if kind == "dot":
        return {"bytes": n * (OUT + 4) + 8.0 * n * C, "flops": 2.0 * n * n * OUT}
    return {"bytes": n * (mean + 4) + 6 * n * k,
            "flops": n * mean * conv + 2.0 * n * n * OUT + 3.0 * n * C * mean * mean}


def exact(case, seed):
    """What run returns, in 64 bits: embeddings, or loss and gradient.  The other cases return whole numbers."""
    if case["kind"] == "embed":
        w = _dictionary_words(case["n"], seed)
        b = {k: torch.from_numpy(v.astype(np.float64)).cuda() for k, v in _param_blocks(_network(w, seed)).items()}
        codes, offs = _cuda(w.codes.astype(np.int64)), _cuda(w.offsets.astype(np.int64))
        out = []
        for lo in range(0, w.n, 50000):
            hi = min(w.n, lo + 50000)
            out.append(_embed64(b, codes[offs[lo]:offs[hi]], offs[lo:hi + 1] - offs[lo]))
        return torch.cat(out)
    if case["kind"] == "grad":
        w, i, j, target = _grad_inputs(case, seed)
        p = torch.from_numpy(_network(w, seed).astype(np.float64)).cuda().requires_grad_()
        both = w.subset(np.concatenate([i, j]).astype(np.int64))
        e = _embed64(_param_blocks(p), _cuda(both.codes.astype(np.int64)), _cuda(both.offsets.astype(np.int64)))
        a, c = e[:case["m"]], e[case["m"]:]
        pred = (a[:, :-1] * c[:, :-1]).sum(1) + a[:, -1] + c[:, -1]
        loss = ((pred - _cuda(target.astype(np.float64))) ** 2).mean()
        loss.backward()
        return float(loss), p.grad.cpu().numpy()
    return None
