"""The work whose time counts: scoring calls, the attention read-out and the cache gradient, through the
public binding, over the sizes this library is used at.

A case is a dict of plain values:
  kind       "score" (Scorer.score_async), "attention" (kvprm_attention), "grad" (kvprm_score_grad)
  layers, d, nq, nkv, hd, ff     the scorer's shape (attention: one layer's heads; d and ff unused)
  n          candidates
  cache      "equal":  every candidate its own `len` tokens
             "ragged": every candidate its own length, len/16 .. len (any remainder, one empty cache)
             "prefix": a prefix of `prefix` tokens that all candidates read, then `len` tokens of their own
             "tree":   leaves of a tree with `fanout` children a node and edges of len/8 .. len tokens
  shape_seed draws the ragged lengths and edges (the sizes belong to the case, the values to the seed)
  rank       the scorer adapter's rank (0: merged weights);  depth: verify tokens per candidate
"""
import math
import random

import numpy as np
import torch

import paper_2607_09153_gb300 as kp

PAGE = 16
BASE, EPS = 1e4, 1e-6
ALPHA = 32.0   # the adapter's alpha, its scale is alpha / rank

SHAPES = {   # the scorer shapes of the repository's workloads, and a head_dim 64 one between them
    "tiny": dict(d=256, nq=4, nkv=2, hd=64, ff=1024),
    "small64": dict(d=1024, nq=16, nkv=4, hd=64, ff=4096),
    "1p5b": dict(d=1536, nq=12, nkv=2, hd=128, ff=8960),
    "7b": dict(d=3584, nq=28, nkv=4, hd=128, ff=18944),
    "8b": dict(d=4096, nq=32, nkv=8, hd=128, ff=14336),
}


def _case(name, kind, shape, layers, n, cache, len_, prefix=0, fanout=4, rank=0, depth=1, shape_seed=1):
    c = dict(name=name, kind=kind, layers=layers, n=n, cache=cache, len=len_, prefix=prefix, fanout=fanout, rank=rank,
             depth=depth, shape_seed=shape_seed)
    c.update(SHAPES[shape])
    return c


def listed():
    return [
        # the smallest call: a handful of short trajectories on a small scorer, latency and launches only
        _case("score_tiny", "score", "tiny", 2, 4, "equal", 128),
        # best-of-16 over finished answers of ordinary length: small batch, weights and cache both count
        _case("score_1p5b", "score", "1p5b", 28, 16, "equal", 2048),
        # the same scorer as a rank-256 adapter over the generator's own weights
        _case("score_adapter_1p5b", "score", "1p5b", 28, 16, "equal", 2048, rank=256),
        # a depth-4 readout (four verify tokens a candidate) of trajectories that stopped at different lengths
        _case("score_depth_ragged_1p5b", "score", "1p5b", 28, 12, "ragged", 3001, depth=4),
        # beam search: 64 siblings behind one long prefix
        _case("score_beam_7b", "score", "7b", 28, 64, "prefix", 512, prefix=4096),
        # tree search: 256 leaves, four levels of edges read by 64, 16, 4 and 1 leaves
        _case("score_tree_7b", "score", "7b", 28, 256, "tree", 2048),
        # few agents with long contexts: the cache is nearly all of the traffic
        _case("score_long_8b", "score", "8b", 32, 8, "equal", 32768),
        # early pruning of a wide batch with short, uneven caches: projections are nearly all of the time
        _case("score_wide_short_7b", "score", "7b", 4, 201, "ragged", 333),
        # the attention step alone, for a runtime that does its own projections: uneven lengths
        _case("attention_ragged_7b", "attention", "7b", 1, 37, "ragged", 9001),
        # the same on the narrow head, siblings behind a prefix that ends inside a page
        _case("attention_prefix_hd64", "attention", "small64", 1, 24, "prefix", 517, prefix=2503),
        # steering: the loss's gradient in every cached key and value, distinct caches
        _case("grad_1p5b", "grad", "1p5b", 28, 16, "equal", 2048),
        # the same for beam siblings, whose prefix collects the gradient of all of them
        _case("grad_beam_7b", "grad", "7b", 4, 32, "prefix", 500, prefix=4096),
    ]


def draw(rng):
    def logint(lo, hi):
        return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))

    while True:
        kind = rng.choice(["score", "score", "score", "attention", "grad"])
        shape = rng.choice(["tiny", "small64", "1p5b", "7b", "8b"])
        cache = rng.choice(["equal", "ragged", "prefix", "tree"])
        fanout = rng.choice([2, 3, 4, 8])
        n = logint(1, 256 if kind != "grad" else 64)
        prefix = logint(64, 8192) if cache == "prefix" else 0
        len_ = logint(16, {"equal": 32768, "ragged": 32768, "prefix": 2048, "tree": 2048}[cache])
        layers = 1 if kind == "attention" else logint(1, 12 if kind == "score" else 4)
        rank = depth = 0
        if kind == "score":
            option = rng.choice(["plain", "plain", "plain", "rank", "depth"])
            rank = rng.choice([64, 256]) if option == "rank" else 0
            depth = rng.choice([2, 3, 4]) if option == "depth" else 1
        c = _case("", kind, shape, layers, n, cache, len_, prefix, fanout, rank, depth or 1, rng.randrange(1 << 30))
        del c["name"]
        if n * c["depth"] > 256:
            continue
        s = _structure(c)
        rows = sum(s.lens)
        # no dearer than the largest listed case, and outputs and caches of a few GB
        if rows * layers > 1 << 22 or rows * c["nq"] * c["hd"] * layers > 1 << 33:
            continue
        if s.n_pages * layers * 2 * c["nkv"] * PAGE * c["hd"] * 2 > (8 << 30 if kind != "grad" else 2 << 30):
            continue
        return c


# ---------------------------------------------------------------- which tokens each candidate reads
class _Structure:
    """lens [n], table [n][blocks] of page numbers 0 .. n_pages - 1.  Two candidates share a page when
    all of its 16 tokens belong to edges both of them pass through at the same positions."""

    def __init__(self, paths):
        self.lens = [sum(length for _, length in p) for p in paths]
        pages = {}
        self.table = np.zeros((len(paths), max(1, max((L + PAGE - 1) // PAGE for L in self.lens))), np.int32)
        for b, path in enumerate(paths):
            end, node = 0, iter(path)
            name = None
            for j in range((self.lens[b] + PAGE - 1) // PAGE):
                last = min(PAGE * (j + 1), self.lens[b])
                while end < last:
                    name, length = next(node)
                    end += length
                # a page the candidate only partly fills is its own
                key = (name, j) if last == PAGE * (j + 1) else ("tail", b)
                self.table[b, j] = pages.setdefault(key, len(pages))
        self.n_pages = max(1, len(pages))
        self.used = sum((L + PAGE - 1) // PAGE for L in self.lens)
        self.unique = len(pages)


def _structure(c):
    rng = random.Random(c["shape_seed"])
    n, L = c["n"], c["len"]
    if c["cache"] == "equal":
        return _Structure([[(("own", b), L)] for b in range(n)])
    if c["cache"] == "ragged":
        lens = [rng.randint(max(1, L // 16), L) for _ in range(n)]
        if n > 2:
            lens[n // 2] = 0   # a trajectory that has not started
        return _Structure([[(("own", b), lens[b])] for b in range(n)])
    if c["cache"] == "prefix":
        return _Structure([[(("prefix",), c["prefix"]), (("own", b), L)] for b in range(n)])
    levels = max(1, math.ceil(math.log(n, c["fanout"]) - 1e-9)) if n > 1 else 1
    edge, paths = {}, []
    for b in range(n):
        path = []
        for lv in range(1, levels + 1):
            node = (lv, b * c["fanout"] ** lv // c["fanout"] ** levels)
            if node not in edge:
                edge[node] = rng.randint(max(1, L // 8), L)
            path.append((node, edge[node]))
        paths.append(path)
    return _Structure(paths)


# ---------------------------------------------------------------- inputs
def _normal(shape, std, gen, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=gen)


def _inputs(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = _structure(c)
    d, nq, nkv, hd, ff, layers, r = (c[k] for k in ("d", "nq", "nkv", "hd", "ff", "layers", "rank"))
    # a few pages that no candidate references, and the pages in no particular order
    total = s.n_pages + 3
    order = np.random.default_rng(seed).permutation(total).astype(np.int32)
    x = dict(lens=np.asarray(s.lens, np.int32), table=np.ascontiguousarray(order[s.table]), n_pages=total)
    x["pool"] = _normal((layers, total, 2, nkv, PAGE, hd), 1.0, gen)
    if c["kind"] == "attention":
        d, ff = 64, 64
        x["q"] = _normal((c["n"], nq, hd), 1.7, gen, torch.float32)   # score spread of a few units, as a scorer's
        x["k_self"] = _normal((c["n"], nkv, hd), 1.0, gen, torch.float32)
        x["v_self"] = _normal((c["n"], nkv, hd), 1.0, gen, torch.float32)

    def gain(k):
        return 1.0 + _normal((k,), 0.1, gen)

    def layer():
        w_qkv = _normal(((nq + 2 * nkv) * hd, d), 0.02, gen)
        # scores q.k / sqrt(hd) with a spread of 2.5: softmax weights concentrated on few of many tokens
        w_qkv[:nq * hd].normal_(0.0, 2.5 / math.sqrt(d), generator=gen)
        return dict(attn_norm=gain(d), w_qkv=w_qkv, w_o=_normal((d, nq * hd), 0.02, gen), mlp_norm=gain(d),
                    w_gate_up=_normal((2 * ff, d), 0.02, gen), w_down=_normal((d, ff), 0.02, gen))

    x["weights"] = dict(embed_verify=_normal((d,), 1.0, gen), final_norm=gain(d), w_plus=_normal((d,), 0.02, gen),
                        w_minus=_normal((d,), 0.02, gen), layers=[layer() for _ in range(layers)])
    if r:
        dims = dict(qkv=((nq + 2 * nkv) * hd, d), o=(d, nq * hd), gate_up=(2 * ff, d), down=(d, ff))
        x["factors"] = []
        for _ in range(layers):
            f = {}
            for k, (out, inp) in dims.items():
                f["a_" + k] = _normal((r, inp), 0.02, gen)
                f["b_" + k] = _normal((out, r), 0.02, gen)
            x["factors"].append(f)
    return x


def prepare(case, seed):
    c = case
    x = _inputs(c, seed)
    d, ff = (64, 64) if c["kind"] == "attention" else (c["d"], c["ff"])
    x["scorer"] = kp.Scorer(c["layers"], d, c["nq"], c["nkv"], c["hd"], ff, x["weights"],
                            max_candidates=c["n"] * c["depth"], max_blocks_per_seq=x["table"].shape[1])
    if c["rank"]:
        x["scorer"].set_lora(c["rank"], ALPHA, x["factors"])
    if c["depth"] > 1:
        x["scorer"].set_depth(c["depth"])
    if c["kind"] == "attention":
        x["out"] = torch.empty_like(x["q"])
    else:
        x["rewards"] = torch.zeros(c["n"], dtype=torch.float32, device="cuda")
    if c["kind"] == "grad":
        # pages that no candidate references keep what the buffer held
        x["grad"] = torch.zeros(x["pool"].shape, dtype=torch.float32, device="cuda")
    x["kind"] = c["kind"]
    return x


def run(state):
    x = state
    if x["kind"] == "score":
        x["scorer"].score_async(x["pool"], x["table"], x["lens"], x["rewards"])
        return x["rewards"]
    stream = torch.cuda.current_stream().cuda_stream
    if x["kind"] == "attention":
        kp.kvprm_attention(x["scorer"].ctx, x["pool"].data_ptr(), x["n_pages"], x["table"], x["lens"], len(x["lens"]),
                           x["q"].data_ptr(), x["k_self"].data_ptr(), x["v_self"].data_ptr(), x["out"].data_ptr(),
                           stream)
        return x["out"]
    p = kp.kvprm_score_grad(x["scorer"].ctx, x["pool"].data_ptr(), x["n_pages"], x["table"], x["lens"], len(x["lens"]),
                            x["grad"].data_ptr(), stream)
    return {"p_plus": p, "grad": x["grad"]}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    c = case
    s = _structure(c)
    rows = c["n"] * c["depth"]
    d, nq, nkv, hd, ff, layers, r = (c[k] for k in ("d", "nq", "nkv", "hd", "ff", "layers", "rank"))
    kv = layers * s.unique * 2 * nkv * PAGE * hd   # elements of the distinct pages
    tables = 4 * (s.used + c["n"])
    attn = 4 * layers * nq * hd * c["depth"] * sum(s.lens)   # q K and w V
    if c["kind"] == "attention":
        return {"bytes": 2 * kv + tables + 4 * c["n"] * hd * (2 * nq + 2 * nkv), "flops": attn}
    params = layers * ((nq + 2 * nkv) * hd * d + nq * hd * d + 3 * ff * d)
    if r:
        params += layers * r * ((nq + 2 * nkv) * hd + d + nq * hd + d + 2 * ff + d + ff + d)
    total = {"bytes": 2 * params + 2 * kv + tables + 4 * c["n"], "flops": 2 * params * rows + attn}
    if c["kind"] == "grad":   # the gradient out in fp32; a transposed product each, and dq, dK, dV, dP
        total["bytes"] += 4 * kv
        total["flops"] += 2 * params * rows + 2 * attn
    return total


def tolerance(case):
    """About four times what the path is off `exact`: activations carry ~17 bits (a bf16 pair) and sums
    are fp32; peaked softmax weights and the layers above amplify that.  Measured: attention 1.8e-6 and
    4.1e-6, the gradient 2.4e-5 .. 3.5e-5 (its sums over candidates come in no fixed order), P(+) 3e-7
    after 2 layers, 5e-6 .. 3.4e-5 after 28."""
    if case["kind"] == "attention":
        return {"rel": 2e-5}
    if case["kind"] == "grad":
        return {"rel": 1.5e-4}
    return {"rel": 4e-5 + 3e-6 * case["layers"]}


# ---------------------------------------------------------------- the same in 64 bits
def _rms64(h, g):
    return h * torch.rsqrt(h.pow(2).mean(-1, keepdim=True) + EPS) * g.double()


def _attend64(pool, table, lens, q, ks, vs):
    """q [n][k][nq][hd], ks / vs [n][k][nkv][hd] (verify tokens, causal among themselves), pool one layer
    [pages][2][nkv][16][hd]; returns [n][k][nq][hd]."""
    n, k, nq, hd = q.shape
    nkv = ks.shape[2]
    causal = torch.ones(k, k, dtype=torch.bool, device=q.device).tril()
    outs = []
    for b in range(n):
        L = int(lens[b])
        ids = torch.as_tensor(table[b, :(L + PAGE - 1) // PAGE].astype(np.int64), device=q.device)
        kv = pool[ids].double().permute(1, 2, 0, 3, 4).reshape(2, nkv, -1, hd)[:, :, :L]
        qb = q[b].reshape(k, nkv, nq // nkv, hd).permute(1, 2, 0, 3)          # [nkv][G][k][hd]
        kk = torch.cat([kv[0], ks[b].transpose(0, 1)], 1)                     # [nkv][L + k][hd]
        vv = torch.cat([kv[1], vs[b].transpose(0, 1)], 1)
        sc = torch.matmul(qb, kk.unsqueeze(1).transpose(-1, -2)) / math.sqrt(hd)
        keep = torch.cat([causal.new_ones(k, L), causal], 1)
        w = torch.softmax(sc.masked_fill(~keep, float("-inf")), -1)
        outs.append(torch.matmul(w, vv.unsqueeze(1)).permute(2, 0, 1, 3).reshape(k, nq, hd))
    return torch.stack(outs)


def _p_plus64(c, x, pools):
    n, k, nq, nkv, hd, ff = (c[key] for key in ("n", "depth", "nq", "nkv", "hd", "ff"))
    W = x["weights"]
    dev = W["embed_verify"].device
    pos = torch.as_tensor(x["lens"].astype(np.float64), device=dev)[:, None] + torch.arange(k, device=dev)
    ang = pos[..., None, None] * BASE ** (-torch.arange(0, hd, 2, dtype=torch.float64, device=dev) / hd)
    cos, sin = ang.cos(), ang.sin()

    def rope(y):
        a, b = y[..., :hd // 2], y[..., hd // 2:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

    def linear(y, l, name):
        out = y @ W["layers"][l]["w_" + name].double().T
        if c["rank"]:
            f = x["factors"][l]
            out = out + (ALPHA / c["rank"]) * ((y @ f["a_" + name].double().T) @ f["b_" + name].double().T)
        return out

    h = W["embed_verify"].double().expand(n, k, -1)
    for l, w in enumerate(W["layers"]):
        y = linear(_rms64(h, w["attn_norm"]), l, "qkv").reshape(n, k, nq + 2 * nkv, hd)
        o = _attend64(pools[l], x["table"], x["lens"], rope(y[:, :, :nq]), rope(y[:, :, nq:nq + nkv]), y[:, :, nq + nkv:])
        h = h + linear(o.reshape(n, k, -1), l, "o")
        gu = linear(_rms64(h, w["mlp_norm"]), l, "gate_up")
        h = h + linear(torch.nn.functional.silu(gu[..., :ff]) * gu[..., ff:], l, "down")
    z = _rms64(h[:, -1], W["final_norm"]) @ (W["w_plus"].double() - W["w_minus"].double())
    return torch.sigmoid(z)


def exact(case, seed):
    c = case
    x = _inputs(c, seed)
    if c["kind"] == "attention":
        with torch.no_grad():
            return _attend64(x["pool"][0], x["table"], x["lens"], x["q"].double()[:, None],
                             x["k_self"].double()[:, None], x["v_self"].double()[:, None])[:, 0]
    if c["kind"] == "score":
        with torch.no_grad():
            return _p_plus64(c, x, x["pool"])
    pools = [x["pool"][l].double().requires_grad_() for l in range(c["layers"])]
    p = _p_plus64(c, x, pools)
    (-p.log().sum()).backward()
    grad = torch.stack([t.grad for t in pools])
    return {"p_plus": p.detach(), "grad": grad}
