"""What a user of this library has it do, as cases that can be timed and compared.

The library builds the draft tree of one speculative-decoding round from a
block drafter's logits (dart.Dart) and runs the attention layer that verifies
the tree (dart.TreeAttention).  Six kinds of case cover its constructions:

  tree   dart.Dart.build_tree: Algorithm 1 with pruning, over the full
         vocabulary (cand_k = 0) or over K candidates per position
  chain  dart.Dart.build_chain_ddtree: causal correction along one chain
  heap   dart.Dart.build_seq_heap: node-wise best-first search
  attn   dart.TreeAttention over [context ; tree] under the ancestor mask

Sizes are those of the workloads this repository benchmarks (workloads/,
bench.py), and odd ones of the same ranges.  Inputs have the distributions
of workloads/, drawn on the GPU.
"""
from __future__ import annotations

import heapq
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2608_13524_gb300 import dart

DEV = "cuda"
BETA = -0.2
EPS = 1e-6


def _tree(name, kind, wdtype, nseq, V, d, L, W, k, B, T, cand_k=0):
    c = dict(kind=kind, wdtype=wdtype, nseq=nseq, V=V, d=d, L=L, W=W, k=k, B=B, T=T, cand_k=cand_k)
    return dict(c, name=name) if name else c


def _attn(name, nseq, B, C, L, W, Hq=32, Hkv=8, fill=1.0):
    c = dict(kind="attn", nseq=nseq, B=B, C=C, L=L, W=W, Hq=Hq, Hkv=Hkv, fill=fill)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest rounds: a tiny fp32 head, where launches and latency are everything
        _tree("toy-f32", "tree", "f32", 1, 4096, 256, 4, 4, 4, 16, 0.0),
        # one user, greedy, a narrow tree
        _tree("qwen3-4b", "tree", "bf16", 1, 151936, 2560, 16, 8, 8, 64, 0.0),
        # one user, sampling: the default benchmark
        _tree("qwen3-8b", "tree", "bf16", 1, 151936, 4096, 16, 16, 16, 256, 1.0),
        # the wide end of the width / budget study
        _tree("sweep-W64-B1024", "tree", "bf16", 1, 151936, 2560, 16, 64, 64, 1024, 0.0),
        # serving: eight sequences share each weight stream
        _tree("batched", "tree", "bf16", 8, 151936, 4096, 16, 32, 32, 512, 1.0),
        # the paper's default scoring, K = 64 candidates per position, for one user ...
        _tree("qwen3-8b-k64", "tree", "bf16", 1, 151936, 4096, 16, 16, 16, 256, 1.0, 64),
        # ... and for eight
        _tree("batched-k64", "tree", "bf16", 8, 151936, 4096, 16, 32, 32, 512, 1.0, 64),
        # another vocabulary and hidden size, nothing a multiple of a tile
        _tree("ragged-3x11", "tree", "bf16", 3, 50021, 1088, 9, 11, 13, 77, 0.7),
        # the two constructions the paper compares with, at the narrow shape
        _tree("chain-ddtree-qwen3-4b", "chain", "bf16", 1, 151936, 2560, 16, 8, 8, 64, 0.0),
        _tree("seq-heap-qwen3-4b", "heap", "bf16", 1, 151936, 2560, 16, 8, 8, 64, 0.0),
        # verification of one user's small tree over a 2048-token context ...
        _attn("verify-qwen3-4b", 1, 64, 2048, 16, 8),
        # ... and of eight users' large ones
        _attn("verify-batched", 8, 512, 2048, 16, 32),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["f32", "full", "full", "full", "cand", "cand", "chain", "heap", "attn", "attn"])
    if kind == "attn":
        L, W = rng.randint(2, 16), _log(rng, 2, 64)
        B = min(1024, max(2, min(L * W, _log(rng, 16, 1024))))
        nseq = rng.randint(1, 8)
        C = _log(rng, 1, 4096) - 1
        Hq, Hkv = rng.choice([(32, 8), (32, 8), (16, 8), (8, 8), (32, 4), (16, 1)])
        return _attn(None, nseq, B, C, L, W, Hq, Hkv, rng.choice([1.0, 1.0, 0.8]))
    L = rng.randint(3, 16)
    T = rng.choice([0.0, 1.0, 0.7])
    if kind == "f32":
        V, d = _log(rng, 500, 20000), 64 * _log(rng, 1, 8)
        L, nseq, W = rng.randint(2, 8), rng.randint(1, 4), _log(rng, 2, 16)
        k = _log(rng, 2, 16)
        return _tree(None, "tree", "f32", nseq, V, d, L, W, k, _log(rng, 4, min(256, L * W)), T)
    V, d = _log(rng, 8000, 151936), 64 * _log(rng, 8, 64)
    if kind in ("chain", "heap"):
        d = min(d, 2560)
        B = _log(rng, 8, 64) if kind == "heap" else _log(rng, 16, 256)
        return _tree(None, kind, "bf16", rng.randint(1, 4), V, d, L, 8, 8, B, T)
    nseq = rng.choice([1, 1, 2, 3, 4, 8])
    W = _log(rng, 2, min(64, 256 // nseq))
    k = min(_log(rng, 4, 64), 64 if nseq * W <= 64 else 32)
    B = _log(rng, 8, min(1024, L * W)) if L * W > 8 else L * W
    K = 0 if kind == "full" else max(k, _log(rng, 32, 256))
    return _tree(None, "tree", "bf16", nseq, V, d, L, W, k, B, T, K)


# ------------------------------------------------------------------ inputs

def _normal(g, shape, std, dtype):
    """N(0, std^2) in fp32, rounded to dtype, a block of rows at a time."""
    out = torch.empty(shape, dtype=dtype, device=DEV)
    step = max(1, (1 << 26) // shape[-1])
    for r in range(0, shape[0], step):
        n = min(step, shape[0] - r)
        out[r:r + n] = torch.randn((n,) + tuple(shape[1:]), generator=g, device=DEV) * std
    return out


def _tree_inputs(c, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * (int(seed) + 1) + 17)
    dt = torch.bfloat16 if c["wdtype"] == "bf16" else torch.float32
    V, d, L, n = c["V"], c["d"], c["L"], c["nseq"]
    W_i = _normal(g, (d, 2 * d), (2.0 * d) ** -0.5, dt)
    W_o = _normal(g, (d, d), d ** -0.5, dt)
    E = _normal(g, (V, d), 0.02, dt)
    h0 = torch.randn((n, d), generator=g, device=DEV)
    D = torch.randn((n, L, V), generator=g, device=DEV) * 3.0
    # the drafter's own pick stands out, less so along the block
    pick = torch.randint(0, V, (n, L, 1), generator=g, device=DEV)
    amp = torch.tensor([8.0 if dt == torch.float32 else 6.0 if i < 8 else 3.0 for i in range(L)], device=DEV)
    D.scatter_add_(2, pick, amp.view(1, L, 1).expand(n, L, 1).contiguous())
    return W_i, W_o, E, D, h0


def _config(c):
    variants = {"tree": 0, "chain": dart.DART_VARIANT_CHAIN_DDTREE, "heap": dart.DART_VARIANT_SEQ_HEAP}[c["kind"]]
    return SimpleNamespace(V=c["V"], d=c["d"], L=c["L"], W=c["W"], k=c["k"], B=c["B"], nseq=c["nseq"], beta=BETA,
                           temperature=c["T"], rms_eps=EPS, pos_offset=0, cand_k=c["cand_k"], variants=variants)


def _random_tree(B, L, W, n, g):
    """parents (-1: child of the root, -2: unused) and depths (0: unused) of
    an n-node tree of at most W nodes a level, in level order."""
    parents, depths = np.full(B, -2, np.int32), np.zeros(B, np.int32)
    prev, i, dep = [-1], 0, 1
    while i < n:
        cnt = n - i if dep == L else min(W, n - i)
        for p in np.sort(g.integers(0, len(prev), size=cnt)):
            parents[i], depths[i] = prev[p], dep
            i += 1
        prev, dep = list(range(i - cnt, i)), dep + 1
    return parents, depths


def _visible(c, seed):
    """[nseq][B][B] ancestor-or-self relation, depths [nseq][B], n_nodes."""
    g = np.random.default_rng([int(seed), 7])
    vis = np.zeros((c["nseq"], c["B"], c["B"]), bool)
    depths, n_nodes = np.zeros((c["nseq"], c["B"]), np.int32), np.zeros(c["nseq"], np.int32)
    for s in range(c["nseq"]):
        n = max(1, int(round(c["fill"] * c["B"])) - (s % 3 if c["fill"] < 1.0 else 0))
        parents, depths[s] = _random_tree(c["B"], c["L"], c["W"], n, g)
        n_nodes[s] = n
        for i in range(n):
            if parents[i] >= 0:
                vis[s, i] = vis[s, parents[i]]
            vis[s, i, i] = True
    return vis, depths, n_nodes


def _attn_inputs(c, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * (int(seed) + 1) + 29)
    n, B, C, dh = c["nseq"], c["B"], c["C"], 128

    def r(length, heads):
        return torch.randn((n, length, heads, dh), generator=g, device=DEV).to(torch.bfloat16)

    return r(B, c["Hq"]), r(B, c["Hkv"]), r(B, c["Hkv"]), r(C, c["Hkv"]), r(C, c["Hkv"])


def prepare(case, seed):
    c = case
    if c["kind"] != "attn":
        W_i, W_o, E, D, h0 = _tree_inputs(c, seed)
        return SimpleNamespace(kind=c["kind"], eng=dart.Dart(_config(c), W_i, W_o, E), D=D, h0=h0)
    vis, depths, n_nodes = _visible(c, seed)
    nw = (c["B"] + 63) // 64
    bits = np.zeros((c["nseq"], c["B"], nw * 64), np.uint8)
    bits[:, :, :c["B"]] = vis
    mask = np.packbits(bits, axis=-1, bitorder="little").view(np.int64).reshape(c["nseq"], c["B"], nw)
    pos = np.where(depths > 0, c["C"] + depths, -1).astype(np.int32)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    return SimpleNamespace(kind="attn", att=dart.TreeAttention(c["nseq"], c["B"], c["C"], c["Hq"], c["Hkv"]),
                           args=_attn_inputs(c, seed) + (dev(pos), dev(mask), dev(n_nodes)))


def run(state):
    if state.kind == "attn":
        return state.att(*state.args)
    if state.kind == "chain":
        return state.eng.build_chain_ddtree(state.D, state.h0)
    if state.kind == "heap":
        return state.eng.build_seq_heap(state.D, state.h0)
    return state.eng.build_tree(state.D, state.h0)


def work(case):
    """Every depth needs the states that the depth before it chose, and E is
    far larger than what the chip can hold, so a pass over E (fp32 toy sizes
    aside) is needed at each of the L depths; the head's weights fit the L2
    and count once.  The node-wise search cannot do with less either: its
    prefixes reach depth L one after another."""
    c = case
    n, B, L = c["nseq"], c["B"], c["L"]
    if c["kind"] == "attn":
        C, Hq, Hkv, dh = c["C"], c["Hq"], c["Hkv"], 128
        # keys a node sees: the context and its root-to-node path (half the
        # depth range on average), for q.k and p.v
        rows = n * B * c["fill"]
        kv = 2 * 2 * n * (B + C) * Hkv * dh
        return {"bytes": kv + n * B * Hq * dh * (2 + 4) + n * B * (4 + 8 * ((B + 63) // 64)),
                "flops": 4.0 * dh * Hq * rows * (C + (L + 1) / 2)}
    V, d, bpe = c["V"], c["d"], 2 if c["wdtype"] == "bf16" else 4
    if c["kind"] == "tree":
        nodes, last = [], 1
        for _ in range(L):
            nodes.append(n * last)
            last = min(c["W"], last * c["k"])
    elif c["kind"] == "chain":
        nodes = [n] * L
    else:
        nodes = [n * B / L] * L  # B corrected prefixes in all
    scored = c["cand_k"] or V
    e_bytes = V * d * bpe if scored == V else n * scored * d * bpe
    passes = 1 if V * d * bpe < (100 << 20) and scored == V else L
    out = n * B * (5 * 4 + 8 * ((B + 63) // 64)) + 4 * n
    return {"bytes": passes * e_bytes + n * L * V * 4 + 3 * d * d * bpe + out,
            "flops": sum(2.0 * m * scored * d for m in nodes) + sum(2.0 * m * 3 * d * d for m in nodes[1:])}


# ------------------------------------------------------------- 64 bits

def _advance(W_i, W_o, E, hp, tok):
    """RMSNorm(h_p + W_o . SiLU(W_i . [h_p ; E[t]])) for rows of hp."""
    u = torch.cat([hp, E[tok].double()], 1) @ W_i.T
    r = hp + torch.nn.functional.silu(u) @ W_o.T
    return r * torch.rsqrt(r.square().mean(1, keepdim=True) + EPS)


def _logq(E, H, rows, T):
    """log q~ over the vocabulary of the rows of H."""
    z = (rows.double() + H @ E.T) / (T if T > 0 else 1.0)
    return (z - torch.logsumexp(z, 1, keepdim=True)).clamp(max=0.0)


def _exact_tree(c, W_i, W_o, E, D, h0):
    n, L, W, k, B, T, K = (c[x] for x in ("nseq", "L", "W", "k", "B", "T", "cand_k"))
    E64 = None if K else E.double()
    H, score = h0.double()[:, None], torch.zeros((n, 1), dtype=torch.float64, device=DEV)
    levels = []
    for dep in range(L):
        P = H.shape[1]
        if K:
            cand = torch.topk(D[:, dep], K, dim=1).indices
            lq = torch.stack([_logq(E[cand[s]].double(), H[s], D[s, dep, cand[s]][None], T) for s in range(n)])
        else:
            lq = _logq(E64, H.reshape(n * P, -1), D[:, dep].repeat_interleave(P, 0), T).view(n, P, -1)
        best, tok = torch.topk(lq, k, dim=2)
        del lq
        if K:
            tok = torch.gather(cand[:, None].expand(n, P, K), 2, tok)
        sc = (score[:, :, None] + best + BETA).view(n, P * k)
        score, at = torch.topk(sc, min(W, P * k), dim=1)
        levels.append(score)
        if dep + 1 < L:
            par, t = at // k, torch.gather(tok.view(n, P * k), 1, at)
            hp = torch.gather(H, 1, par[:, :, None].expand(-1, -1, H.shape[2]))
            H = _advance(W_i, W_o, E, hp.reshape(-1, H.shape[2]), t.reshape(-1)).view(n, -1, H.shape[2])
    allsc = torch.cat(levels, 1)
    out = torch.full((n, B), -math.inf, dtype=torch.float64, device=DEV)
    keep = min(B, allsc.shape[1])
    ids = torch.topk(allsc, keep, dim=1).indices.sort(1).values
    out[:, :keep] = torch.gather(allsc, 1, ids)
    return out


def _exact_chain(c, W_i, W_o, E, D, h0):
    n, L, B, T = (c[x] for x in ("nseq", "L", "B", "T"))
    E64, h, lists = E.double(), h0.double(), []
    for dep in range(L):
        best, tok = torch.topk(_logq(E64, h, D[:, dep], T), min(B, c["V"]), dim=1)
        lists.append(best.cpu().numpy())
        if dep + 1 < L:
            h = _advance(W_i, W_o, E, h, tok[:, 0])
    out = np.full((n, B), -np.inf)
    for s in range(n):
        heap, seq = [(-(lists[0][s][0] + BETA), 0, 0, 0, 0.0)], 0  # (-score, order, depth, rank, parent's score)
        for i in range(B):
            if not heap:
                break
            neg, _, dep, rank, base = heapq.heappop(heap)
            out[s, i] = -neg
            if rank + 1 < lists[dep].shape[1]:
                seq += 1
                heapq.heappush(heap, (-(base + lists[dep][s][rank + 1] + BETA), seq, dep, rank + 1, base))
            if dep + 1 < L:
                seq += 1
                heapq.heappush(heap, (-(-neg + lists[dep + 1][s][0] + BETA), seq, dep + 1, 0, -neg))
    return torch.from_numpy(out)


def _exact_heap(c, W_i, W_o, E, D, h0):
    n, L, B, T = (c[x] for x in ("nseq", "L", "B", "T"))
    E64, out = E.double(), np.full((n, B), -np.inf)
    for s in range(n):
        def children(h, dep):
            best, tok = torch.topk(_logq(E64, h, D[s, dep][None], T)[0], min(B, c["V"]))
            return best.cpu().numpy(), tok.cpu().numpy()

        h = h0[s:s + 1].double()
        lists, seq = children(h, 0), 0
        heap = [(-(lists[0][0] + BETA), 0, 0, 0, 0.0, h, lists)]
        for i in range(B):
            if not heap:
                break
            neg, _, dep, rank, base, hp, lists = heapq.heappop(heap)
            out[s, i] = -neg
            if rank + 1 < len(lists[0]):
                seq += 1
                heapq.heappush(heap, (-(base + lists[0][rank + 1] + BETA), seq, dep, rank + 1, base, hp, lists))
            if dep + 1 < L and i + 1 < B:
                h = _advance(W_i, W_o, E, hp, torch.tensor([int(lists[1][rank])], device=DEV))
                new = children(h, dep + 1)
                seq += 1
                heapq.heappush(heap, (-(-neg + new[0][0] + BETA), seq, dep + 1, 0, -neg, h, new))
    return torch.from_numpy(out)


def _exact_attn(c, seed):
    q, kt, vt, kc, vc = _attn_inputs(c, seed)
    vis, depths, n_nodes = _visible(c, seed)
    n, B, C, Hq, Hkv, dh = c["nseq"], c["B"], c["C"], c["Hq"], c["Hkv"], 128
    freq = 1.0e6 ** (-2.0 * torch.arange(dh // 2, dtype=torch.float64, device=DEV) / dh)
    out = torch.zeros((n, B, Hq, dh), dtype=torch.float64, device=DEV)
    for s in range(n):
        m = int(n_nodes[s])
        pos = torch.from_numpy(depths[s, :m]).to(DEV).double() + C
        cos, sin = torch.cos(pos[:, None] * freq)[:, None], torch.sin(pos[:, None] * freq)[:, None]

        def rope(x):
            a, b = x[..., :dh // 2], x[..., dh // 2:]
            return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

        seen = torch.cat([torch.ones((m, C), dtype=torch.bool, device=DEV),
                          torch.from_numpy(vis[s, :m, :m]).to(DEV)], 1)
        Q, KT = rope(q[s, :m].double()), rope(kt[s, :m].double())
        for g in range(Hkv):
            heads = slice(g * (Hq // Hkv), (g + 1) * (Hq // Hkv))
            keys = torch.cat([kc[s, :, g].double(), KT[:, g]])
            vals = torch.cat([vc[s, :, g].double(), vt[s, :m, g].double()])
            x = torch.einsum("ihd,jd->ihj", Q[:, heads], keys) * dh ** -0.5
            out[s, :m, heads] = torch.softmax(x.masked_fill(~seen[:, None], -math.inf), -1) @ vals
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "attn":
        return _exact_attn(c, seed)
    W_i, W_o, E, D, h0 = _tree_inputs(c, seed)
    build = {"tree": _exact_tree, "chain": _exact_chain, "heap": _exact_heap}[c["kind"]]
    scores = build(c, W_i.double(), W_o.double(), E, D, h0)
    # the other arrays of the tree are whole numbers
    return dict(tokens=None, parents=None, depths=None, pos_ids=None, scores=scores, n_nodes=None, mask=None)
