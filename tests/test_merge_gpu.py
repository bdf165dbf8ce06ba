"""The merge + frontier kernel alone, on logits known exactly: with E = 0 a
node's scaled logits are its drafter row, so its k best children, and from
the kernel's own log q~ the frontier, follow from numpy sorts bit for bit."""
import numpy as np
import pytest
import torch

from workloads import Config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dart():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13524_gb300 import dart as d
    d.lib()
    return d


def rows(pattern, nseq, L, V, g):
    x = g.standard_normal((nseq, L, V), dtype=np.float32) * np.float32(3.0)
    if pattern == "ties":       # few distinct values: ties by token, parent and rank
        x = np.round(x)
    elif pattern == "dense":    # the best logits fill some vocabulary ranges: more survivors than are ranked
        x[:, :, :30 * 128] += np.float32(40.0)
    elif pattern == "sparse":   # fewer finite children than k
        x[:, :, 5:] = -np.inf
    return x


# (nseq, V, W, k, cand_k, pattern): one node, k at and past the group threshold's limit and off the
# 32-byte lists, 16 / 17 / 33 / 64 parents, more than 256 ranges, candidate lists, the radix fallback
CASES = [(1, 1000, 1, 1, 0, "normal"), (2, 40000, 16, 16, 0, "ties"), (1, 40000, 17, 17, 0, "normal"),
         (3, 20000, 11, 13, 0, "normal"), (1, 20000, 33, 33, 0, "ties"), (1, 19456, 64, 64, 0, "dense"),
         (2, 19456, 64, 64, 0, "normal"), (1, 40000, 8, 64, 0, "dense"), (1, 700, 4, 8, 0, "sparse"),
         (2, 3000, 32, 20, 600, "normal"), (1, 5000, 16, 16, 64, "ties"), (4, 2000, 64, 5, 37, "normal")]


@pytest.mark.parametrize("nseq,V,W,k,cand_k,pattern", CASES)
def test_merge_select(dart, nseq, V, W, k, cand_k, pattern):
    L, d, beta = 3, 64, np.float32(-0.2)
    cfg = Config("merge", nseq, V, d, L, W, k, 8, "bf16", 0.0, 1, beta=float(beta), cand_k=cand_k)
    g = np.random.Generator(np.random.PCG64([V, W, k, cand_k]))
    D = rows(pattern, nseq, L, V, g)
    z = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    Dt = torch.from_numpy(D).cuda()
    h0 = torch.from_numpy(g.standard_normal((nseq, d), dtype=np.float32)).cuda()
    eng = dart.Dart(cfg, z(d, 2 * d), z(d, d), z(V, d))
    try:
        prev = [[np.float32(0.0)] for _ in range(nseq)]
        for dep in range(1, L + 1):
            dart.dart_expand_depth(eng.h, dep, Dt, h0)
            tok, lq, lse = (t.cpu().numpy() for t in dart.dart_get_node_topk(eng.h, cfg))
            ft, fp, fs, fc = (t.cpu().numpy() for t in dart.dart_get_frontier(eng.h, dep, cfg))
            assert dart.dart_status_sync(eng.h) == 0
            P = tok.shape[0] // nseq
            for s in range(nseq):
                row = D[s, dep - 1]
                pool = np.sort(np.lexsort((np.arange(V), -row))[:cand_k]) if cand_k else np.arange(V)
                order = pool[np.lexsort((pool, -row[pool]))][:k]
                fin = row[pool][np.isfinite(row[pool])].astype(np.float64)
                want = np.log(np.sum(np.exp(fin - fin.max()))) + fin.max()
                keys = []
                for p in range(len(prev[s])):
                    n = s * P + p
                    nf = np.isfinite(row[order])
                    np.testing.assert_array_equal(tok[n][nf], order[nf])
                    assert abs(lse[n] - want) < 1e-5 * max(1.0, abs(want))
                    np.testing.assert_array_equal(lq[n][nf], np.minimum(row[order][nf] - lse[n], np.float32(0.0)))
                    assert np.all(lq[n][~nf] == -np.inf)
                    for j in range(k):
                        sc = (prev[s][p] + lq[n, j]) + beta
                        if sc > -np.inf:
                            keys.append((-sc, p, j, tok[n, j]))
                keys.sort()
                top = keys[:W]
                assert fc[s] == len(top)
                np.testing.assert_array_equal(fs[s, :len(top)], np.array([-t[0] for t in top], np.float32))
                np.testing.assert_array_equal(ft[s, :len(top)], [t[3] for t in top])
                np.testing.assert_array_equal(fp[s, :len(top)], [-1 if dep == 1 else t[1] for t in top])
                assert np.all(ft[s, len(top):] == -1) and np.all(fs[s, len(top):] == -np.inf)
                prev[s] = [-t[0] for t in top]
    finally:
        eng.close()


# fewer vocabulary ranges than k: one, k - 1, an odd number of keys in all, more than are read at
# once (63 lists of 64), ties, keys that are few or dense enough for the radix fallback, k <= 16
FEW = [(1, 100, 8, 64, 0, "normal"), (2, 63 * 128, 8, 64, 0, "normal"), (1, 48 * 128, 64, 49, 0, "ties"),
       (1, 33 * 128 - 5, 17, 63, 0, "normal"), (3, 20 * 128, 3, 57, 0, "normal"), (1, 40 * 128, 16, 61, 0, "dense"),
       (1, 12 * 128, 4, 40, 0, "sparse"), (2, 5 * 128 + 1, 9, 9, 0, "ties")]


@pytest.mark.parametrize("nseq,V,W,k,cand_k,pattern", FEW)
def test_merge_select_fewer_lists_than_k(dart, nseq, V, W, k, cand_k, pattern):
    test_merge_select(dart, nseq, V, W, k, cand_k, pattern)


def test_few_lists_cost_no_more_than_many(dart):
    """Fewer lists than k hold fewer keys than many do: merging them takes no
    longer (a thread that walks its list waits for a round trip per four keys:
    four times as long at 20 lists of 57)."""
    us = {}
    for V in (20 * 128, 150 * 128):
        cfg = Config("few", 2, V, 64, 4, 3, 57, 8, "bf16", 0.0, 1)
        g = np.random.Generator(np.random.PCG64(V))
        t = lambda a, dt: torch.from_numpy(a.astype(np.float32)).to(dt).cuda()  # noqa: E731
        eng = dart.Dart(cfg, t(g.standard_normal((64, 128)) * 0.1, torch.bfloat16),
                        t(g.standard_normal((64, 64)) * 0.1, torch.bfloat16),
                        t(g.standard_normal((V, 64)) * 0.02, torch.bfloat16))
        D, h0 = t(g.standard_normal((2, 4, V)) * 3, torch.float32), t(g.standard_normal((2, 64)), torch.float32)
        try:
            dart.dart_set_profiling(eng.h, True)
            eng.build_tree(D, h0)
            dart.dart_profile_read_kinds(eng.h)
            for _ in range(5):
                eng.build_tree(D, h0)
            ms, n = dart.dart_profile_read_kinds(eng.h)["merge_select"]
            assert dart.dart_status_sync(eng.h) == 0
        finally:
            eng.close()
        us[V] = ms / n * 1e3
    print(us)
    assert us[20 * 128] < 1.5 * us[150 * 128], us
