"""GPU parity of the best-first constructions the paper compares DARTree
with (Table 2) and of DARTree (fixed) (Sec. 5.1), through the C ABI, against
the fp64 oracle: Domino-chain + DDTree (dart_build_chain_ddtree) and
sequential correction with heap (dart_build_seq_heap)."""
import numpy as np
import pytest
import torch

import oracle
from parity import (chain_path_score, compare_pop_order_tree, compare_with_oracle, corrected_path_score,
                    gpu_supertree, to_device, tol_of, tree_to_numpy)
from workloads import Q4B, Q8B, Config, make_inputs

pytestmark = pytest.mark.gpu

BOTH = 3  # DART_VARIANT_CHAIN_DDTREE | DART_VARIANT_SEQ_HEAP


@pytest.fixture(scope="module")
def dart():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13524_gb300 import dart as d
    d.lib()
    return d


def C(name, nseq, V, d, L, B, wdtype="bf16", T=0.0, seed=1, **kw):
    return Config(name, nseq, V, d, L, 4, 4, B, wdtype, T, seed, variants=BOTH, **kw)


CASES = [
    C("heap-f32", 1, 1500, 128, 4, 12, "f32", 0.0, 61),
    C("heap-bf16", 2, 3000, 256, 5, 20, "bf16", 1.0, 62),
    C("heap-multitile", 1, 50000, 256, 4, 64, "bf16", 0.7, 63),
    C("heap-B1", 1, 800, 128, 3, 1, "bf16", 0.0, 64),
    C("heap-L1", 2, 900, 128, 1, 9, "bf16", 0.0, 65),
    C("heap-beta0", 1, 1200, 128, 4, 25, "bf16", 0.0, 66, beta=0.0),
    C("heap-B200", 3, 700, 64, 6, 200, "bf16", 0.0, 67, pos_offset=11),
    C("heap-V<B", 1, 40, 64, 3, 300, "bf16", 0.0, 68),
    C("heap-d4096", 1, 20000, 4096, 4, 30, "bf16", 1.0, 69),
]


def chain_check(dart, eng, cfg, ref, tol):
    tok, lse = dart.dart_get_chain(eng.h, cfg)
    tok, lse = tok.cpu().numpy(), lse.cpu().numpy()
    np.testing.assert_allclose(lse, ref["chain_lse"], rtol=0, atol=tol)
    if not np.array_equal(tok, ref["chain_tok"]):
        # allowed only where the oracle's chain has a near tie at its argmax
        s, i = [int(v[0]) for v in np.nonzero(tok != ref["chain_tok"])]
        raise AssertionError(f"chain differs at sequence {s}, depth {i + 1}")


@pytest.mark.parametrize("cfg", CASES, ids=[c.name for c in CASES])
def test_chain_ddtree_and_seq_heap_parity(dart, cfg):
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    tol = tol_of(cfg)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        g1 = tree_to_numpy(eng.build_chain_ddtree(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        ref = oracle.chain_ddtree(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
        chain_check(dart, eng, cfg, ref, tol)
        rep = compare_pop_order_tree(cfg, ref, g1, tol, chain_path_score(cfg, x, ref["chain_tok"]))
        print(cfg.name, "chain+DDTree", rep)
        g2 = tree_to_numpy(eng.build_seq_heap(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        ref2 = oracle.seq_heap(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
        rep2 = compare_pop_order_tree(cfg, ref2, g2, tol, corrected_path_score(cfg, x))
        print(cfg.name, "seq heap", rep2)
        # graph replays are deterministic, and the constructions do not disturb each other
        for build, want in ((eng.build_chain_ddtree, g1), (eng.build_seq_heap, g2)):
            again = tree_to_numpy(build(dx["Dlog"], dx["h0"]))
            for k in want:
                np.testing.assert_array_equal(again[k], want[k], err_msg=k)
        assert dart.dart_status_sync(eng.h) == 0
    finally:
        eng.close()


def test_variants_and_algorithm1_on_one_handle(dart):
    """DARTree rounds, the test hooks and the best-first constructions on one
    handle: each round gives the same tree as on its own, and the
    Algorithm 1 test hooks refuse to read after a best-first round."""
    cfg = C("heap-mixed", 2, 2000, 128, 4, 16, "bf16", 0.5, 70)
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        a = tree_to_numpy(eng.build_tree(dx["Dlog"], dx["h0"]))
        gst = gpu_supertree(dart, eng.h, cfg)
        b = tree_to_numpy(eng.build_chain_ddtree(dx["Dlog"], dx["h0"]))
        with pytest.raises(dart.DartError) as e:
            dart.dart_get_frontier(eng.h, 1, cfg)
        assert e.value.code == dart.DART_ERR_STATE
        c = tree_to_numpy(eng.build_seq_heap(dx["Dlog"], dx["h0"]))
        with pytest.raises(dart.DartError) as e:
            dart.dart_get_chain(eng.h, cfg)
        assert e.value.code == dart.DART_ERR_STATE
        a2 = tree_to_numpy(eng.build_tree(dx["Dlog"], dx["h0"]))
        b2 = tree_to_numpy(eng.build_chain_ddtree(dx["Dlog"], dx["h0"]))
        c2 = tree_to_numpy(eng.build_seq_heap(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        for u, v in ((a, a2), (b, b2), (c, c2)):
            for k in u:
                np.testing.assert_array_equal(u[k], v[k], err_msg=k)
    finally:
        eng.close()
    ref = oracle.build_tree(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
    compare_with_oracle(cfg, ref, gst, a, tol_of(cfg), x=x)


def test_variant_entry_points_need_their_workspace(dart):
    cfg = Config("heap-none", 1, 500, 64, 3, 2, 2, 4, "bf16", 0.0, 71)
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        for fn in (dart.dart_build_chain_ddtree, dart.dart_build_seq_heap):
            with pytest.raises(dart.DartError) as e:
                fn(eng.h, dx["Dlog"], dx["h0"], eng.out)
            assert e.value.code == dart.DART_ERR_STATE
    finally:
        eng.close()
    # restricted candidate sets and more than 64 sequences are not supported by the variants
    for bad in (cfg.replace(variants=1, cand_k=8), cfg.replace(variants=2, nseq=65, W=1)):
        with pytest.raises(dart.DartError) as e:
            dart.Dart(bad, dx["Wi"], dx["Wo"], dx["E"])
        assert e.value.code == dart.DART_ERR_UNSUPPORTED


def test_dartree_fixed(dart):
    """DARTree (fixed), Sec. 5.1: W = 4 nodes per depth over 16 depths, the
    64-node supertree is the verification tree (no pruning)."""
    cfg = Config("dartree-fixed", 2, 30000, 512, 16, 4, 4, 64, "bf16", 0.0, 72)
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        g = tree_to_numpy(eng.build_tree_fixed(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        gst = gpu_supertree(dart, eng.h, cfg)
        assert list(g["n_nodes"]) == [64, 64]
    finally:
        eng.close()
    ref = oracle.build_tree(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
    compare_with_oracle(cfg, ref, gst, g, tol_of(cfg), x=x)
    small = cfg.replace(B=63)
    eng = dart.Dart(small, dx["Wi"], dx["Wo"], dx["E"])
    try:
        with pytest.raises(dart.DartError) as e:
            eng.build_tree_fixed(dx["Dlog"], dx["h0"])
        assert e.value.code == dart.DART_ERR_INVALID
    finally:
        eng.close()


FULL = [Q8B.replace(name="qwen3-8b-heap", variants=BOTH), Q4B.replace(name="qwen3-4b-heap", variants=BOTH)]


@pytest.mark.parametrize("cfg", FULL, ids=[c.name for c in FULL])
def test_full_size_best_first_parity(dart, cfg):
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    tol = tol_of(cfg)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        g1 = tree_to_numpy(eng.build_chain_ddtree(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        ref = oracle.chain_ddtree(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
        chain_check(dart, eng, cfg, ref, tol)
        g2 = tree_to_numpy(eng.build_seq_heap(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
    finally:
        eng.close()
    del dx
    rep = compare_pop_order_tree(cfg, ref, g1, tol, chain_path_score(cfg, x, ref["chain_tok"]))
    print(cfg.name, "chain+DDTree", rep)
    ref2 = oracle.seq_heap(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
    rep2 = compare_pop_order_tree(cfg, ref2, g2, tol, corrected_path_score(cfg, x))
    print(cfg.name, "seq heap", rep2)


# targets per pass (16 / nseq with bf16 weights, 4 / nseq with fp32) and the
# sizes at which a pass or a list is cut: (nseq, V, L, B, wdtype)
PASSES = [(3, 900, 5, 33, "bf16"), (1, 70, 2, 2, "bf16"), (16, 300, 3, 18, "bf16"), (17, 300, 3, 9, "bf16"),
          (2, 800, 4, 31, "f32"), (1, 5000, 9, 130, "bf16"), (1, 6, 3, 40, "bf16")]


@pytest.mark.parametrize("nseq,V,L,B,wdtype", PASSES)
def test_seq_heap_passes(dart, nseq, V, L, B, wdtype):
    """The search that corrects several prefixes a pass pops what the oracle's
    one-prefix-at-a-time search pops, as a graph (conditional passes) and as
    the fixed launch sequence that a capturing caller gets."""
    cfg = Config("heap-pass", nseq, V, 128, L, 2, 2, B, wdtype, 0.8, 75, variants=2)
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        g = tree_to_numpy(eng.build_seq_heap(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        ref = oracle.seq_heap(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
        compare_pop_order_tree(cfg, ref, g, tol_of(cfg), corrected_path_score(cfg, x))
        cg = torch.cuda.CUDAGraph()
        with torch.cuda.graph(cg):
            out = eng.build_seq_heap(dx["Dlog"], dx["h0"])
        for t in out.values():
            t.zero_()
        cg.replay()
        torch.cuda.synchronize()
        for k, v in tree_to_numpy(out).items():
            np.testing.assert_array_equal(v, g[k], err_msg=k)
        assert dart.dart_status_sync(eng.h) == 0
    finally:
        eng.close()


def test_idle_passes_do_not_score(dart):
    """As a fixed launch sequence the fp32 search launches B - 1 passes, of
    which few have a prefix to correct: the others' LM-head streams no E.
    (Bound: with B = 2 both passes score; of the forty of B = 40 a search of
    depth 4 that corrects four prefixes a pass needs well under half.)"""
    per_launch = {}
    for B in (2, 40):
        cfg = Config("heap-idle", 1, 60000, 512, 4, 2, 2, B, "f32", 0.0, 76, variants=2)
        x = make_inputs(cfg)
        dx = to_device(cfg, x)
        eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
        try:
            g = tree_to_numpy(eng.build_seq_heap(dx["Dlog"], dx["h0"]))
            dart.dart_set_profiling(eng.h, True)
            eng.build_seq_heap(dx["Dlog"], dx["h0"])
            dart.dart_profile_read_kinds(eng.h)
            p = tree_to_numpy(eng.build_seq_heap(dx["Dlog"], dx["h0"]))
            ms, launches = dart.dart_profile_read_kinds(eng.h)["lmhead"]
            for k in g:
                np.testing.assert_array_equal(p[k], g[k], err_msg=k)
            assert dart.dart_status_sync(eng.h) == 0
        finally:
            eng.close()
        assert launches == B
        per_launch[B] = ms / launches
    assert per_launch[40] < 0.625 * per_launch[2], per_launch
