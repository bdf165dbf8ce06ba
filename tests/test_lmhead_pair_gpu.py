"""The LM-head's CTA pairs (more than 64 nodes per depth) against the oracle:
ranges of unequal length, an odd number of ranges (single CTAs), one and two
node groups, ragged vocabularies and the tiled copy of E."""
import pytest
import torch

import oracle
from parity import compare_with_oracle, gpu_supertree, to_device, tol_of, tree_to_numpy
from workloads import Config, make_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dart():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13524_gb300 import dart as d
    d.lib()
    return d


# (nseq, V, d, W, k, weights_tiled)
CASES = [(5, 128 * 31 + 5, 128, 13, 13, 0), (5, 128 * 15, 64, 13, 5, 0), (8, 40000, 64, 32, 9, 0),
         (2, 20001, 128, 64, 33, 0), (3, 9000, 192, 43, 20, 1), (2, 200, 64, 33, 40, 0)]


@pytest.mark.parametrize("nseq,V,d,W,k,tiled", CASES)
def test_lmhead_pairs(dart, nseq, V, d, W, k, tiled):
    cfg = Config("pair", nseq, V, d, 3, W, k, 60, "bf16", 0.9, 81, weights_tiled=tiled)
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    ref = oracle.build_tree(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        g = tree_to_numpy(eng.build_tree(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        gst = gpu_supertree(dart, eng.h, cfg)
    finally:
        eng.close()
    compare_with_oracle(cfg, ref, gst, g, tol_of(cfg), x=x)


# 32 candidate slots per node (no starting bound, ranges of one tile) and 16, pairs and single CTAs
SLOTS = [(8, 128 * 90, 64, 32, 40, 2), (8, 128 * 90, 64, 32, 40, 1), (3, 128 * 75, 128, 40, 64, 2),
         (5, 128 * 31 + 5, 128, 13, 13, 2), (16, 128 * 160, 64, 6, 34, 2), (16, 128 * 5 - 3, 64, 6, 34, 1)]


@pytest.mark.parametrize("nseq,V,d,W,k,bound", SLOTS)
def test_candidate_slots(dart, nseq, V, d, W, k, bound):
    cfg = Config("slots", nseq, V, d, 3, W, k, 60, "bf16", 0.0, 82, topk_bound=bound)
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    ref = oracle.build_tree(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        g = tree_to_numpy(eng.build_tree(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        gst = gpu_supertree(dart, eng.h, cfg)
    finally:
        eng.close()
    compare_with_oracle(cfg, ref, gst, g, tol_of(cfg), x=x)


def test_slots_without_a_bound(dart):
    """96 nodes without the starting bound: at 16 slots the merge rounds of the
    first tiles made a pass 2.0 times as long as one of 64 nodes (32 slots)."""
    us = {}
    for W in (4, 6):
        cfg = Config("slots-time", 16, 6000, 1024, 3, W, 34, 8, "bf16", 0.0, 83, topk_bound=2)
        x = make_inputs(cfg)
        dx = to_device(cfg, x)
        eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
        try:
            dart.dart_set_profiling(eng.h, True)
            eng.build_tree(dx["Dlog"], dx["h0"])
            dart.dart_profile_read_kinds(eng.h)
            for _ in range(5):
                eng.build_tree(dx["Dlog"], dx["h0"])
            ms, n = dart.dart_profile_read_kinds(eng.h)["lmhead"]
            assert dart.dart_status_sync(eng.h) == 0
        finally:
            eng.close()
        us[W] = ms / n * 1e3
    print(us)
    assert us[6] < 1.7 * us[4], us
