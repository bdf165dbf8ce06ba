"""Row top-K over several slices (a block each, merged by the row's last block) against the oracle:
rows that are not 16-byte aligned, more keys at the bound than are ranked at
once (equal values, large K), rows of almost one value (radix select), infinities,
and the by-value lists of the best-first constructions."""
import numpy as np
import pytest
import torch

import oracle
from parity import (compare_pop_order_tree, compare_with_oracle, corrected_path_score, gpu_supertree, to_device, tol_of,
                    tree_to_numpy)
from workloads import Config, make_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dart():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13524_gb300 import dart as d
    d.lib()
    return d


# (nseq, V, K, what the drafter rows are made to hold)
CASES = [(1, 20001, 64, "plain"), (3, 8192, 300, "plain"), (1, 33000, 1000, "steps"), (2, 16385, 37, "one"),
         (1, 40960, 64, "inf"), (1, 12288, 1024, "one")]


@pytest.mark.parametrize("nseq,V,K,kind", CASES)
def test_candidate_slices(dart, nseq, V, K, kind):
    cfg = Config("topk", nseq, V, 64, 3, 6, 6, 20, "bf16", 0.0, 91, cand_k=K)
    x = make_inputs(cfg)
    D = x["Dlog"]
    if kind == "steps":
        np.round(D, out=D)
    elif kind == "one":
        D[D < 8.0] = 0.0
        D[:, 1, ::2] = -0.0
    elif kind == "inf":
        D[:, 0, 100:] = -np.inf
        D[:, 1, V // 2:] = -np.inf
    dx = to_device(cfg, x)
    ref = oracle.build_tree(cfg, x["Wi"], x["Wo"], x["E"], D, x["h0"])
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        g = tree_to_numpy(eng.build_tree(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
        gst = gpu_supertree(dart, eng.h, cfg)
    finally:
        eng.close()
    compare_with_oracle(cfg, ref, gst, g, tol_of(cfg), x=x)


@pytest.mark.parametrize("nseq,V,B", [(1, 20001, 300), (2, 32768, 130)])
def test_by_value_slices(dart, nseq, V, B):
    cfg = Config("topk-value", nseq, V, 64, 4, 4, 4, B, "bf16", 1.0, 92, variants=dart.DART_VARIANT_SEQ_HEAP)
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        g = tree_to_numpy(eng.build_seq_heap(dx["Dlog"], dx["h0"]))
        assert dart.dart_status_sync(eng.h) == 0
    finally:
        eng.close()
    ref = oracle.seq_heap(cfg, x["Wi"], x["Wo"], x["E"], x["Dlog"], x["h0"])
    compare_pop_order_tree(cfg, ref, g, tol_of(cfg), corrected_path_score(cfg, x))
