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
