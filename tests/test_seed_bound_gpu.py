"""The starting bound of the LM-head's top-k filters where a block of the seed
kernel scores more than eight nodes: with it on, the supertree and the tree are
bit-identical to those without it (equal shares, a last share and a last chunk
of fewer nodes, one share per sequence)."""
import numpy as np
import pytest
import torch

from parity import to_device
from test_parity_gpu import run_depthwise
from workloads import Config, make_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dart():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13524_gb300 import dart as d
    d.lib()
    return d


# (nseq, V, d, W, k)
CASES = [(8, 3000, 4096, 32, 32), (5, 2501, 4096, 27, 20), (6, 2000, 3072, 42, 30), (25, 1500, 2560, 10, 9)]


@pytest.mark.parametrize("nseq,V,d,W,k", CASES)
def test_shares_of_many_nodes(dart, nseq, V, d, W, k):
    cfg = Config("bound-share", nseq, V, d, 3, W, k, 60, "bf16", 0.8, 83)
    dx = to_device(cfg, make_inputs(cfg))
    _, st_on, on = run_depthwise(dart, cfg.replace(topk_bound=1), dx)
    _, st_off, off = run_depthwise(dart, cfg.replace(topk_bound=2), dx)
    for a, b in ((on, off), (st_on, st_off)):
        for key in a:
            np.testing.assert_array_equal(a[key], b[key], err_msg=key)
