"""Candidate scoring alone, at the edges of its blocking, against fp64 dot
products of the states the GPU itself scored (dart_get_states)."""
import numpy as np
import pytest
import torch

from parity import to_device
from workloads import Config, bf16_bits_to_f32, make_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dart():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13524_gb300 import dart as d
    d.lib()
    return d


# (nseq, V, d, W, k, K, wdtype): several d-slices per block of the cluster, node states staged in
# parts, slices of a few columns, the tiles of 4 and of 2 candidates, ragged groups, fp32
CASES = [(1, 64, 4096, 2, 2, 8, "bf16"), (1, 300, 4160, 64, 64, 70, "bf16"), (3, 2000, 64, 11, 5, 9, "bf16"),
         (2, 500, 256, 32, 16, 33, "f32"), (1, 500, 192, 9, 4, 17, "f32"), (8, 900, 512, 9, 9, 64, "bf16"),
         (7, 900, 1088, 9, 9, 31, "bf16")]


@pytest.mark.parametrize("nseq,V,d,W,k,K,wdtype", CASES)
def test_cand_score(dart, nseq, V, d, W, k, K, wdtype):
    cfg = Config("cand-score", nseq, V, d, 3, W, k, 8, wdtype, 0.8, 91, cand_k=K)
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    E = (bf16_bits_to_f32(x["E"]) if wdtype == "bf16" else x["E"]).astype(np.float64)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        h, count = x["h0"].astype(np.float64)[:, None], [1] * nseq
        for dep in range(1, 4):
            dart.dart_expand_depth(eng.h, dep, dx["Dlog"], dx["h0"])
            tok, lq, lse = (t.cpu().numpy() for t in dart.dart_get_node_topk(eng.h, cfg))
            fc = dart.dart_get_frontier(eng.h, dep, cfg)[3].cpu().numpy()
            assert dart.dart_status_sync(eng.h) == 0
            P = tok.shape[0] // nseq
            for s in range(nseq):
                row = x["Dlog"][s, dep - 1]
                c = np.sort(np.lexsort((np.arange(V), -row))[:K])
                for p in range(count[s]):
                    n = s * P + p
                    z = (row[c].astype(np.float64) + E[c] @ h[s, p]) / 0.8
                    # rounding of a sum of d products in fp32, of the addition and of the division by T
                    tol = 2.0 ** -24 * ((d + 4) * np.max(np.abs(E[c]) @ np.abs(h[s, p])) + 8 * np.max(np.abs(z))) / 0.8
                    want = np.log(np.sum(np.exp(z - z.max()))) + z.max()
                    assert abs(lse[n] - want) < tol + 1e-5
                    got = np.searchsorted(c, tok[n])
                    np.testing.assert_array_equal(c[got], tok[n])
                    assert np.max(np.abs(lq[n] - np.minimum(z[got] - want, 0.0))) < 2 * tol + 2e-5
                    assert len(set(tok[n])) == k and z[got].min() >= np.sort(z)[-k] - 2 * tol
            if dep < 3:
                st = dart.dart_get_states(eng.h, cfg).cpu().numpy().astype(np.float64)
                h, count = st.reshape(nseq, -1, d), [int(v) for v in fc]
    finally:
        eng.close()
