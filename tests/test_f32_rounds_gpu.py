"""The fp32 rounds of separate launches: a round takes no longer than its
kernels one after another.  Its LM-head and head GEMMs have about one block per
SM; placed while other kernels' waiting blocks held some SMs they shared the
rest, and a round took twice its kernels' time."""
import pytest
import torch

from parity import to_device
from workloads import Config, make_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dart():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13524_gb300 import dart as d
    d.lib()
    return d


# candidate sets and large head GEMMs; the full vocabulary and many small head updates
CASES = [Config("f32-cand", 4, 4000, 2048, 4, 39, 18, 60, "f32", 0.0, 95, cand_k=20),
         Config("f32-full", 16, 30000, 768, 4, 5, 4, 20, "f32", 0.0, 96),
         Config("f32-small-head", 5, 20502, 1024, 4, 2, 2, 8, "f32", 0.0, 97, cand_k=204)]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_round_is_no_longer_than_its_kernels(dart, cfg):
    x = make_inputs(cfg)
    dx = to_device(cfg, x)
    eng = dart.Dart(cfg, dx["Wi"], dx["Wo"], dx["E"])
    try:
        dart.dart_set_profiling(eng.h, True)
        eng.build_tree(dx["Dlog"], dx["h0"])
        dart.dart_profile_read_kinds(eng.h)
        for _ in range(5):
            eng.build_tree(dx["Dlog"], dx["h0"])
        kernels = sum(v[0] for v in dart.dart_profile_read_kinds(eng.h).values()) / 5
        dart.dart_set_profiling(eng.h, False)
        for _ in range(3):
            eng.build_tree(dx["Dlog"], dx["h0"])
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            eng.build_tree(dx["Dlog"], dx["h0"])
        b.record()
        torch.cuda.synchronize()
        assert dart.dart_status_sync(eng.h) == 0
    finally:
        eng.close()
    ms = a.elapsed_time(b) / 10
    print(cfg.name, ms, kernels)
    assert ms < 1.15 * kernels, (ms, kernels)
