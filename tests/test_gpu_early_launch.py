"""Searches whose kernels are launched early, back to back and replayed from a graph, against waited ones."""
import numpy as np
import pytest
import torch

import paper_2206_12205_gb300 as fd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fd.build.build()
    torch.cuda.set_device(0)


def _searches(precision, n, **kw):
    zmax, m = (20, 64) if "direct" in precision else (84, 256)
    cfg = fd.make_config(n, zmax, m, 4096 if precision != "fp32" else 2048, max_harm=16, thr=(14, 20, 30, 44, 70),
                         max_peaks=1 << 14, precision=precision, **kw)
    return fd.Search(cfg, device="cuda")


# 2^19 and below are launched early on 152 SMs, 2^20 is not
@pytest.mark.parametrize("n", [1 << 14, 1 << 17, 1 << 19, 1 << 20])
@pytest.mark.parametrize("precision,kw", [("fp32", {}), ("bf16", {}), ("fp16_scaled", {}), ("bf16_direct", {}),
                                          ("bf16", {"norm_block": 4096}), ("bf16", {"harm_mode": 1}),
                                          ("fp32", {"harm_mode": 1})])
def test_early_launches_change_nothing(precision, kw, n):
    s, ref = _searches(precision, n, **kw), _searches(precision, n, **kw)
    rng = np.random.default_rng(n + len(precision))
    xs = [torch.from_numpy(rng.standard_normal(n).astype(np.float32)).cuda() for _ in range(3)]
    want = []
    for x in xs:                                     # each search waited for, its list by the plainly launched fdas_peaks
        ref.search(x)
        torch.cuda.synchronize()
        plane = ref.plane.clone()
        ref.find_peaks()
        torch.cuda.synchronize()
        want.append((plane, ref.peak_list().copy()))
    x = xs[0].clone()
    for _ in range(4):                               # back to back, no synchronisation between the searches
        for k in (1, 2, 0):
            x.copy_(xs[k])
            s.search(x)
    torch.cuda.synchronize()
    assert torch.equal(s.plane.view(torch.uint8), want[0][0].view(torch.uint8))
    assert np.array_equal(s.peak_list(), want[0][1]) and len(want[0][1]) > 0
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        s.search(x, torch.cuda.current_stream())
    for k in (1, 2, 0, 2, 1):
        x.copy_(xs[k])
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(s.plane.view(torch.uint8), want[1][0].view(torch.uint8))
    assert np.array_equal(s.peak_list(), want[1][1])
