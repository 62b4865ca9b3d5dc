"""Level 1 after a marking plane kernel, with units of one to all 16 words of cells above the threshold (about 0,
3, 7 and 13 of them on noise): the same list as the unmarked pass over the plane, which tests whole units."""
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


@pytest.mark.parametrize("thr1", [20.0, 10.0, 8.0, 6.0])
@pytest.mark.parametrize("precision,anchored", [("fp32", 0), ("bf16", 0), ("bf16", 1), ("bf16_direct", 0)])
def test_marked_level1_by_words(precision, anchored, thr1):
    n, zmax = 1 << 16, 20
    s = fd.Search(fd.make_config(n, zmax, 64, 1024 if precision == "fp32" else 4096, max_harm=4, max_peaks=1 << 17,
                                 thr=(thr1, 1.6 * thr1, 2.6 * thr1), precision=precision, harm_mode=anchored), device="cuda")
    x = torch.from_numpy(np.random.default_rng(int(thr1)).standard_normal(n).astype(np.float32)).cuda()
    s.search(x)
    torch.cuda.synchronize()
    got = s.peak_list().copy()
    s.find_peaks()
    torch.cuda.synchronize()
    want = s.peak_list()
    assert (want["harm"] == 1).sum() > 5 and np.array_equal(got, want)
