"""Peak lists on both sides of the unit list's capacity, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2206_12205_gb300 as fd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fd.build.build()
    oracle.build()
    torch.cuda.set_device(0)


# FP32: 197, 3282 (both listed) and 4149, 10965 non-empty units (every count
# scanned); at 1.0 most cells of a unit are above the threshold; capacity 4096
@pytest.mark.parametrize("thr1,listed", [(20.0, True), (14.0, True), (13.4, False), (8.0, False), (1.0, False)])
@pytest.mark.parametrize("anchored", [0, 1])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_peak_lists_around_the_capacity(thr1, listed, anchored, precision):
    n, zmax, max_out = 1 << 17, 64, 1 << 21
    K, nb = zmax + 1, n // 2
    rng = np.random.default_rng(9100 + int(10 * thr1))
    pl = rng.exponential(2.0, size=(K, nb)).astype(np.float32)
    if precision == "bf16":                          # the stored values themselves
        pl = torch.from_numpy(pl).bfloat16().float().numpy()
    thr = (thr1, thr1 * 1.6, thr1 * 2.6)
    s = fd.Search(fd.make_config(n, zmax, 64, 1024, max_harm=4, thr=thr, max_peaks=max_out, harm_mode=anchored,
                                 precision=precision), device="cuda")
    s.plane.copy_(torch.from_numpy(pl.ravel()).to(s.plane.dtype))
    s.find_peaks()
    torch.cuda.synchronize()
    want, cnt = oracle.peaks_f32(pl, zmax, 4, thr, max_out=max_out, anchored=bool(anchored))
    if not anchored:
        assert (len({(int(w["h"]), int(w["zi"]), int(w["r"]) // 512) for w in want}) <= 4096) == listed
    got = s.peak_list()
    assert int(s.npeaks.item()) == cnt == len(got)
    for a, b in (("harm", "h"), ("zi", "zi"), ("r", "r")):
        assert np.array_equal(got[a].astype(np.int64), want[b].astype(np.int64))
    assert np.array_equal(got["power"].view(np.uint32), want["power"].astype(np.float32).view(np.uint32))
