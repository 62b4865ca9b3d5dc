"""The 3x3 rule where it can go wrong: planes of small integers (ties everywhere: along a row, across rows,
over the edges of units and of the plane), with and without NaN and infinities, from a few cells above the
threshold in a unit to nearly all.  Bit for bit against the oracle."""
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


def _plane(kind, K, nb, seed):
    rng = np.random.default_rng(seed)
    share, top = {"few": (0.002, 4), "some": (0.1, 4), "most": (0.9, 8)}[kind.split("+")[0]]
    pl = np.where(rng.random((K, nb)) < share, rng.integers(1, top, (K, nb)), 0).astype(np.float32)
    edges = np.concatenate([np.arange(0, nb, 512), np.arange(511, nb, 512)])
    pl[:, edges] = rng.integers(1, top, (K, edges.size))        # both sides of every unit's edge
    if "+" in kind:
        for v in (np.nan, np.inf):
            pl[rng.integers(0, K, 200), rng.integers(0, nb, 200)] = v
            pl[rng.integers(0, K, 40), rng.choice(edges, 40)] = v
    return pl


@pytest.mark.parametrize("kind", ["few", "some", "most", "few+nonfinite", "most+nonfinite"])
@pytest.mark.parametrize("anchored", [0, 1])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("n,zmax", [(1 << 11, 2), (1 << 15, 34)])
def test_peaks_of_tied_cells(n, zmax, precision, anchored, kind):
    K, nb, max_out = zmax + 1, n // 2, 1 << 20
    pl = _plane(kind, K, nb, 31 * zmax + len(kind))              # every value is a BF16 number
    thr = (0.5, 0.5, 1.5, 2.5, 4.5) if kind.startswith("few") else (1.5, 3.5, 8.5, 18.5, 40.5)
    s = fd.Search(fd.make_config(n, zmax, 32, 1024, max_harm=16, thr=thr, max_peaks=max_out, harm_mode=anchored,
                                 precision=precision), device="cuda")
    s.plane.copy_(torch.from_numpy(pl.ravel()).to(s.plane.dtype))
    s.find_peaks()
    torch.cuda.synchronize()
    want, cnt = oracle.peaks_f32(pl, zmax, 16, thr, max_out=max_out, anchored=bool(anchored))
    got = s.peak_list()
    assert int(s.npeaks.item()) == cnt == len(got) > 0
    for a, b in (("harm", "h"), ("zi", "zi"), ("r", "r")):
        assert np.array_equal(got[a].astype(np.int64), want[b].astype(np.int64))
    assert np.array_equal(got["power"].view(np.uint32), want["power"].astype(np.float32).view(np.uint32))
