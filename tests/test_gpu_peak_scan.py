"""The peak output's scan of all units: shares of a few units a block, and more than one round of 4096."""
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


def _level1(pl, thr):
    """(row, bin) of the 3x3 maxima above thr, in row-major order."""
    K, nb = pl.shape
    ok = pl > thr
    for di in (-1, 0, 1):
        for dr in (-1, 0, 1):
            if di == 0 and dr == 0:
                continue
            a = (slice(max(0, -di), K - max(0, di)), slice(max(0, -dr), nb - max(0, dr)))
            b = (slice(max(0, di), K - max(0, -di)), slice(max(0, dr), nb - max(0, -dr)))
            ok[a] &= pl[a] > pl[b] if (di, dr) < (0, 0) else pl[a] >= pl[b]
    return torch.nonzero(ok)


# units (rows x chunks of 512 bins): 33 x 128 = 4224, a few beyond the list; 5 x 1024 = 5120; 255 x 4096, two
# rounds a block on 152 SMs
@pytest.mark.parametrize("n,zmax,thr", [(1 << 17, 32, 6.0), (1 << 20, 4, 6.0), (1 << 22, 254, 18.0)])
def test_scan_shares(n, zmax, thr):
    K, nb = zmax + 1, n // 2
    g = torch.Generator(device="cuda").manual_seed(n + zmax)
    pl = torch.empty(K, nb, device="cuda").exponential_(0.5, generator=g).bfloat16()
    want = _level1(pl, thr).cpu().numpy()
    units = np.unique(want[:, 0] * (nb // 512) + want[:, 1] // 512).size
    assert units > 4096
    s = fd.Search(fd.make_config(n, zmax, 32, 1024, max_harm=1, thr=(thr,), max_peaks=len(want) + 5, precision="bf16"),
                  device="cuda")
    s.plane.copy_(pl.view(-1))
    s.find_peaks()
    torch.cuda.synchronize()
    got = s.peak_list()
    assert int(s.npeaks.item()) == len(want) == len(got)
    assert np.array_equal(got["zi"].astype(np.int64), want[:, 0]) and np.array_equal(got["r"].astype(np.int64), want[:, 1])
    vals = pl.view(-1)[torch.from_numpy(want[:, 0] * nb + want[:, 1]).cuda()].float().cpu().numpy()
    assert np.array_equal(got["power"].astype(np.float32), vals)
