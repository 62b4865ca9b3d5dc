"""The FP64 interpolated power of points whose window lies off the spectrum, far ones among them: taps
outside [0, Nb) count as zero, and the points beside them keep their values."""
import numpy as np
import pytest
import torch

import oracle
import paper_2206_12205_gb300 as fd
from paper_2206_12205_gb300 import fdas as ft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fd.build.build()
    oracle.build()
    torch.cuda.set_device(0)


def _power(plan, x, r, z):
    pts = torch.from_numpy(np.stack([r, z], 1)).cuda()
    out = torch.full((len(r), 3), 7.0, dtype=torch.float64, device="cuda")
    ft.fdas_interp_power(plan, x, pts, out, fp64=True)
    return out.cpu().numpy()


@pytest.mark.parametrize("m", [2, 64])
def test_points_off_the_spectrum(m):
    n = 1 << 14
    nb = n // 2
    X = np.random.default_rng(m).standard_normal(n).astype(np.float32)
    x = torch.from_numpy(X).cuda()
    plan = fd.fdas_plan(fd.make_config(n, 2, m, 1024))
    far = np.array([m, 2.0 ** 24, 2.0 ** 31, 2.0 ** 31 + 12, 3e9, 2.0 ** 32, 1e12 + 0.25, 4e15])
    r = np.concatenate([nb + far, -far])
    z = np.array([0.0, 0.3, -0.3, 0.999, -0.999, 1.0, -1.0, 40.0, -40.0])
    rr, zz = (a.ravel() for a in np.meshgrid(r, z, indexing="ij"))
    assert np.all(_power(plan, x, rr, zz) == 0.0)
    # the same among points on the spectrum, enough of them that a warp takes several in turn
    rr, zz = np.tile(rr, 30), np.tile(zz, 30)
    ron = np.random.default_rng(1).uniform(m, nb - m, len(rr))
    alone = _power(plan, x, ron, zz)
    mixed = _power(plan, x, np.stack([ron, rr], 1).ravel(), np.repeat(zz, 2))
    assert np.array_equal(mixed[0::2], alone) and np.all(mixed[1::2] == 0.0)
    c = X.view(np.complex64).astype(np.complex128)
    for i in range(0, 144, 7):
        P = oracle.interp_power(c, m, float(ron[i]), float(zz[i]), int(np.floor(ron[i] + 0.5)))[0]
        assert abs(alone[i, 0] - P) <= 1e-10 * max(P, 2.0)
