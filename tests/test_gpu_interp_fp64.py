"""The FP64 interpolated power where its forms meet (|z| at 0 and 1, far and near taps, windows off the
spectrum, rejected points), against the FP64 oracle with the parity test's tolerances."""
import numpy as np
import pytest
import torch

import fdas_synth as synth
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


def _case(n, zmax, seed):
    x = (synth.noise(n, synth.rng_for(80, seed)) + synth.chirp(n, 0.25, n / 13.3, zmax * 0.6)).astype(np.float32)
    xr, _ = oracle.spectrum(x)
    c64 = np.ascontiguousarray(xr.astype(np.complex64))
    return torch.from_numpy(c64.view(np.float32)).cuda(), c64.astype(np.complex128)


@pytest.mark.parametrize("m", [2, 34, 250])
def test_interp_fp64_forms(m):
    n = 1 << 14
    xdev, xin = _case(n, 20, m)
    nb = n // 2
    plan = fd.fdas_plan(fd.make_config(n, 2, m, 2048))
    rng = np.random.default_rng(5 + m)
    z = np.concatenate([[0.0, -0.0, 1e-9, 0.999999, -0.999999, 1.0, -1.0, 1.000001, 84.0, -84.0, 300.0, -300.0],
                        rng.uniform(-1, 1, 4), rng.uniform(-90, 90, 8)])
    r = np.concatenate([rng.uniform(m, nb - m, z.size - 8),
                        [0.0, 0.49, -3.25, nb - 1.0, nb + 2.5, 1000.0, 1000.5, 1234.25]])
    for shift in (0, 7, -90):
        k0 = np.floor(r + 0.5).astype(np.int64) + shift
        pts = torch.from_numpy(np.stack([r, z], 1)).cuda()
        out = torch.empty(z.size, 3, dtype=torch.float64, device="cuda")
        ft.fdas_interp_power(plan, xdev, pts, out, k0=torch.from_numpy(k0).cuda(), fp64=True)
        got = out.cpu().numpy()
        for i in range(z.size):
            P, gr, gz = oracle.interp_power(xin, m, float(r[i]), float(z[i]), int(k0[i]))
            sc = max(P, 2.0)
            assert abs(got[i, 0] - P) <= 1e-10 * sc
            assert abs(got[i, 1] - gr) <= 1e-9 * (sc + abs(gr)) and abs(got[i, 2] - gz) <= 1e-9 * (sc + abs(gz))


def test_interp_fp64_marks_bad_points_and_keeps_infinities():
    n, m = 1 << 12, 32
    plan = fd.fdas_plan(fd.make_config(n, 2, m, 1024))
    x = torch.zeros(n, device="cuda")
    x[2 * 500] = float("inf")
    pts = torch.tensor([[100.0, 2.0], [float("nan"), 1.0], [50.0, 2.0 ** 20], [500.2, 3.0], [300.0, float("inf")]],
                       dtype=torch.float64, device="cuda")
    out = torch.zeros(5, 3, dtype=torch.float64, device="cuda")
    ft.fdas_interp_power(plan, x, pts, out, fp64=True)
    got = out.cpu().numpy()
    assert np.all(got[0] == 0.0)
    assert np.all(np.isnan(got[[1, 2, 4]]))
    assert not np.any(np.isfinite(got[3]))
