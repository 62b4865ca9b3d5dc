"""The split plane at segment, row and item remainders, against the FP64 oracle with the parity test's
bound."""
import numpy as np
import pytest
import torch

import fdas_synth as synth
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


def _case(n, zmax, seed):
    x = (synth.noise(n, synth.rng_for(80, seed)) + synth.chirp(n, 0.25, n / 13.3, zmax * 0.6)).astype(np.float32)
    xr, _ = oracle.spectrum(x)
    c64 = np.ascontiguousarray(xr.astype(np.complex64))
    return torch.from_numpy(c64.view(np.float32)).cuda(), c64.astype(np.complex128)


# one segment only, a ragged last segment, more and fewer items than SMs
@pytest.mark.parametrize("n,zmax,m", [(1 << 11, 0, 8), (1 << 13, 2, 2000), (1 << 14, 4, 30), (1 << 17, 12, 150), (1 << 19, 20, 64)])
def test_split_plane_remainders(n, zmax, m):
    xdev, xin = _case(n, zmax, zmax + m)
    s = fd.Search(fd.make_config(n, zmax, m, 8192, precision="bf16_split"), device="cuda")
    s.plane.fill_(-1.0)
    s.plane_from_spectrum(xdev)
    torch.cuda.synchronize()
    got = s.plane_2d().cpu().numpy().astype(np.float64)
    ref = oracle.plane(xin, zmax, m)
    assert np.max(np.abs(got - ref) / np.maximum(ref, 2.0)) <= 5e-4
    assert fd.fdas_device_status(s.plan) == 0
