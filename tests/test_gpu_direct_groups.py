"""The direct plane around its register and window groups, against the FP64 oracle with the parity
test's bounds."""
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


# templates around the register groups (padded counts 32 | 40, 64 | 72), taps around the 96-thread
# window passes ((512 + m) / 4 groups of 4 words: 96 and 192 are whole passes)
@pytest.mark.parametrize("n,zmax,m", [(1 << 14, 30, 64), (1 << 14, 32, 72), (1 << 13, 62, 128), (1 << 13, 64, 136),
                                       (1 << 12, 8, 256), (1 << 12, 8, 264), (1 << 11, 6, 512)])
def test_direct_plane_groups(n, zmax, m):
    xdev, xin = _case(n, zmax, zmax + m)
    s = fd.Search(fd.make_config(n, zmax, m, 8192, precision="bf16_direct"), device="cuda")
    s.plane_from_spectrum(xdev)
    torch.cuda.synchronize()
    got = s.plane_2d().float().cpu().numpy().astype(np.float64)
    ref = oracle.plane(xin, zmax, m)
    fr = np.abs(got - ref) / np.maximum(ref, 2.0)
    local = np.maximum.reduceat(np.maximum(ref, 2.0), np.arange(0, ref.shape[1], 64), axis=1)
    local = np.maximum(local, np.maximum(np.roll(local, 1, axis=1), np.roll(local, -1, axis=1)))
    bound = 0.03 * np.maximum(ref, 2.0) + 0.02 * np.sqrt(np.maximum(ref, 2.0) * np.repeat(local, 64, axis=1)[:, :ref.shape[1]])
    assert np.all(np.abs(got - ref) <= bound)
    assert np.sqrt(np.mean(fr ** 2)) <= 0.006 and np.percentile(fr, 99.9) <= 0.015
