"""Searches whose kernels are launched early against the plainly launched steps, and on two streams at once.
sigma2 = 2 makes the normalisation factor 1, so that fdas_spectrum and fdas_plane form the products of the
search bit for bit."""
import numpy as np
import pytest
import torch

import paper_2206_12205_gb300 as fd
from paper_2206_12205_gb300 import fdas as ft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fd.build.build()
    torch.cuda.set_device(0)


def _search(precision, n, zmax, m):
    return fd.Search(fd.make_config(n, zmax, m, 2048 if precision == "fp32" else 4096, max_harm=16,
                                    thr=(14, 20, 30, 44, 70), max_peaks=1 << 17, precision=precision, sigma2=2.0),
                     device="cuda")


def _series(n, seed):
    return torch.from_numpy((np.random.default_rng(seed).standard_normal(n) * np.sqrt(2.0 / n)).astype(np.float32)).cuda()


def _plain(s, x):
    """The plane of the waited-for, plainly launched steps, and the list of that plane."""
    xhat = torch.empty(x.numel(), device="cuda")
    ft.fdas_spectrum(s.plan, x, s.workspace, xhat)
    torch.cuda.synchronize()
    ft.fdas_plane(s.plan, xhat, s.workspace, s.plane)
    torch.cuda.synchronize()
    plane = s.plane.clone()
    s.find_peaks()
    torch.cuda.synchronize()
    return plane, s.peak_list().copy()


# 2^19, 255 templates: 127 x 64 entries in the level search's order, whose work list k4_compact writes
CASES = [("bf16", 1 << 14, 84, 256), ("bf16", 1 << 18, 84, 256), ("bf16", 1 << 19, 84, 256), ("bf16", 1 << 19, 254, 256),
         ("fp32", 1 << 14, 84, 256), ("fp32", 1 << 18, 84, 256), ("fp32", 1 << 19, 254, 256), ("fp16_scaled", 1 << 18, 84, 256),
         ("fp16_scaled", 1 << 19, 84, 256), ("bf16_direct", 1 << 18, 20, 64), ("fp8_direct", 1 << 18, 20, 64)]


@pytest.mark.parametrize("precision,n,zmax,m", CASES)
def test_early_search_equals_the_plain_steps(precision, n, zmax, m):
    ref, s = _search(precision, n, zmax, m), _search(precision, n, zmax, m)
    xs = [_series(n, 17 * k + zmax) for k in range(3)]
    want = [_plain(ref, x) for x in xs]
    assert all(len(w[1]) > 0 for w in want)
    x = xs[0].clone()
    for k in (1, 2, 0, 1, 0, 2, 1):                  # back to back, no synchronisation between the searches
        x.copy_(xs[k])
        s.search(x)
    torch.cuda.synchronize()
    assert torch.equal(s.plane.view(torch.uint8), want[1][0].view(torch.uint8))
    assert np.array_equal(s.peak_list(), want[1][1])


@pytest.mark.parametrize("precision,n,zmax,m", [c for c in CASES if c[2] != 254])
def test_early_searches_on_two_streams(precision, n, zmax, m):
    ref = _search(precision, n, zmax, m)
    xs = [_series(n, 5 * k + zmax) for k in range(2)]
    want = [_plain(ref, x) for x in xs]
    ss = [_search(precision, n, zmax, m) for _ in xs]
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()
    for _ in range(12):
        for s, x, st in zip(ss, xs, streams):
            s.search(x, st)
    torch.cuda.synchronize()
    for s, w in zip(ss, want):
        assert torch.equal(s.plane.view(torch.uint8), w[0].view(torch.uint8))
        assert np.array_equal(s.peak_list(), w[1])
        assert fd.fdas_device_status(s.plan) == 0
