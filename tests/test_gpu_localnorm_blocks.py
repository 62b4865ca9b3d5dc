"""Every block size of the local normalisation against the exact median."""
import numpy as np
import pytest
import torch

import fdas_synth as synth
import paper_2206_12205_gb300 as fd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fd.build.build()
    torch.cuda.set_device(0)


# The scale of a block is sqrt(2 ln 2 / median); its roundings (the power, the quotient, the root and
# the product, each 2^-24 relative, the power's halved by the root) stay below 4 x 2^-23.
@pytest.mark.parametrize("block", [64, 128, 256, 512, 1024, 8192, 16384, 32768, 65536])
def test_local_norm_block_sizes(block):
    n = 1 << 18
    x = torch.from_numpy(synth.noise(n, synth.rng_for(81, 0)).astype(np.float32)).cuda()
    raw = fd.Search(fd.make_config(n, 2, 32, 1024, sigma2=2.0), device="cuda").spectrum(x)
    got = fd.Search(fd.make_config(n, 2, 32, 1024, norm_block=block), device="cuda").spectrum(x)
    torch.cuda.synchronize()
    X = raw.cpu().numpy().view(np.complex64).astype(np.complex128)
    p = np.abs(X) ** 2
    p[0] = np.inf
    p = np.sort(p.reshape(-1, block), axis=1)
    med = p[:, (block - 1) // 2].copy()
    med[0] = p[0, (block - 2) // 2]
    want = X.reshape(-1, block) * np.sqrt(2 * np.log(2.0) / med)[:, None]
    err = np.abs(got.cpu().numpy().view(np.complex64).reshape(-1, block) - want)
    assert np.all(err <= 4 * 2.0 ** -23 * np.abs(want))
