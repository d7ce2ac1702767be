"""GPU: the Fourier parts' own branches against the oracle: generator grids whose half
spectrum lies along x (odd n2, even n0), and the hybrid correction's pruned transforms and
symbol tables on padded nests of sides that are not powers of two, order by order."""

import numpy as np
import pytest

from oracle.hybrid import hybrid_correction
from oracle.noise import gaussian_field, white_noise
from synthetic import Geometry, NestSpec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1103_6031_gb300 as pkg
    return pkg


# tolerance of the generator's other grids: a transform of N points rounds to about
# 1e-16 log2 N
@pytest.mark.parametrize("shape", [(2, 2, 3), (18, 35, 33), (32, 20, 27), (64, 17, 131)])
def test_half_spectrum_along_x(lib, shape):
    import torch
    h = 0.7
    amp = 1.0 / (1.0 + np.linspace(0.0, 9.0, 512))
    dk = 2 * np.pi / h * np.sqrt(3) * 0.45 / 511  # the corner modes lie beyond the table
    noise = white_noise(3, int(np.prod(shape))).reshape(shape)
    ref = gaussian_field(noise, h, amp, dk)
    f = lib.Field(shape, h, amp, dk)
    dev = torch.from_numpy(noise).cuda()
    out = f.convolve(dev)
    assert np.sqrt(np.sum((out.cpu().numpy() - ref) ** 2) / np.sum(ref ** 2)) < 1e-12
    assert torch.equal(dev, torch.from_numpy(noise).cuda())  # the input is left alone
    assert torch.equal(f.convolve(dev, out=dev), out)        # and may be the output
    f.close()


# the oracle forms the multiplier as the difference of its two fractions, which cancels at
# small k: its own error there is eps / (t^n) with t = 2 pi / N, about 1e-9 at order 6, N = 68
@pytest.mark.parametrize("order", (2, 4, 6))
def test_hybrid_padded_sides(lib, order):
    import torch
    geom = Geometry((40, 28, 36), 20.0, order, (NestSpec((34, 18, 26), (9, 8, 10)),))
    h = lib.Hierarchy(lib.config_from_geometry(geom))
    f = np.random.Generator(np.random.PCG64(6)).standard_normal((34, 18, 26))
    psi = [torch.zeros(f.shape, dtype=torch.float64, device="cuda") for _ in range(3)]
    h.hybrid_correction(torch.from_numpy(f).cuda(), psi)
    want = hybrid_correction(f, 0.25, order, pad=True)
    for a, b in zip(psi, want):
        assert np.sqrt(np.sum((a.cpu().numpy() - b) ** 2) / np.sum(b ** 2)) < 1e-9
    h.close()
