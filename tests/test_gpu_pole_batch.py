"""Pole pixels do not depend on how many maps share a call: the FP64 direct sum of a pole pixel is
taken in the same order for a map alone, in a batch and in chunks of a host call.

The maps are antisymmetric about the meridian of pixel 0 (pixel q of a cap ring of 4 i pixels and pixel
i - 1 - q are mirror images), so the sums at pixels 0 and 2 of the pole rings cancel to the rounding
errors of their order of summation."""
import numpy as np
import pytest

import oracle
from paper_1104_0672_gb300 import inputs

pytestmark = pytest.mark.gpu


def _antisymmetric(nside, B):
    _, _, _, n, off = oracle.geometry(("healpix", nside))
    x = inputs.white_noise(inputs.npix(("healpix", nside)), B, config=26).copy()
    for r in list(range(nside - 1)) + list(range(3 * nside, 4 * nside - 1)):
        q = np.arange(n[r])
        ring = x[:, off[r]:off[r] + n[r]]
        x[:, off[r]:off[r] + n[r]] = ring - ring[:, (n[r] // 4 - 1 - q) % n[r]]
    return x


@pytest.mark.parametrize("supports", [[9.0], [20.0], [20.0, 5.0, 9.0, 14.0]])  # 364 to 1860 pixels of the pole's rings
def test_pole_pixels_of_a_batch_and_of_single_maps(supports):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    nside, B = 64, 20
    g = ark.Grid.healpix(nside)
    ks = [ark.Kernel(g, inputs.gaussian_knots(0.4 * s * inputs.DEG, s * inputs.DEG, 100), s * inputs.DEG) for s in supports]
    per_map = [ks[b % len(ks)] for b in range(B)]
    xh = torch.from_numpy(_antisymmetric(nside, B)).pin_memory()
    x = xh.cuda()
    for flags in (0, ark.FLAG_3XTF32):
        y = ark.convolve(g, ks[0] if len(ks) == 1 else per_map, x, flags)
        poles = torch.cat([y[:, :4], y[:, -4:]], 1)
        assert poles.isfinite().all() and (poles[:, 1].abs() > 1e-6).all()
        assert (poles[:, 0].abs() < 1e-12).all() and (poles[:, 0] != 0).any()  # cancelled to rounding errors
        host = ark.convolve_host(g, ks[0] if len(ks) == 1 else per_map, xh, flags, maps_per_chunk=3)
        torch.cuda.synchronize()
        assert torch.equal(host, y.cpu())
        for b in range(B):
            assert torch.equal(ark.convolve(g, per_map[b], x[b], flags), y[b]), b
