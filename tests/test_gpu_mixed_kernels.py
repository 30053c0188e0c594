"""Kernels of different kinds in one call: weighted sums of kernels that share one support radius (and
so the widest kernel's sample slots) but differ in knot count, against the sum of the oracle's
convolutions; per-map beams of which some need the wide form, bit for bit the single calls."""
import numpy as np
import pytest

import oracle
from paper_1104_0672_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("supports", [[11.0, 11.0, 11.0], [11.0, 24.0, 24.0, 7.0]])
@pytest.mark.parametrize("form", ["fp32", "tf32"])
def test_weighted_sum_of_kernels_of_different_knot_counts(supports, form):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    spec, T, w = ("healpix", 32), [17, 400, 3, 64], [0.75, -0.5, 1.25, 2.0]
    g = ark.Grid.healpix(spec[1])
    prof = [(inputs.gaussian_knots((0.3 + 0.1 * i) * s * inputs.DEG, s * inputs.DEG, T[i]), s * inputs.DEG)
            for i, s in enumerate(supports)]
    ks = [ark.Kernel(g, k, gm) for k, gm in prof]
    x = inputs.white_noise(inputs.npix(spec), 2, config=27)
    flags = ark.FLAG_3XTF32 if form == "tf32" else 0
    y = ark.convolve_multi(g, ks, torch.from_numpy(x).cuda(), w[:len(ks)], flags).cpu().numpy()
    for b in range(2):
        ref = sum(w[i] * oracle.convolve(spec, k, gm, x[b].astype(np.float64)) for i, (k, gm) in enumerate(prof))
        err = float(np.linalg.norm(y[b] - ref) / np.linalg.norm(ref))
        assert err < 1e-5, (b, err)


@pytest.mark.parametrize("spec,supports", [
    (("healpix", 64), [5.0, 29.0, 9.0, 14.2]),
    (("healpix", 512), [1.0, 6.0]),             # the wide one has untabulated pairs of over 128 samples
    (("ecp", 61, 720), [20.0, 60.0, 3.1]),
])
@pytest.mark.parametrize("form", ["fp32", "tf32"])
def test_per_map_beams_of_which_some_are_wide(spec, supports, form):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    g = ark.Grid.healpix(spec[1]) if spec[0] == "healpix" else ark.Grid.ecp(spec[1], spec[2])
    ks = [ark.Kernel(g, inputs.gaussian_knots(0.4 * s * inputs.DEG, s * inputs.DEG, 100), s * inputs.DEG) for s in supports]
    bands = [ark.kernel_info(k)[2] for k in ks]
    assert min(bands) <= 32 < max(bands)
    x = torch.from_numpy(inputs.white_noise(inputs.npix(spec), len(ks), config=28)).cuda()
    flags = ark.FLAG_3XTF32 if form == "tf32" else 0
    y = ark.convolve(g, ks, x, flags)
    for b, k in enumerate(ks):
        assert torch.equal(ark.convolve(g, k, x[b], flags), y[b]), b


@pytest.mark.parametrize("spec,supports", [
    (("ecp", 64, 128), [17.4, 20.2]),     # groups of four reach 16 and 18 slots
    (("ecp", 64, 128), [17.4, 8.0]),
    (("healpix", 32), [7.3, 9.0, 11.5]),  # 14 to 22 slots
])
@pytest.mark.parametrize("form", ["fp32", "tf32"])
def test_narrow_bands_around_sixteen_slots(spec, supports, form):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    g = ark.Grid.healpix(spec[1]) if spec[0] == "healpix" else ark.Grid.ecp(spec[1], spec[2])
    prof = [(inputs.gaussian_knots(0.4 * s * inputs.DEG, s * inputs.DEG, 80), s * inputs.DEG) for s in supports]
    ks = [ark.Kernel(g, k, gm) for k, gm in prof]
    x = inputs.white_noise(inputs.npix(spec), len(ks), config=31)
    xt = torch.from_numpy(x).cuda()
    flags = ark.FLAG_3XTF32 if form == "tf32" else 0
    y = ark.convolve(g, ks, xt, flags)
    for b, k in enumerate(ks):
        assert torch.equal(ark.convolve(g, k, xt[b], flags), y[b]), b
        ref = oracle.convolve(spec, *prof[b], x[b].astype(np.float64))
        err = float(np.linalg.norm(y[b].cpu().numpy() - ref) / np.linalg.norm(ref))
        assert err < 1e-5, (b, err)
