"""A pixel that is not finite reaches only the output rings whose band holds its ring (|theta_i -
theta_j| <= gamma_max; on a pole ring that is summed directly, only the pixels inside the support),
for bands of at most 32 rings, in both forms and every launch shape; every other ring, and every other
map of the call, is bit for bit that of the clean input."""
import numpy as np
import pytest

import oracle
from paper_1104_0672_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spec,support", [
    (("healpix", 64), 3.1),    # 11 rings
    (("healpix", 64), 8.4),    # little left of the 32 slots in groups of four
    (("healpix", 64), 9.3),    # 31 rings: groups of two in the tensor-core form
    (("healpix", 9), 24.0),    # partial ring blocks
    (("ecp", 40, 64), 20.3),
])
@pytest.mark.parametrize("form", ["fp32", "tf32", 1, 3, 4, 5])
def test_non_finite_pixel_stays_in_its_band(spec, support, form):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    g = ark.Grid.healpix(spec[1]) if spec[0] == "healpix" else ark.Grid.ecp(spec[1], spec[2])
    k = ark.Kernel(g, inputs.gaussian_knots(0.4 * support * inputs.DEG, support * inputs.DEG, 60), support * inputs.DEG)
    assert ark.kernel_info(k)[2] <= 32
    flags = 0 if form == "fp32" else ark.FLAG_3XTF32
    B = 3
    if isinstance(form, int):
        ark.set_launch_shape(g, k, B, flags, tc_form=form)
    theta, _, _, n, off = oracle.geometry(spec)
    R = len(theta)
    x = torch.from_numpy(inputs.white_noise(inputs.npix(spec), B, config=24)).cuda()
    clean = ark.convolve(g, k, x, flags).cpu()
    assert clean.isfinite().all()
    for ring, value in ((1, "nan"), (3, "inf"), (R // 3, "nan"), (R // 2, "-inf"), (R - 6, "inf"), (R - 2, "nan")):
        bad = x.clone()
        bad[1, int(off[ring]) + 1] = float(value)
        y = ark.convolve(g, k, bad, flags).cpu()
        assert torch.equal(y[0], clean[0]) and torch.equal(y[2], clean[2])
        for i in range(R):
            a, c = (t[1, int(off[i]):int(off[i] + n[i])] for t in (y, clean))
            if abs(theta[i] - theta[ring]) > support * inputs.DEG:
                assert torch.equal(a, c), (ring, i)
            elif spec[0] == "healpix" and i in (0, R - 1):
                assert ((~a.isfinite()) | (a == c)).all(), (ring, i)
            else:
                assert not a.isfinite().any(), (ring, i)


@pytest.mark.parametrize("ring", [2, 5, 8, 20, 60])
@pytest.mark.parametrize("form", ["fp32", "tf32"])
def test_knots_that_a_non_finite_pixel_reaches(ring, form):
    """With many knots some segments hold no sample of the bad ring's pairs: their gradients stay, to the
    relative 2-norm of 1e-5 of the other knot-gradient tests (pairs next to the poles are projected two to
    a transform, and alone where one of the two is not finite, which rounds differently)."""
    import torch

    import paper_1104_0672_gb300 as ark
    nside, gmax, T = 256, 2.0 * inputs.DEG, 4096
    g = ark.Grid.healpix(nside)
    k = ark.Kernel(g, inputs.gaussian_knots(0.4 * gmax, gmax, T), gmax)
    flags = ark.FLAG_NO_POLE_FIX | (ark.FLAG_3XTF32 if form == "tf32" else 0)
    x, gr = (torch.from_numpy(inputs.white_noise(g.npix, 1, config=29, salt=s)).cuda() for s in (0, 1))
    clean = ark.convolve_backward(g, k, x, gr, False, True, flags)[1][0].cpu().numpy()
    theta, _, _, n, off = oracle.geometry(("healpix", nside))
    x[0, int(off[ring]) + 1] = float("nan")
    bad = ark.convolve_backward(g, k, x, gr, False, True, flags)[1][0].cpu().numpy()
    # knots of the samples of the pairs (i, ring): cap rings of different lengths sample at 2 pi k / N
    N, ut = 4 * nside, 4.0 * np.sin(0.5 * gmax * np.arange(T) / (T - 1)) ** 2
    s2 = np.sin(np.pi * np.arange(N // 2 + 1) / N) ** 2
    reached = np.zeros(T, bool)
    for i in range(2 * ring + 200):
        if abs(theta[i] - theta[ring]) > gmax:
            continue
        A, B = np.sin(0.5 * (theta[i] + theta[ring])) ** 2, np.sin(0.5 * (theta[i] - theta[ring])) ** 2
        u = 4.0 * (B * (1.0 - s2) + A * s2)
        for v in (u * (1.0 - 1e-12), u, u * (1.0 + 1e-12)):  # (either segment where a sample lies on a knot)
            t = np.clip(np.searchsorted(ut, v[v <= ut[-1] * (1.0 + 1e-12)], "right") - 1, 0, T - 2)
            reached[t] = reached[t + 1] = True
    finite = np.isfinite(bad)
    assert not finite[0]
    assert not (~finite & ~reached).any()
    assert np.linalg.norm(bad[finite] - clean[finite]) < 1e-5 * np.linalg.norm(clean[finite])
    assert ring > 20 or (~reached).sum() > 100

