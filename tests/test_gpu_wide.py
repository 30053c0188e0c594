"""Bands wider than 32 input rings (the 32 slots of the contraction move along the band), in both
forms, against the FP64 oracle: one window past the narrow form, several windows, bands over most of
the sphere, partial ring blocks, kernel grids that are no power of two, rings of more than 128
samples with and without tabulated coefficients.  Tolerance: the method's fractional RMS, 1e-5,
as in test_gpu_parity.py."""
import numpy as np
import pytest

import oracle
from paper_1104_0672_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _setup(spec, supports, nmaps):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    g = ark.Grid.healpix(spec[1]) if spec[0] == "healpix" else ark.Grid.ecp(spec[1], spec[2])
    prof = [(inputs.gaussian_knots(0.4 * s * inputs.DEG, s * inputs.DEG, 100), s * inputs.DEG) for s in supports]
    ks = [ark.Kernel(g, k, gm) for k, gm in prof]
    assert max(ark.kernel_info(k)[2] for k in ks) > 32
    x = inputs.white_noise(inputs.npix(spec), nmaps, config=21)
    return ark, g, prof, ks, x, torch.from_numpy(x).cuda()


@pytest.mark.parametrize("spec,supports,nmaps,basic,rings", [
    (("healpix", 64), [14.2], 1, False, None),                # 33-36 rings: one slot past the window
    (("healpix", 64), [29.0], 3, False, None),                # three windows, maps summed through memory
    (("healpix", 64), [29.0], 2, True, None),
    (("healpix", 19), [75.0], 1, False, None),                # bands over most of the sphere, partial blocks
    (("healpix", 48), [20.0, 16.5, 33.0], 3, False, None),    # per-map beams of different widths
    (("ecp", 90, 178), [42.0], 2, False, None),               # N no power of two
    (("ecp", 61, 720), [60.0], 1, False, None),               # over 128 samples in every pair near a pole
    (("healpix", 512), [6.0], 1, False, [0, 1, 15, 16, 40, 170, 186, 511, 512, 1023, 1900, 2046]),  # untabulated
])
@pytest.mark.parametrize("form", ["tf32", "fp32"])
def test_wide_band(spec, supports, nmaps, basic, rings, form):
    ark, g, prof, ks, x, xt = _setup(spec, supports, nmaps)
    flags = (ark.FLAG_3XTF32 if form == "tf32" else 0) | (ark.FLAG_BASIC if basic else 0)
    y = ark.convolve(g, ks[0] if len(ks) == 1 else ks, xt, flags).cpu().numpy()
    _, _, _, n, off = oracle.geometry(spec)
    at = slice(None) if rings is None else np.concatenate([np.arange(off[r], off[r] + n[r]) for r in rings])
    for b in range(nmaps):
        knots, gmax = prof[b % len(prof)]
        ref = oracle.convolve(spec, knots, gmax, x[b].astype(np.float64), variant="basic" if basic else "enhanced",
                              rings=rings)
        ref = ref[at] if ref.size == y.shape[1] else ref
        err = float(np.linalg.norm(y[b][at] - ref) / np.linalg.norm(ref))
        assert err < TOL, (b, err)


def test_wide_band_non_finite_input_stays_in_its_support():
    ark, g, prof, ks, x, xt = _setup(("healpix", 64), [29.0], 1)
    _, _, _, n, off = oracle.geometry(("healpix", 64))
    for ring in (3, 70, 127, 200):
        bad = xt.clone()
        bad[0, int(off[ring]) + 1] = float("nan")
        a, b = (torch_isnan(ark.convolve(g, ks[0], bad, f)) for f in (0, ark.FLAG_3XTF32))
        assert a.any() and not a.all()
        assert (a == b).all()


def torch_isnan(t):
    return t.isnan().cpu().numpy()
