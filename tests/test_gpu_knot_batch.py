"""Knot gradients of several kernels in one call: bit for bit those of one call per kernel, and
against the FP64 oracle, for kernels whose lists of FFT-projected pairs differ in length, with and
without them, in both forms and with one to many knots.  Tolerance: the relative 2-norm 1e-5 of
the other knot-gradient tests."""
import numpy as np
import pytest

import oracle
from paper_1104_0672_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.mark.parametrize("spec,supports,T,check", [
    (("healpix", 256), [2.0, 1.1, 2.6, 1.7], 97, [0]),        # FFT pairs of different numbers
    (("healpix", 24), [30.7, 44.3], 2, [0, 1]),               # two knots, no FFT pairs, wide band
    (("ecp", 31, 90), [35.0, 21.0, 60.0], 40, [0, 2]),        # N no power of two
    (("healpix", 64), [9.0, 6.0], 4096, [1]),                 # fewer bins per CTA
    (("ecp", 33, 600), [40.0, 30.0], 64, [0]),                # pairs of more than 128 samples, no FFT
])
@pytest.mark.parametrize("form", ["fp32", "tf32"])
def test_knot_gradients_of_several_kernels(spec, supports, T, check, form):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    g = ark.Grid.healpix(spec[1]) if spec[0] == "healpix" else ark.Grid.ecp(spec[1], spec[2])
    prof = [(inputs.gaussian_knots(0.4 * s * inputs.DEG, s * inputs.DEG, T), s * inputs.DEG) for s in supports]
    ks = [ark.Kernel(g, k, gm) for k, gm in prof]
    n = len(ks)
    x, gr = (inputs.white_noise(inputs.npix(spec), n, config=23, salt=s) for s in (0, 1))
    xt, gt = torch.from_numpy(x).cuda(), torch.from_numpy(gr).cuda()
    flags = ark.FLAG_3XTF32 if form == "tf32" else 0
    _, gk = ark.convolve_backward(g, ks, xt, gt, True, True, flags)
    for b in range(n):
        _, one = ark.convolve_backward(g, ks[b], xt[b:b + 1], gt[b:b + 1], False, True, flags)
        assert torch.equal(one[0], gk[b])
    for b in check:
        ref = oracle.knot_grad(spec, prof[b][0], prof[b][1], x[b].astype(np.float64), gr[b].astype(np.float64))
        err = float(np.linalg.norm(gk[b].cpu().numpy() - ref) / np.linalg.norm(ref))
        assert err < TOL, (b, err)
