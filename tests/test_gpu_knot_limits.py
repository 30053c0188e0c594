"""Knot gradients at the limits of a call: as many knots as a kernel may have on the longest kernel grid
(the knot tables beside the projection's 16384-point transform), against the FP64 oracle (relative
2-norm 1e-5, as the other knot-gradient tests); and the workspace of many kernels."""
import numpy as np
import pytest

import oracle
from paper_1104_0672_gb300 import inputs

pytestmark = pytest.mark.gpu


# The transform's buffer takes 139392 of 232448 bytes; a table of T doubles 8 T: three tables fit up to
# T = 3877, two up to the largest T = 4096.
@pytest.mark.parametrize("T", [3877, 3878, 4096])
def test_knot_gradient_of_many_knots_on_the_longest_grid(T):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    spec, gmax = ("ecp", 3, 16384), 20.3 * inputs.DEG  # one pair per ring, of 920 samples or more
    g = ark.Grid.ecp(*spec[1:])
    knots = inputs.gaussian_knots(8.0 * inputs.DEG, gmax, T)
    k = ark.Kernel(g, knots, gmax)
    x, gr = (inputs.white_noise(inputs.npix(spec), 1, config=25, salt=s) for s in (0, 1))
    _, gk = ark.convolve_backward(g, k, torch.from_numpy(x).cuda(), torch.from_numpy(gr).cuda(), False, True)
    ref = oracle.knot_grad(spec, knots, gmax, x[0].astype(np.float64), gr[0].astype(np.float64))
    err = float(np.linalg.norm(gk[0].cpu().numpy() - ref) / np.linalg.norm(ref))
    assert err < 1e-5, err


# Pairs of more than 128 samples without a transform, projected by warps with bins of their own (up to
# 1052 knots) or that 2, 4 and 8 warps share.
@pytest.mark.parametrize("T", [1052, 1053, 1894, 1895, 3157, 3158, 4096])
def test_knot_gradient_of_many_knots_without_a_transform(T):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    spec, supports = ("ecp", 17, 600), [35.3, 24.7]
    g = ark.Grid.ecp(*spec[1:])
    prof = [(inputs.gaussian_knots(0.4 * s * inputs.DEG, s * inputs.DEG, T), s * inputs.DEG) for s in supports]
    ks = [ark.Kernel(g, k, gm) for k, gm in prof]
    x, gr = (inputs.white_noise(inputs.npix(spec), 2, config=30, salt=s) for s in (0, 1))
    xt, gt = torch.from_numpy(x).cuda(), torch.from_numpy(gr).cuda()
    _, gk = ark.convolve_backward(g, ks, xt, gt, False, True)
    for b in range(2):
        _, one = ark.convolve_backward(g, ks[b], xt[b:b + 1], gt[b:b + 1], False, True)
        assert torch.equal(one[0], gk[b])
        ref = oracle.knot_grad(spec, prof[b][0], prof[b][1], x[b].astype(np.float64), gr[b].astype(np.float64))
        err = float(np.linalg.norm(gk[b].cpu().numpy() - ref) / np.linalg.norm(ref))
        assert err < 1e-5, (b, err)


def test_workspace_of_many_kernels_stays_bounded():
    """Kernels of one call share launches in batches; what a batch adds for its kernels -- rows of Q,
    projections and FP64 partial sums together -- stays within 256 MiB, or what one kernel needs."""
    import paper_1104_0672_gb300 as ark

    def knot_bytes(g, ks):  # the backward workspace less the forward one and the gradients' spectra
        n = len(ks)
        spec = n * ((g.nrings + 1) // 2) * (g.nlon // 2 + 1) * 16
        return ark.workspace_size(g, ks, n, 0, True) - ark.workspace_size(g, ks, n, 0, False) - spec

    for nside, support, T in ((16, 20.0, 4096), (8, 89.0, 4096), (16, 20.0, 100), (128, 40.0, 1000)):
        g = ark.Grid.healpix(nside)
        knots = inputs.gaussian_knots(0.4 * support * inputs.DEG, support * inputs.DEG, T)
        ks = [ark.Kernel(g, knots, support * inputs.DEG) for _ in range(32)]
        assert knot_bytes(g, ks) <= max(256 << 20, knot_bytes(g, ks[:1])) + 4096, (nside, support, T)
