"""Ring lengths at the edges of the transform classes: the last short Bluestein buffer, odd and
even halves just inside and outside each split-convolution buffer, the longest rings; analysis
and synthesis against numpy's FFT in FP64 (every HEALPix length is in test_gpu_parity.py, whose
tolerance of 2e-6 per ring applies here too)."""
import numpy as np
import pytest

from paper_1104_0672_gb300 import inputs

pytestmark = pytest.mark.gpu

LENGTHS = [510, 514, 518, 1022, 1024, 1026, 1028, 1030, 2044, 2050, 2052, 3000, 4094, 4100, 5120, 8188, 8190, 8192, 8196,
           12288, 16380, 16384]


@pytest.mark.parametrize("nphi", LENGTHS)
def test_ring_lengths_at_class_edges(nphi):
    import torch

    import paper_1104_0672_gb300 as ark
    assert torch.cuda.is_available()
    R, B, nh = 5, 3, nphi // 2
    g = ark.Grid.ecp(R, nphi)
    x = inputs.white_noise(R * nphi, B, config=22, salt=nphi)
    spec = ark.ring_analysis(g, torch.from_numpy(x).cuda()).cpu().numpy().reshape(B, R, nh + 1)
    ref = np.fft.rfft(x.reshape(B, R, nphi).astype(np.float64))
    err = np.linalg.norm(spec - ref, axis=2) / np.linalg.norm(ref, axis=2)
    assert err.max() < 2e-6, err.max()
    rng = inputs.rng(22, nphi)
    c = (rng.standard_normal((B, R, nh + 1)) + 1j * rng.standard_normal((B, R, nh + 1))).astype(np.complex64)
    h = np.full(nh + 1, float(nphi))
    h[nh] = 0.5 * nphi
    d = c.astype(np.complex128) * h
    d[:, :, 0] = d[:, :, 0].real
    d[:, :, nh] = 2.0 * d[:, :, nh].real  # half of the +N/2 and of the -N/2 term
    for flags in (0, ark.FLAG_BASIC):
        y = ark.ring_synthesis(g, torch.from_numpy(c).cuda(), flags).cpu().numpy().reshape(B, R, nphi)
        ref = np.fft.irfft(d, nphi)
        err = np.linalg.norm(y - ref, axis=2) / np.linalg.norm(ref, axis=2)
        assert err.max() < 2e-6, (flags, err.max())


def test_ring_lengths_past_the_buffers_are_refused():
    import paper_1104_0672_gb300 as ark
    for nphi in (8194, 16388, 32768):
        with pytest.raises(Exception, match="FFT buffer"):
            ark.Grid.ecp(5, nphi)
