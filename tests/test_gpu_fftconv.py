"""The FP64 Poisson solve's pruned transforms (musr_fftconv.cu) where their plans differ: every radix
alone and in products, lengths that are padded to the next such product, odd and even half lengths
(the self-conjugate frequencies), a last row without a partner, the block widths of long axes, axes
too long for the kernels (cuFFT).  Against numpy's FFT of the doubled mesh in FP64: both round each
of O(log2 N) stages by about 1e-16 of the largest potential, far below 1e-12 of it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _numpy(rho, h):
    n = rho.shape
    d = [np.minimum(np.arange(2 * k), 2 * k - np.arange(2 * k)) * w for k, w in zip(n, h)]
    r = np.sqrt(d[0][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[2][None, None, :] ** 2)
    r[0, 0, 0] = min(h)
    s = [2 * k for k in n]
    phi = np.fft.irfftn(np.fft.rfftn(rho, s, (0, 1, 2)) * np.fft.rfftn(1.0 / r), s, (0, 1, 2))
    return phi[:n[0], :n[1], :n[2]] * h[0] * h[1] * h[2]


@pytest.mark.parametrize("shape", [
    (2, 3, 4), (5, 7, 8), (9, 10, 25), (14, 21, 35), (16, 49, 15), (64, 8, 64), (11, 13, 17), (23, 19, 31),
    (1, 1, 300), (1, 37, 1), (300, 1, 2), (3, 520, 5), (2, 3, 1030), (1100, 2, 3), (2, 2050, 1), (1, 4096, 2),
    (4100, 1, 2), (2, 1, 5003), (1, 65, 129), (40, 96, 33)])
def test_meshes(musr_lib, shape):
    from paper_1509_07685_gb300 import binding as B
    rng = np.random.default_rng(sum(shape))
    rho, h = rng.normal(size=shape), (0.31, 0.2, 0.45)
    ref = _numpy(rho, h)
    with B.Poisson(shape, h, B.MUSR_FP64) as ps:
        for _ in range(2):  # the second solve finds the first one's buffers
            phi = ps.solve(rho)
            assert np.max(np.abs(phi - ref)) <= 1e-12 * np.max(np.abs(ref))
