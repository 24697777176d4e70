"""The FP64 Poisson solve's kernels on meshes with few lines (fewer columns to a block than its length
allows) and at the rule that leaves long axes with few lines to the library.  Reference and tolerance:
test_gpu_fftconv.py's."""
import numpy as np
import pytest

from test_gpu_fftconv import _numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [
    (1, 1, 1), (1, 1, 300), (300, 1, 1), (1, 300, 1), (2, 2, 500), (3, 700, 2), (5, 3, 1024), (40, 5, 6), (152, 1, 3),
    (1536, 2, 3), (1537, 4, 7), (1537, 4, 8), (6, 2048, 5), (6, 2048, 6), (5, 7, 4000), (7, 5, 2050), (4096, 6, 5),
    (4096, 6, 6)])
def test_thin_meshes(musr_lib, shape):
    from paper_1509_07685_gb300 import binding as B
    rng = np.random.default_rng(sum(shape))
    rho, h = rng.normal(size=shape), (0.31, 0.2, 0.45)
    ref = _numpy(rho, h)
    with B.Poisson(shape, h, B.MUSR_FP64) as ps:
        for _ in range(2):
            assert np.max(np.abs(ps.solve(rho) - ref)) <= 1e-12 * np.max(np.abs(ref))
