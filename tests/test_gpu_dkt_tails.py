"""Tables of the dynamic Kubo-Toyabe factor whose last block of 256 grid points is nearly empty, at the
change between its two ways of summing a history (160 points in FP32, 255 in FP64) and full.  Tolerance:
test_gpu_dkt.py's."""
import numpy as np
import pytest

import musr_inputs as mi
import oracle
from test_gpu_dkt import FP64_TOL, SPLIT_EPS, _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [256, 257, 300, 336, 415, 416, 417, 511, 512, 513])
def test_last_block(musr_lib, K):
    """K intervals on the coarser grid, 2 K on the finer: 1 .. 256 points in the last block."""
    from paper_1509_07685_gb300 import binding as B
    nbins, width = 800, 12.5
    for prec, step, tol in ((B.MUSR_FP64, 0.02, FP64_TOL), (B.MUSR_SPLIT, 0.03, SPLIT_EPS)):
        nu = step * (K - 0.5) / ((nbins - 1) * width * 1e-3)
        p = mi.dkt_zf(nhist=2, nbins=nbins, bin_width_ns=width, seed=23, delta=0.3, nu_c=nu)
        with B.Context(p) as ctx:
            v, g, st = ctx.eval(p.truth, 1, prec)
            assert st == 0
            _check(p, p.truth, v, g, oracle.cost(p, p.truth, 1), tol)
