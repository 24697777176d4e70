"""The launch paths of the evaluation kernels at their limits, against the oracle: parameters that go
with the launch (up to 128) or are copied, jobs of one chunk (columns and lists in shared memory, up
to 255 parameters and 256 columns) and of several, chunks with unused histograms, rows of a chunk in
groups of 16 and remainders, single calls and batches, alternating so that every call finds
another's job table.  Tolerances: the two paths' own (test_gpu_parity)."""
import numpy as np
import pytest

import musr_inputs as mi
import oracle
from test_gpu_parity import _check_fp64, _check_split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nhist,nbins", [(1, 700), (7, 9000), (8, 34000), (9, 5000), (41, 1500), (42, 1500), (90, 600)])
def test_single_and_batched_calls(musr_lib, nhist, nbins):
    from paper_1509_07685_gb300 import binding as B
    p = mi.cfg2(nhist=nhist, nbins=nbins, bin_width_ns=12800.0 / nbins, seed=nhist, n0=60.0)  # 4 + 3 nhist parameters
    X = mi.jitter(p.truth, 3, seed=nhist, lo=0.98, hi=1.02)
    ref = {m: [oracle.cost(p, x, m) for x in X] for m in (0, 1)}
    with B.Context(p) as ctx:
        for mode in (0, 1):
            for prec, check in ((B.MUSR_SPLIT, _check_split), (B.MUSR_FP64, _check_fp64)):
                for i in (0, 1):  # another point through the same job table
                    v, g, st = ctx.eval(X[i], mode, prec)
                    assert st == 0
                    check(v, g, ref[mode][i])
                vals, grads, st = ctx.eval_batch(X, mode, prec)
                assert st == 0
                for i in range(3):
                    check(vals[i], grads[i], ref[mode][i])
                v, _, _ = ctx.eval(X[2], mode, prec, grad=False)
                v2, _, _ = ctx.eval(X[2], mode, prec)
                assert v == v2
