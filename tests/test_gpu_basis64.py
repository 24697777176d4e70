"""The FP64 basis kernels (musr_kernels_f64.cuh) against the oracle where they can go wrong: the
edges of a CTA iteration (256 bins) and of the bins between two fresh evaluations of the time
factors (32 iterations), chunks of one to nine histograms, every shape, time zero inside the
histogram, the Gauss-Newton matrix in one pass (musr_gram64.cu), parameters whose factors under- or overflow (evaluated afresh in every bin), FP64 and
FP32 stores.  Tolerance: the FP64 path's, 1e-12 of the value and of each gradient scale."""
import numpy as np
import pytest

import musr_inputs as mi
import oracle
from test_gpu_parity import _check_fp64

pytestmark = pytest.mark.gpu

TF, KT, LKT, EXP, GAUSS = "TFCOS", "KT", "LKT", "EXP", "GAUSS"
# shape name -> terms over slots 0 N0, 1 Nbkg, 2 A, 3 lambda, 4 nu, 5 phi, 6 sigma, 7 Delta, 8 nu2
TERMS = {
    "T1": [[("AMP", (2,)), (EXP, (3,)), (GAUSS, (6,)), (TF, (4, 5))]],
    "N1": [[("AMP", (2,)), (KT, (7,)), (EXP, (3,))]],
    "N1 Lorentzian": [[("AMP", (2,)), (LKT, (7,))]],
    "T1N1": [[("AMP", (2,)), (GAUSS, (6,)), (TF, (4, 5))], [("AMP", (2,)), (KT, (7,)), (GAUSS, (6,))]],
    "T2": [[("AMP", (2,)), (EXP, (3,)), (TF, (4, 5))], [("AMP", (2,)), (GAUSS, (6,)), (TF, (8, 5))]],
    "T2N1": [[("AMP", (2,)), (EXP, (3,)), (TF, (4, 5))], [("AMP", (2,)), (GAUSS, (6,)), (TF, (8, 5))],
             [("AMP", (2,)), (KT, (7,))]],
    "T2m": [[("AMP", (9,)), (EXP, (3,)), (TF, (4, 5))], [("AMP", (9,)), (GAUSS, (6,)), (TF, (8, 5))]],
    "T2N1m": [[("AMP", (9,)), (EXP, (3,)), (TF, (4, 5))], [("AMP", (9,)), (GAUSS, (6,)), (TF, (8, 5))],
              [("AMP", (9,)), (KT, (7,))]],
    "generic": [[("AMP", (2,)), (EXP, (3,))], [("AMP", (2,)), (GAUSS, (6,)), (EXP, (3,))], [("AMP", (2,)), (LKT, (7,))],
                [("AMP", (2,)), (TF, (4, 5))]],
}
SHARED = [0.06, 0.4, 3.0, 0.35, 0.5, 3.4]  # A, lambda, nu, sigma, Delta, nu2


def _problem(shape, nhist, nbins, t0=0.0, dtype=np.float64, shared=SHARED, fit=None):
    """Counts near the model's size (their values only have to be the same on both sides)."""
    rng = np.random.default_rng(nbins * 64 + nhist)
    dt = 12.8 / nbins if nbins > 100 else 0.05
    n = np.arange(nbins)
    base = 40.0 * np.exp(-np.maximum((n - t0) * dt, 0.0) / mi.TAU_MU_US) + 1.5
    counts = rng.poisson(base, size=(nhist, nbins)).astype(dtype)
    rows = [[6 + 3 * j, 7 + 3 * j, 0, 1, 2, 8 + 3 * j, 3, 4, 5, -1] for j in range(nhist)]
    truth = list(shared)
    for j in range(nhist):
        truth += [40.0 + j, 1.5, 17.0 + 45.0 * j]
    names = [f"p{i}" for i in range(len(truth))]
    return mi.Problem(counts, np.full(nhist, float(t0)), dt * 1000.0, fit or (0.5 * dt, nbins * dt), TERMS[shape],
                      np.array(rows, np.int32), np.array([0.07]), len(truth), np.array(truth), names)


def _check(p, x, modes=(0, 1), gn=False):
    from paper_1509_07685_gb300 import binding as B
    with B.Context(p) as ctx:
        for mode in modes:
            v, g, st = ctx.eval(x, mode, B.MUSR_FP64)
            ref = oracle.cost(p, x, mode)
            if np.isfinite(ref[0]):
                _check_fp64(v, g, ref)
            else:  # the cost itself overflows: reported as such, with no gradient
                assert st == B.MUSR_ENONFINITE and np.isinf(v) and not g.any()
            v1, _, _ = ctx.eval(x, mode, B.MUSR_FP64, grad=False)
            assert v1 == v
            if gn:
                H, ref = ctx.gauss_newton(x, mode, B.MUSR_FP64), oracle.gauss_newton(p, x, mode)
                d = np.sqrt(np.diag(ref))
                assert np.all(np.abs(H - ref) <= 1e-12 * np.outer(d, d) + 1e-300)
                _, prod, _ = ctx.gn_product(x, np.eye(x.size), mode, B.MUSR_FP64)  # the same by products
                assert np.all(np.abs(H - 0.5 * (prod + prod.T)) <= 1e-12 * np.outer(d, d) + 1e-300)


@pytest.mark.parametrize("shape", list(TERMS))
@pytest.mark.parametrize("nhist,nbins", [(1, 258), (3, 8193), (9, 771)])
def test_shapes(musr_lib, shape, nhist, nbins):
    p = _problem(shape, nhist, nbins)
    _check(p, p.truth, gn=nbins < 8000)


@pytest.mark.parametrize("nbins", [2, 255, 256, 257, 8191, 8192, 8448, 70001])
def test_edges(musr_lib, nbins):
    p = _problem("T2", 2, nbins, dtype=np.float32)
    _check(p, p.truth)


@pytest.mark.parametrize("lam,sigma,delta", [(400.0, 0.3, 0.5), (0.4, 90.0, 60.0), (-45.0, 0.3, 0.5), (-3.0, 2.0, 900.0)])
def test_factors_out_of_range(musr_lib, lam, sigma, delta):
    """Bins before time zero and rates whose factors leave the double range somewhere in the fit
    (chi^2: the likelihood's logarithm of such values says nothing)."""
    shared = [0.06, lam, 3.0, sigma, delta, 3.4]
    for shape in ("T2N1", "T1N1"):
        p = _problem(shape, 2, 9000, t0=700.25, shared=shared, fit=(-0.8, 12.0))
        _check(p, p.truth, modes=(0,))
