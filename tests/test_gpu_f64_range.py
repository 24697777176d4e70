"""The FP64 basis kernels where a cost is defined but its counts, model or rates lie far from 1, against
the oracle: counts far below the model (fractional counts of FP64 histograms, growing rates) and far
above it.  Tolerance: the FP64 path's, 1e-12 of the value and of each gradient scale; every term of the
value is formed with a relative error of a few roundings of the larger of d and N."""
import numpy as np
import pytest

import musr_inputs as mi
import oracle
from test_gpu_parity import _check_fp64

pytestmark = pytest.mark.gpu

# slots: 0 N0, 1 Nbkg, 2 A, 3 lambda, 4 nu, 5 phi, 6 sigma
TERMS = {
    "T1": [[("AMP", (2,)), ("EXP", (3,)), ("TFCOS", (4, 5))]],
    "N1": [[("AMP", (2,)), ("EXP", (3,)), ("GAUSS", (6,))]],
    "generic": [[("AMP", (2,)), ("EXP", (3,))], [("AMP", (2,)), ("GAUSS", (6,))]],
}


def _problem(terms, counts, truth, dt=0.02, fit=None):
    nhist, nbins = counts.shape
    rows = np.array([[0, 1, 2, 3, 4, 5, 6]] * nhist, np.int32)
    return mi.Problem(counts, np.zeros(nhist), dt * 1000.0, fit or (0.0, nbins * dt), terms, rows, np.zeros(1), 7,
                      np.array(truth), [f"p{i}" for i in range(7)])


def _check(p, mode=1):
    from paper_1509_07685_gb300 import binding as B
    with B.Context(p) as ctx:
        ref = oracle.cost(p, p.truth, mode)
        assert np.isfinite(ref[0])
        v, g, st = ctx.eval(p.truth, mode, B.MUSR_FP64)
        assert st == B.MUSR_OK and np.all(np.isfinite(g))
        _check_fp64(v, g, ref)
        assert ctx.eval(p.truth, mode, B.MUSR_FP64, grad=False)[0] == v


@pytest.mark.parametrize("shape", list(TERMS))
def test_counts_far_below_the_model(musr_lib, shape):
    rng = np.random.default_rng(5)
    counts = 10.0 ** rng.uniform(-25.0, 1.0, size=(2, 611))
    counts[:, ::7] = 0.0
    _check(_problem(TERMS[shape], counts, [40.0, 1.5, 0.06, 0.4, 3.0, 17.0, 0.35]))


@pytest.mark.parametrize("shape", ["N1", "generic"])
@pytest.mark.parametrize("lam,n0", [(-3.3, 1.0), (-5.0, 40.0), (0.4, 1e18), (60.0, 1e-20)])
def test_integer_counts_far_from_the_model(musr_lib, shape, lam, n0):
    rng = np.random.default_rng(6)
    counts = rng.poisson(3.0, size=(3, 611)).astype(np.float32)
    _check(_problem(TERMS[shape], counts, [n0, 0.0, 0.3, lam, 3.0, 17.0, 0.1]))


def test_subnormal_model(musr_lib):
    """N below 2^-1022 (no background, a tiny N0): finite with fractional counts."""
    rng = np.random.default_rng(7)
    counts = rng.uniform(0.5e-6, 2e-6, size=(2, 97))
    _check(_problem(TERMS["N1"], counts, [1.3e-308, 0.0, 0.3, 0.4, 3.0, 17.0, 0.1]))


@pytest.mark.parametrize("mode,count,bkg", [(1, 5.0, 6e307), (0, 6e307, 2.0)])
def test_largest_counts_and_model(musr_lib, mode, count, bkg):
    """One bin with N, or d, above 2^1022, where 1 / N and 1 / d are subnormal: -2lnL = 2 N and its gradient 2
    along Nbkg; chi^2 = d and -2."""
    from paper_1509_07685_gb300 import binding as B
    p = _problem(TERMS["N1"], np.full((1, 4), count), [1.0, bkg, 0.3, 0.4, 3.0, 17.0, 0.1], fit=(0.019, 0.021))
    with B.Context(p) as ctx:
        assert ctx.bins_in_fit() == 1
        v, g, st = ctx.eval(p.truth, mode, B.MUSR_FP64)
        want, slope = (2.0 * bkg, 2.0) if mode else (count, -2.0)
        assert st == B.MUSR_OK and abs(v / want - 1.0) <= 1e-12 and abs(g[1] - slope) <= 1e-12
        assert ctx.eval(p.truth, mode, B.MUSR_FP64, grad=False)[0] == v
        H, (_, prod, _) = ctx.gauss_newton(p.truth, mode, B.MUSR_FP64), ctx.gn_product(p.truth, np.eye(7), mode, B.MUSR_FP64)
        curv = 2.0 * count / bkg / bkg if mode else 2.0 / count  # d^2 cost / dN^2
        assert abs(H[1, 1] - curv) <= 1e-12 * curv + 1e-323 and abs(prod[1, 1] - curv) <= 1e-12 * curv + 1e-323


@pytest.mark.parametrize("shape,lam,sigma", [("N1", 0.4, 1e170), ("generic", 0.4, 1e170), ("rates", 1.2e308, 0.1)])
def test_rates_whose_combination_overflows(musr_lib, shape, lam, sigma):
    """sigma^2 and a sum of rates beyond the double range: the factor is 1 at time zero and 0 after it."""
    terms = [[("AMP", (2,)), ("EXP", (3,)), ("EXP", (3,))]] if shape == "rates" else TERMS[shape]
    counts = np.random.default_rng(8).poisson(3.0, size=(2, 300)).astype(np.float64)
    p = _problem(terms, counts, [4.0, 1.5, 0.3, lam, 3.0, 17.0, sigma])
    for mode in (0, 1):
        _check(p, mode)


@pytest.mark.parametrize("prim", ["EXP", "LKT"])
def test_factors_that_overflow_past_the_window(musr_lib, prim):
    """A growing factor that stays finite up to the last bin (its amplitude keeps N near 1) and overflows within
    the rest of a CTA iteration: the bins past the window leave the gradient alone."""
    nbins, dt = 300, 0.5
    rate = -700.0 / (nbins * dt)
    a = 1e-290 if prim == "EXP" else 1e-293
    counts = np.random.default_rng(9).poisson(20.0, size=(2, nbins)).astype(np.float64)
    terms = [[("AMP", (2,)), (prim, (3,))], [("AMP", (6,)), ("EXP", (4,))]]
    p = _problem(terms, counts, [2.0, 1.5, a, rate, 0.3, 17.0, 0.2], dt=dt)
    for mode in (0, 1):
        _check(p, mode)


@pytest.mark.parametrize("lam,sigma,kt,t0", [(0.4, 48.8, 0.5, 3.0), (0.4, 0.3, 48.8, 3.0), (0.4, 90.0, 0.1, 1.0),
                                             (0.2, 12.0, 12.0, 40.25), (-11.5, 0.1, 0.1, 1600.0),
                                             (0.1, 1.3, 1.3, 1600.0)])
def test_factors_taken_over_many_steps(musr_lib, lam, sigma, kt, t0):
    """Rates whose factors a thread takes over up to 31 steps of 256 bins from a bin before time zero, where the
    cross term of a Gaussian grows with every step: a batch of vectors, whose tiles hold that many steps."""
    from paper_1509_07685_gb300 import binding as B
    terms = [[("AMP", (2,)), ("EXP", (3,)), ("GAUSS", (6,))], [("AMP", (2,)), ("KT", (4,))]]
    counts = np.random.default_rng(10).poisson(9.0, size=(3, 3150)).astype(np.float64)
    p = _problem(terms, counts, [4.0, 1.5, 0.1, lam, kt, 17.0, sigma], dt=0.0103, fit=(-40.0, 40.0))
    p.t0[:] = t0
    X = np.stack([p.truth] * 700)
    with B.Context(p) as ctx:
        for mode in (0, 1):
            ref = oracle.cost(p, p.truth, mode)
            vals, grads, st = ctx.eval_batch(X, mode, B.MUSR_FP64)
            assert st == B.MUSR_OK and np.isfinite(ref[0]) and np.all(np.isfinite(grads))
            for i in (0, 699):
                _check_fp64(vals[i], grads[i], ref)
