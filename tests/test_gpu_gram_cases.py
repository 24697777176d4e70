"""The FP64 Gauss-Newton matrix in one pass (musr_gram64.cu) for maps and theories beyond the plain ones,
against the oracle's matrix and the products with unit vectors (1e-12 of sqrt(H_ii H_jj): the path's
tolerance)."""
import numpy as np
import pytest

import musr_inputs as mi
import oracle

pytestmark = pytest.mark.gpu


def _counts(nhist, nbins, seed=9):
    rng = np.random.default_rng(seed)
    return rng.poisson(30.0, size=(nhist, nbins)).astype(np.float64)


def _check(p, modes=(0, 1)):
    from paper_1509_07685_gb300 import binding as B
    with B.Context(p) as ctx:
        for mode in modes:
            H, ref = ctx.gauss_newton(p.truth, mode, B.MUSR_FP64), oracle.gauss_newton(p, p.truth, mode)
            _, prod, _ = ctx.gn_product(p.truth, np.eye(p.nparams), mode, B.MUSR_FP64)
            d = np.sqrt(np.diag(ref))
            tol = 1e-12 * np.outer(d, d) + 1e-300
            assert np.all(np.abs(H - ref) <= tol), (mode, np.max(np.abs(H - ref) / tol))
            assert np.all(np.abs(H - 0.5 * (prod + prod.T)) <= tol)


@pytest.mark.parametrize("terms", [
    [[("AMP", (0,)), ("EXP", (2,))]],                      # the amplitude reads N0's slot
    [[("AMP", (2,)), ("EXP", (0,))]],                      # the rate does
    [[("AMP", (2,)), ("TFCOS", (3, 0))]],                  # the phase
    [[("AMP", (1,)), ("EXP", (2,))]],                      # the amplitude reads Nbkg's slot
    [[("AMP", (2,)), ("GAUSS", (1,)), ("TFCOS", (3, 4))]],  # the width does
])
def test_primitives_on_the_first_slots(musr_lib, terms):
    """N0 = 3, Nbkg = 0.4, A = 0.3 (N > 0 throughout)."""
    truth = np.array([3.0, 0.4, 0.3, 1.7, 20.0])
    rows = np.array([[0, 1, 2, 3, 4]] * 2, np.int32)
    used = {0, 1} | {s for t in terms for _, slots in t for s in slots}
    if 4 not in used:  # parameters nothing reads: constants
        rows = np.where(np.isin(rows, list(used)), rows, -1 - rows)
    idx = {s: i for i, s in enumerate(sorted(used))}
    rows = np.array([[idx[v] if v >= 0 else v for v in r] for r in rows], np.int32)
    p = mi.Problem(_counts(2, 700), np.zeros(2), 8.0, (0.0, 5.6), terms, rows, truth.copy(), len(idx),
                   truth[sorted(used)], [f"p{i}" for i in idx])
    _check(p)


def test_more_parameters_than_a_launch_carries(musr_lib):
    """Beyond 128 parameters they are copied to the device; the first call on a context takes the same
    kernel as the next one (the same bits)."""
    from paper_1509_07685_gb300 import binding as B
    p = mi.cfg2(nhist=48, nbins=700, bin_width_ns=16.0, seed=4, n0=60.0)  # 4 + 3 x 48 parameters
    assert p.nparams > 128
    for mode in (0, 1):
        with B.Context(p) as ctx:
            H = ctx.gauss_newton(p.truth, mode, B.MUSR_FP64)
            assert np.array_equal(ctx.gauss_newton(p.truth, mode, B.MUSR_FP64), H)
            v, g, _ = ctx.eval(p.truth, mode, B.MUSR_FP64)  # the context's tables still hold
            ref = oracle.cost(p, p.truth, mode)
            assert abs(v - ref[0]) <= 1e-12 * abs(ref[0]) and np.all(np.abs(g - ref[1]) <= 1e-12 * ref[2] + 1e-300)
        ref = oracle.gauss_newton(p, p.truth, mode)
        d = np.sqrt(np.diag(ref))
        assert np.all(np.abs(H - ref) <= 1e-12 * np.outer(d, d) + 1e-300)


def test_matrix_scratch_is_given_back_within_a_budget(musr_lib):
    """The smallest memory budget that holds the products of a matrix and then a batch holds the matrix and
    then the batch too: the one-pass kernel's rows do not stay in the batch's way."""
    from paper_1509_07685_gb300 import binding as B
    p = mi.cfg2(nhist=8, nbins=6000, bin_width_ns=2.0, seed=5, n0=60.0)
    X, eye = mi.jitter(p.truth, 1000, seed=5, lo=0.98, hi=1.02), np.eye(p.nparams)

    def runs(budget, matrix):
        try:
            with B.Context(p, hbm_budget_bytes=budget) as ctx:
                matrix(ctx)
                return ctx.eval_batch(X, 1, B.MUSR_FP64)
        except B.MusrError as e:
            assert e.status == B.MUSR_ENOMEM
            return None

    products = lambda ctx: ctx.gn_product(p.truth, eye, 1, B.MUSR_FP64)
    lo, hi = 1 << 16, 1 << 28
    assert runs(hi, products)
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if runs(mid, products) else (mid, hi)
    got = runs(hi, lambda ctx: ctx.gauss_newton(p.truth, 1, B.MUSR_FP64))
    assert got
    for i in (0, 999):
        ref = oracle.cost(p, X[i], 1)
        assert abs(got[0][i] - ref[0]) <= 1e-12 * abs(ref[0])
        assert np.all(np.abs(got[1][i] - ref[1]) <= 1e-12 * ref[2] + 1e-300)


@pytest.mark.parametrize("top", [150.0, 160.0, 200.0, 290.0])
def test_weights_of_a_model_that_grows_beyond_its_square(musr_lib, top):
    """N from 1 to 10^top within the window: 2 d / N^2 is 0 where N^2 overflows."""
    nbins, dt = 900, 0.02
    rate = -np.log(10.0) * top / (nbins * dt)
    p = mi.Problem(_counts(2, nbins), np.zeros(2), dt * 1000.0, (0.0, nbins * dt),
                   [[("AMP", (2,)), ("EXP", (3,))]], np.array([[0, 1, 2, 3]] * 2, np.int32), np.zeros(1), 4,
                   np.array([30.0, 1.5, 0.4, rate]), ["N0", "Nbkg", "A", "lambda"])
    _check(p, modes=(1,))


def test_matrix_of_an_undefined_cost_is_refused(musr_lib):
    """A model that overflows in bins without a count: the cost is infinite, and the matrix refused as the products
    are."""
    from paper_1509_07685_gb300 import binding as B
    counts = _counts(2, 600)
    counts[:, 300:] = 0.0
    p = mi.Problem(counts, np.zeros(2), 20.0, (0.0, 12.0), [[("AMP", (2,)), ("EXP", (3,))]],
                   np.array([[0, 1, 2, 3]] * 2, np.int32), np.zeros(1), 4, np.array([30.0, 1.5, 0.4, -90.0]),
                   ["N0", "Nbkg", "A", "lambda"])
    with B.Context(p) as ctx:
        assert ctx.eval(p.truth, 1, B.MUSR_FP64)[2] == B.MUSR_ENONFINITE
        assert ctx.gn_product(p.truth, np.eye(4), 1, B.MUSR_FP64)[2] == B.MUSR_ENONFINITE
        with pytest.raises(B.MusrError) as e:
            ctx.gauss_newton(p.truth, 1, B.MUSR_FP64)
        assert e.value.status == B.MUSR_ENONFINITE
