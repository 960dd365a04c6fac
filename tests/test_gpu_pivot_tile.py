"""The 32 x 32 FP64 pivot tile, the 32-row panel solve and fronts with a diagonal pivot
block, through factor + solve of one dense front (every width of the last tile, rows below
it or not) in each form of the factorization, against the oracle.  Bound: 64 n 2^-53 for
x of a matrix with a unit-scale spectrum (dominance n), n rounding errors of a few units
each way."""
import numpy as np
import pytest

import oracle
from spigen import random_spd

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1305_5683_gb300 as P
    P.build.build()
    return P


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 32, 33, 34, 35, 48, 63, 64, 65, 97, 130])
@pytest.mark.parametrize("form", [dict(force_panel=1, dag=1), dict(force_panel=2, dag=1), dict(dag=2),
                                  dict(force_panel=1, dag=2)])
def test_dense_front_every_form(P, n, form):
    pb = random_spd(n, 1.0, n + 7, dominance=float(n))
    ref = oracle.OracleFactor.from_problem(pb).solve(pb.b)
    for precision, tol in ((0, 64 * max(n, 16) * EPS), (1, 1e-8)):
        s = P.Solver.for_problem(pb, precision=precision, **form)
        s.factor(pb.values)
        assert np.abs(s.solve(pb.b) - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("scale", [1e-290, 1e-30, 1.0, 1e30, 1e290])
def test_pivot_reciprocals_over_the_exponent_range(P, scale):
    """Pivots near both ends of the exponent range."""
    pb = random_spd(40, 1.0, 3, dominance=40.0)
    ref = oracle.OracleFactor.from_problem(pb).solve(pb.b)
    s = P.Solver.for_problem(pb)
    s.factor(pb.values * scale)
    x = s.solve(pb.b) * scale
    assert np.abs(x - ref).max() <= 64 * 40 * EPS * np.abs(ref).max()


@pytest.mark.parametrize("bad", [0, 5, 31, 32, 39])
def test_bad_pivot_is_reported(P, bad):
    pb = random_spd(40, 1.0, 3, dominance=40.0)
    v = pb.values.copy()
    v[pb.colptr[bad]] = -1.0
    for form in (dict(force_panel=1, dag=1), dict(force_panel=2, dag=1), dict(dag=2)):
        s = P.Solver.for_problem(pb, ordering=1, **form)
        with pytest.raises(P.SpiError) as e:
            s.factor(v)
        assert e.value.code == 3 and s.info()["bad_pivot"] == bad


def ulps(a, b):
    """a - b in units in the last place of b (positive normal numbers)."""
    return a.view(np.int64) - b.view(np.int64)


def wide_range(count, seed):
    """Random significands over every normal exponent, both ends included."""
    rng = np.random.default_rng(seed)
    e = np.concatenate([np.arange(-1022, -1010), np.arange(1010, 1024), rng.integers(-1022, 1024, count)])
    return np.ldexp(1.0 + rng.random(len(e)), e)


def chain_problem(d, w, at):
    """Per entry of d a dense front of order w + 1: pivots 1 but d at position `at`, coupled by a
    power of two t to the last row alone (explicit zeros elsewhere), whose pivot stays 2^90.
    With b = e_at the last x is -l / 2^90, l = t (1 / d)."""
    import dataclasses
    n, rows = (w + 1) * len(d), []
    t = np.ldexp(1.0, np.frexp(d)[1] // 2)
    low = np.tril(np.ones((w + 1, w + 1), bool))
    r, c = np.nonzero(low.T)[1], np.nonzero(low.T)[0]   # column by column
    base = (w + 1) * np.arange(len(d))
    vals = np.zeros((len(d), len(r)))
    vals[:, r == c] = 1.0
    vals[:, (r == at) & (c == at)] = d[:, None]
    vals[:, (r == w) & (c == at)] = t[:, None]
    vals[:, (r == w) & (c == w)] = 2.0 ** 90
    colptr = np.concatenate([[0], np.cumsum(np.tile(np.arange(w + 1, 0, -1), len(d)))]).astype(np.int64)
    pb = dataclasses.replace(random_spd(2, 0.0, 1), n=n, colptr=colptr,
                             rowind=(base[:, None] + r).astype(np.int32).ravel(), values=vals.ravel())
    b = np.zeros(n)
    b[base + at] = 1.0
    return pb, b, base + w, t


@pytest.mark.parametrize("at,w", [(0, 1), (13, 31), (31, 32), (5, 34)])
@pytest.mark.parametrize("form,bound", [(dict(force_panel=1, dag=1), 1), (dict(force_panel=2, dag=1), 0), (dict(dag=2), 0),
                                        (dict(force_panel=1, dag=2), 0)])
def test_pivot_reciprocals(P, form, bound, at, w):
    """The reciprocals themselves, read out through x, over every exponent: within the pivot tile
    (the last row is one of its 32) at most one unit in the last place from the rounded 1 / d; in
    the panel solve below it correctly rounded, except on the block-step chain (at most one)."""
    d = wide_range(3000 if w == 1 else 300, w)
    pb, b, last, t = chain_problem(d, w, at)
    s = P.Solver.for_problem(pb, ordering=1, relax=0, **form)
    s.factor(pb.values)
    r = -s.solve(b)[last] * 2.0 ** 90 / t
    off = ulps(r, 1.0 / d)[1.0 / d >= 2.0 ** -1022]
    assert np.abs(off).max() <= (1 if w < 32 else bound)
