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
    """Pivots near both ends of the exponent range (the reciprocal's division branch among them)."""
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
