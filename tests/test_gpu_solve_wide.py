"""The FP64 solve in 64-column steps through the inverted diagonal tiles (launch kinds 15
and 16), against the oracle, at the edges of a step, of a 128-column tile and of the 64
rows or columns a CTA takes.  Bound: x of a well-conditioned matrix (random_spd with a
unit shift) to 64 n 2^-53, n rounding errors of a few units each way; the SPI members to
the 1e-10 of the parity tests."""
import numpy as np
import pytest

import exact
import oracle
import shim
from spigen import SCALE, BAND, generate, generate_bands, random_spd, scaled

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


@pytest.mark.parametrize("n", [1, 2, 31, 63, 64, 65, 127, 128, 129, 191, 193, 256, 257, 330])
def test_one_dense_front(P, n):
    pb = random_spd(n, 1.0, n, dominance=float(n))
    s = P.Solver.for_problem(pb, dag=1)
    s.factor(pb.values)
    x, ref = s.solve(pb.b), oracle.OracleFactor.from_problem(pb).solve(pb.b)
    assert np.abs(x - ref).max() <= 64 * max(n, 16) * EPS * np.abs(ref).max()


@pytest.mark.parametrize("points", [300, 1501, 2600])
@pytest.mark.parametrize("precision", [0, 1])
def test_spi_members_repeat_and_alias(P, points, precision):
    """Several solves on one factor, a new factorization, and x aliasing b."""
    pb = generate(scaled(SCALE, points, seed=points))
    f = oracle.OracleFactor.from_problem(pb)
    s = P.Solver.for_problem(pb, precision=precision, dag=1)
    tol = 1e-10 if precision == 0 else 1e-8
    rng = np.random.default_rng(points)
    for scale in (1.0, 1.0, 3.0):
        s.factor(pb.values * scale)
        for _ in range(2):
            b = rng.standard_normal(pb.n)
            ref = f.solve(b) / scale
            assert np.abs(s.solve(b) - ref).max() <= tol * np.abs(ref).max()
            x = b.copy()
            s.solve(x, x)
            assert np.abs(x - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("precision", [0, 1])
def test_bands_with_fused_and_stepped_levels(P, precision):
    bands = generate_bands(scaled(BAND, 900, seed=4), 3)
    s = P.Solver(bands.n, bands.colptr, bands.rowind, batch=3, precision=precision, dag=1)
    s.factor_batch(bands.values)
    x = s.solve_batch(bands.b).reshape(3, -1)
    for k in range(3):
        pb = bands.band(k)
        ref = oracle.OracleFactor.from_problem(pb).solve(pb.b)
        assert np.abs(x[k] - ref).max() <= (1e-10 if precision == 0 else 1e-8) * np.abs(ref).max()


def ill_conditioned(kind, c, n):
    """Matrices whose diagonal blocks have large inverses: a Gaussian kernel plus a diagonal of
    10^-c, and the square of a second difference plus 10^-c."""
    if kind == "kernel":
        t = np.linspace(0.0, 1.0, n)
        return np.exp(-((t[:, None] - t) / 0.1) ** 2) + 10.0 ** -c * np.eye(n)
    a = 2.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1)
    return a @ a + 10.0 ** -c * np.eye(n)


def beside_a_chain(pb):
    """The forest of pb and a front of 400 columns, whose many steps make the factorization prepare
    the wide steps of every supernode (alone, a small pb may be solved in 32-column steps)."""
    return [pb, random_spd(400, 1.0, 7, dominance=400.0)]


@pytest.mark.parametrize("n", [1, 2, 31, 63, 64, 65, 127, 128, 129, 191, 193, 256, 257, 330])
def test_wide_steps_of_every_width(P, n):
    probs = beside_a_chain(random_spd(n, 1.0, n, dominance=float(n)))
    s = P.Solver.for_problems(probs, dag=1)
    s.factor(np.concatenate([p.values for p in probs]))
    x = s.solve(np.concatenate([p.b for p in probs]))[:n]
    ref = oracle.OracleFactor.from_problem(probs[0]).solve(probs[0].b)
    assert np.abs(x - ref).max() <= 64 * max(n, 16) * EPS * np.abs(ref).max()


@pytest.mark.parametrize("n", [40, 64, 65, 130, 200])
@pytest.mark.parametrize("kind,c", [("kernel", 4), ("kernel", 8), ("kernel", 11), ("difference", 4), ("difference", 9)])
def test_ill_conditioned_front(P, kind, c, n):
    """The steps' inverted blocks leave no larger residual than substitution (the
    dependency-driven form, dag = 2), whatever the blocks' condition: a backward error within
    n 2^-53, and within four times substitution's or the unit roundoff."""
    a = ill_conditioned(kind, c, n)
    probs = beside_a_chain(exact.problem(a))
    values, rest = np.concatenate([p.values for p in probs]), probs[1].b
    rng = np.random.default_rng(n + c)
    err = {1: [], 2: []}
    for _ in range(3):
        b = a @ rng.standard_normal(n)
        for dag in err:
            s = P.Solver.for_problems(probs, dag=dag)
            s.factor(values)
            err[dag].append(exact.backward_error(a, s.solve(np.concatenate([b, rest]))[:n], b))
    assert max(err[1]) <= n * EPS
    assert np.median(err[1]) <= 4 * max(np.median(err[2]), EPS)


def test_inverses_are_made_where_they_pay(P, tmp_path):
    """The factorization inverts the diagonal tiles for a long chain of steps, and not for many small
    fronts, whose solve they shorten by less than they take; there the tensor-core variances, when
    asked for, make their own.  Both against the SIMT kernel and the oracle's x."""
    code = """
import numpy as np
import paper_1305_5683_gb300 as P
from spigen import random_spd
pbs = [random_spd({n}, 1.0, i, dominance={n}.0) for i in range({count})]
s = P.Solver.for_problems(pbs, dag=1, diag_tc_min_pivots=1)
s.factor(np.concatenate([p.values for p in pbs]))
x = s.solve(np.concatenate([p.b for p in pbs]))
if {variances}:
    v = [s.diag_inverse(), s.diag_inverse(np.arange(5, dtype=np.int32))]
    r = P.Solver.for_problems(pbs, diag_tc_min_pivots=-1)
    r.factor(np.concatenate([p.values for p in pbs]))
    w = r.diag_inverse()
    assert abs(v[0] / w - 1).max() < 1e-12 and abs(v[1] / w[:5] - 1).max() < 1e-12
    assert s.info()["launches_diag"] == {launches}
np.save({out!r}, x)
"""
    so, out = shim.build(tmp_path), str(tmp_path / "x.npy")
    for n, count, variances, launches, made in ((400, 1, False, 0, True), (400, 1, True, 2, True), (60, 100, False, 0, False),
                                                (60, 100, True, 3, True)):
        _, kernels, _ = shim.run(so, tmp_path, code.format(n=n, count=count, variances=variances, launches=launches, out=out))
        assert any("k_fx_tinv" in k for k in kernels) == made
        assert any("k_fwd_wide64" in k for k in kernels) == (n == 400)
        x = np.load(out)[:n]
        pb = random_spd(n, 1.0, 0, dominance=float(n))
        assert np.abs(x - oracle.OracleFactor.from_problem(pb).solve(pb.b)).max() <= 64 * n * EPS * np.abs(x).max()


@pytest.mark.parametrize("n,count", [(33, 33), (160, 40), (161, 2), (544, 32), (545, 33), (700, 65)])
def test_many_right_hand_sides_of_one_factor(P, n, count):
    """The unpruned variances' full solves, 32 at a time: rows below a step at the edges of 128 and
    512, a last pass of one right-hand side."""
    pb = random_spd(n, 1.0, n, dominance=float(n))
    s = P.Solver.for_problem(pb, diag_unpruned=True)
    s.factor(pb.values)
    idx = np.random.default_rng(n).permutation(n)[:count].astype(np.int32)
    ref = oracle.OracleFactor.from_problem(pb).inv_diag(idx)
    assert np.abs(s.diag_inverse(idx) / ref - 1).max() <= 64 * n * EPS
