"""FP64 Schur complements on the tensor cores (128 x 32 tiles, 32 pivots at a time) through
factor + solve of a dense leaf block over a dense root (the second leaf of two_leaves is merged into
the root by the default amalgamation) and of a three-level tree of seven fronts, at the edges of the
tiles and pivot chunks, against the oracle and the SIMT kernel.  Bound: 64 n 2^-53 for x of a
diagonally dominant matrix, n rounding errors of a few units each way; and, tighter, errors and
residuals against extended precision next to the SIMT kernel's own."""
import dataclasses

import numpy as np
import pytest
import scipy.sparse as sp

import exact
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


def two_leaves(k, r, seed):
    """Columns 0..k and k..2k coupled to the last r only."""
    n = 2 * k + r
    pb = random_spd(n, 1.0, seed, dominance=float(n))
    a = sp.csc_matrix((pb.values, pb.rowind, pb.colptr), shape=(n, n)).toarray()
    a[k:2 * k, :k] = 0.0
    a[np.diag_indices(n)] = np.abs(a + np.tril(a, -1).T).sum(axis=0)
    low = sp.csc_matrix(np.tril(a))
    low.sort_indices()
    return dataclasses.replace(pb, colptr=low.indptr.astype(np.int64), rowind=low.indices.astype(np.int32),
                               values=low.data.astype(np.float64))


@pytest.mark.parametrize("r", [64, 65, 96, 97, 127, 128, 129, 160, 257])
@pytest.mark.parametrize("k", [4, 15, 16, 17, 32, 33, 48, 65])
def test_two_leaves(P, k, r):
    pb = two_leaves(k, r, 100 * k + r)
    ref = oracle.OracleFactor.from_problem(pb).solve(pb.b)
    for scale in (1.0, 1e-280, 1e280):
        xs = []
        for form in (dict(dag=1), dict(dag=1, force_schur=1)):
            s = P.Solver.for_problem(pb, **form)
            s.factor(pb.values * scale)
            xs.append(s.solve(pb.b) * scale)
        tol = 64 * pb.n * EPS * np.abs(ref).max()
        assert np.abs(xs[0] - ref).max() <= tol and np.abs(xs[0] - xs[1]).max() <= tol


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_nonfinite_entries_are_reported(P, value):
    """A NaN or infinity in a leaf's rows reaches the root's pivots, as in the SIMT kernel."""
    pb = two_leaves(32, 128, 5)
    v = pb.values.copy()
    v[pb.colptr[3] + 40] = value  # row below the leaf's pivots
    for form in (dict(dag=1), dict(dag=1, force_schur=1)):
        s = P.Solver.for_problem(pb, **form)
        with pytest.raises(P.SpiError) as e:
            s.factor(v)
        assert e.value.code == 3


def test_badly_scaled_columns(P):
    """Rows and columns scaled by powers of two up to 2^+-40: x unscaled as before."""
    pb = two_leaves(40, 200, 9)
    ref = oracle.OracleFactor.from_problem(pb).solve(pb.b)
    t = 2.0 ** np.random.default_rng(1).integers(-40, 41, pb.n)
    col = np.repeat(np.arange(pb.n), np.diff(pb.colptr))
    s = P.Solver.for_problem(pb, dag=1)
    s.factor(pb.values * t[pb.rowind] * t[col])
    x = s.solve(pb.b * t) * t
    assert np.abs(x - ref).max() <= 64 * pb.n * EPS * np.abs(ref).max()


@pytest.mark.parametrize("kind", ["schur", "panel"])
def test_wait_timeout_reported(P, kind):
    """wait_limit < 0: the first wait for the products gives up; the kernel drains them, frees its
    tensor memory and spi_factor returns SPI_ERR_TIMEOUT; a new context on the device works.
    Without tensor-core launches nothing waits."""
    pb = two_leaves(32, 128, 5) if kind == "schur" else random_spd(300, 1.0, 3, dominance=300.0)
    s = P.Solver.for_problem(pb, dag=1, force_panel=1, wait_limit=-1)
    with pytest.raises(P.SpiError) as e:
        s.factor(pb.values)
    assert e.value.code == 6
    with pytest.raises(P.SpiError) as e:
        s.solve(pb.b)
    assert e.value.code == 7
    ref = oracle.OracleFactor.from_problem(pb).solve(pb.b)
    for kw in (dict(force_schur=1, wait_limit=-1), dict()):
        s = P.Solver.for_problem(pb, dag=1, force_panel=1, **kw)
        s.factor(pb.values)
        assert np.abs(s.solve(pb.b) - ref).max() <= 64 * pb.n * EPS * np.abs(ref).max()


def three_levels(leaf, k, kept, seed):
    """Four leaves of `leaf` columns under two middle blocks of k columns under a root of 1.4 `kept`:
    natural order A1 A2 M1 A3 A4 M2 R; every block is dense, a leaf meets its middle block, and both
    meet the same `kept` columns of the root (their family's own), so that the row maps skip rows."""
    rng = np.random.default_rng(seed)
    r = kept + (2 * kept) // 5
    sizes = [leaf, leaf, k, leaf, leaf, k, r]
    at = np.concatenate([[0], np.cumsum(sizes)])
    n = int(at[-1])
    on = np.zeros((n, n), bool)
    for i, up in enumerate([2, 2, 2, 5, 5, 5, 6]):
        own = slice(at[i], at[i + 1])
        on[own, own] = True
        on[at[up]:at[up + 1], own] = True
    for family in ((0, 1, 2), (3, 4, 5)):
        rows = at[6] + np.r_[0, 1 + np.sort(rng.permutation(r - 1)[:kept - 1])]  # (one root: all meet its first)
        for i in family:
            on[rows[:, None], np.arange(at[i], at[i + 1])] = True
    on = np.tril(on)
    a = np.tril(np.where(on, rng.uniform(-1.0, 1.0, (n, n)), 0.0), -1)
    a = a + a.T
    a[np.diag_indices(n)] = 0.3 * np.abs(a).sum(axis=0) + np.sqrt(n)  # coupled well, still positive definite
    return exact.problem(a, on), a


# a middle block's pivots around one and two chunks of 128 and its rows below around the tiles'
# 32 and 128 (64: the fewest that take the tensor cores); the last: enough work for several chunks
# of pivots per CTA
@pytest.mark.parametrize("leaf,k,kept", [(5, 127, 64), (33, 128, 97), (40, 129, 128), (64, 257, 129), (130, 40, 257),
                                         (150, 520, 800)])
def test_children_siblings_and_chunks(P, leaf, k, kept):
    """Fronts with children below (their sums in the update area), a parent that has an update area,
    and siblings: x and variances against the oracle and the SIMT kernels, x by its residual too."""
    pb, a = three_levels(leaf, k, kept, leaf + k + kept)
    xs, vs, work = [], [], []
    for more in ({}, {"force_schur": 1}):
        s = P.Solver.for_problem(pb, ordering=1, relax=0, dag=1, **more)
        assert s.info()["n_supernodes"] == 7 and s.info()["n_levels"] == 3
        s.factor(pb.values)
        xs.append(s.solve(pb.b)), vs.append(s.diag_inverse()), work.append(s.info()["factor_work_flops"])
    # the tensor-core launches took the six fronts' Schur complements: 32 x 32 tiles of 2 32^2 k flops
    gone = sum(2 * 2.0 * 32 ** 2 * t * (t + 1) / 2 * (c * p) for t, c, p in
               (((k + kept) // 32, 2, leaf), (kept // 32, 1, k)))
    assert work[1] - work[0] >= gone > 0
    f = oracle.OracleFactor.from_problem(pb)
    ref = f.solve(pb.b)
    tol = 64 * pb.n * EPS
    assert np.abs(xs[0] - ref).max() <= tol * np.abs(ref).max() and np.abs(xs[0] - xs[1]).max() <= tol * np.abs(ref).max()
    assert np.abs(vs[0] / vs[1] - 1).max() <= tol and np.abs(vs[0] / f.inv_diag() - 1).max() <= tol
    be = [exact.backward_error(a, x, pb.b) for x in xs]
    assert be[0] <= 4 * max(be[1], EPS / 4)


@pytest.mark.parametrize("dominance", [0.1, 10.0, 300.0])
def test_accuracy_is_that_of_the_fp64_pipe(P, dominance):
    """One front of 300 pivots (two rank-128 updates): the root mean square error of the variances
    against extended precision at most twice that of the SIMT factorization (an emulation gives
    1.0 times; with six digits instead of seven 30 to 190 times)."""
    pb = random_spd(300, 1.0, 3, dominance=dominance)
    ref = np.diag(exact.inverse(exact.dense(pb)))
    rms = []
    for more in ({}, {"force_schur": 1}):
        s = P.Solver.for_problem(pb, dag=1, force_panel=1, **more)
        s.factor(pb.values)
        rms.append(float(np.sqrt(np.mean((s.diag_inverse() / ref - 1) ** 2))))
    assert rms[0] <= 2 * max(rms[1], EPS)
