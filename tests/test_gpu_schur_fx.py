"""FP64 Schur complements on the tensor cores (128 x 32 tiles, 32 pivots at a time) through
factor + solve of two dense leaf blocks over a dense root, at the edges of the tiles and
pivot chunks, against the oracle and the SIMT kernel.  Bound: 64 n 2^-53 for x of a
diagonally dominant matrix, n rounding errors of a few units each way."""
import dataclasses

import numpy as np
import pytest
import scipy.sparse as sp

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
