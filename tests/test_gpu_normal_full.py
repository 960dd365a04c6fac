"""The whole product N = H^T W H, b = H^T W y on the device over the shapes of its row groups
(rows x columns of a group: one row, few, a full group; pairs at and around the CTA's 256
threads), against a dense FP64 product.  Bound: a sum of R terms and one addition per
group into an entry, (rows + groups) 2^-53 of the sum of magnitudes."""
import numpy as np
import pytest
import scipy.sparse as sp

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


@pytest.mark.parametrize("rows", [1, 2, 3, 31, 32, 33, 70])
@pytest.mark.parametrize("c", [1, 2, 21, 22, 23, 32, 33, 63, 256, 300])
def test_group_shapes(P, rows, c):
    rng = np.random.default_rng(1000 * rows + c)
    n = 310
    pb = random_spd(n, 1.0, 3, dominance=float(n))  # the full lower pattern
    H = np.zeros((rows + 3, n))
    cols = np.sort(rng.choice(n, c, replace=False))
    H[:rows, cols] = rng.standard_normal((rows, c))
    H[0, cols[0]] = 0.0                     # a ragged first row
    H[rows + 1, ::2] = rng.standard_normal(n // 2)  # after an empty row, one on its own
    H = sp.csr_matrix(H)
    w = rng.uniform(-1.0, 2.0, rows + 3)
    y = rng.standard_normal(rows + 3)
    s = P.Solver.for_problem(pb).normal_setup(H)
    nv, b = s.normal_assemble(H.data, w, y)
    D = H.toarray()
    ref, mag = D.T @ (w[:, None] * D), abs(D).T @ (abs(w)[:, None] * abs(D))
    colj = np.repeat(np.arange(n), np.diff(pb.colptr))
    tol = (2 * rows + 8) * EPS
    assert (np.abs(nv - ref[pb.rowind, colj]) <= tol * mag[pb.rowind, colj]).all()
    assert (np.abs(b - D.T @ (w * y)) <= tol * (abs(D).T @ abs(w * y))).all()


def test_term_without_a_place_is_reported(P):
    n = 40
    pb = random_spd(n, 1.0, 3, dominance=float(n))
    low = sp.csc_matrix(np.eye(n))
    pb.colptr, pb.rowind, pb.values = low.indptr.astype(np.int64), low.indices.astype(np.int32), low.data
    for rows in (1, 2):  # in place, and as a dense group
        H = sp.csr_matrix(np.pad(np.ones((rows, 2)), ((0, 0), (3, n - 5))))
        s = P.Solver.for_problem(pb).normal_setup(H)
        with pytest.raises(P.SpiError):
            s.normal_assemble(H.data, np.ones(rows), np.ones(rows))
