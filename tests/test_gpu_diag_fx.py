"""The FP64 form's variances on the tensor cores (exact integer pieces, diag_fx.cu)
against the SIMT kernel on the same factor (diag_tc_min_pivots = -1) and the oracle.

Bound: both kernels compute z = L^-1 e with a backward error of a few units in the
last place per multiply-add, at most n of them on a path, so two of them differ by
at most about n 2^-53 times the condition of the (scaled) triangles; 64 n 2^-53 leaves
a factor 64 for that condition and the two operands' fixed-point grids (2^-56 of
their largest entries).  Tighter: the errors against extended precision next to the SIMT
kernel's own."""
import numpy as np
import pytest

import exact
import oracle
from spigen import SCALE, BAND, generate, generate_bands, random_spd, scaled, sky_scaled

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


def both(P, pb, values=None, idx=None, **kw):
    """(tensor cores, SIMT) variances of one problem, whichever the rule would choose."""
    out = []
    for more in (dict(kw, diag_tc_min_pivots=1), {"diag_tc_min_pivots": -1}):
        s = P.Solver.for_problem(pb, **more)
        s.factor(pb.values if values is None else values)
        out.append(s.diag_inverse(idx))
    return out


def rel(a, b):
    return float((np.abs(a - b) / b).max())


# one dense front of order n: tiles, pieces and row groups just below, at and above their
# edges, a single column, several 128-column chunks with a ragged last one
@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 31, 33, 127, 128, 129, 144, 255, 257, 400])
@pytest.mark.parametrize("block", [16, 64])
def test_dense_front_edges(P, n, block):
    pb = random_spd(n, 1.0, n, dominance=0.1)
    fx, simt = both(P, pb, rhs_block=block)
    assert rel(fx, oracle.OracleFactor.from_problem(pb).inv_diag()) <= 64 * max(n, 16) * EPS
    assert rel(fx, simt) <= 64 * max(n, 16) * EPS


@pytest.mark.parametrize("block", [16, 32, 64])
def test_spi_problem_blocks(P, block):
    pb = generate(scaled(SCALE, 2003, seed=5))
    fx, simt = both(P, pb, rhs_block=block)
    assert rel(fx, simt) <= 64 * 600 * EPS  # paths of at most 600 columns
    ref = oracle.OracleFactor.from_problem(pb).inv_diag()
    assert rel(fx, ref) <= 1e-10


@pytest.mark.parametrize("count", [1, 16, 17, 333, 2500])
def test_index_subsets(P, count):
    pb = generate(scaled(SCALE, 1500, seed=3))
    idx = np.random.default_rng(count).permutation(pb.n)[:count].astype(np.int32)
    fx, simt = both(P, pb, idx=idx)
    assert rel(fx, simt) <= 64 * 600 * EPS


def test_wide_front_and_repeat(P):
    """A sky front of many chunks; two calls give the same bits (fixed summation order)."""
    pb = generate(sky_scaled(600, 3.0, 12))
    s = P.Solver.for_problem(pb, diag_tc_min_pivots=1)
    s.factor(pb.values)
    a, b = s.diag_inverse(), s.diag_inverse()
    assert np.array_equal(a, b)
    f = oracle.OracleFactor.from_problem(pb)
    assert rel(a, f.inv_diag()) <= 1e-10


def test_badly_scaled_columns(P):
    """N' = S N S with S over 40 powers of ten: the variances are those of N over S^2, as
    closely as the SIMT kernel gives them (the scaling by powers of two keeps the fixed-point grids on
    the entries' own scale)."""
    pb = generate(scaled(SCALE, 1000, seed=7))
    s = 10.0 ** np.random.default_rng(1).uniform(-20, 20, pb.n)
    col = np.repeat(np.arange(pb.n), np.diff(pb.colptr))
    values = pb.values * s[col] * s[pb.rowind]
    fx, simt = both(P, pb, values=values)
    assert rel(fx, simt) <= 64 * 600 * EPS
    ref = oracle.OracleFactor.from_problem(pb).inv_diag() / s ** 2
    assert rel(fx, ref) <= 1e-10


def test_fp64_bands_and_forest(P):
    bands = generate_bands(scaled(BAND, 700, seed=2), 3)
    s = P.Solver(bands.n, bands.colptr, bands.rowind, batch=3, diag_tc_min_pivots=1)
    s.factor_batch(bands.values)
    v = s.diag_inverse_batch().reshape(3, -1)
    for k in range(3):
        assert rel(v[k], oracle.OracleFactor.from_problem(bands.band(k)).inv_diag()) <= 1e-10
    probs = [random_spd(m, 0.2, m) for m in (3, 40, 150)]
    s = P.Solver.for_problems(probs, diag_tc_min_pivots=1)
    s.factor(np.concatenate([p.values for p in probs]))
    v = s.diag_inverse()
    assert rel(v, np.concatenate([oracle.OracleFactor.from_problem(p).inv_diag() for p in probs])) <= 1e-10


@pytest.mark.parametrize("count", [1, 16, 40, 512])
def test_inverse_block_beside_variances(P, count):
    pb = generate(scaled(SCALE, 1200, seed=9))
    idx = np.sort(np.random.default_rng(count).permutation(pb.n)[:count]).astype(np.int32)
    s = P.Solver.for_problem(pb)
    s.factor(pb.values)
    G = s.inverse_block(idx)
    R = oracle.OracleFactor.from_problem(pb).inv_block(idx)
    d = np.sqrt(np.diag(R))
    assert np.abs(G - R).max() <= 1e-10 * np.abs(R).max()
    assert (np.abs(G - R) / np.outer(d, d)).max() <= 64 * 600 * EPS + 1e-10


@pytest.mark.parametrize("weak", [1e-3, 1e-8, 1e-14])
def test_covariances_of_weakly_coupled_unknowns(P, weak):
    """Two groups of unknowns in one front, coupled `weak` times as strongly as within a group: the
    covariances between the groups, `weak` times the variances, keep their own digits."""
    n = 60
    rng = np.random.default_rng(4)
    g = np.arange(n) % 2
    a = rng.uniform(0.5, 1.0, (n, n)) * np.where(g[:, None] == g, 1.0, weak)
    a = np.tril(a, -1)
    a = a + a.T + np.diag(np.full(n, float(n)))
    ref = exact.inverse(a)
    s = P.Solver.for_problem(exact.problem(a))
    s.factor(exact.problem(a).values)
    got = s.inverse_block(np.arange(n, dtype=np.int32))
    err = np.abs(got / ref.astype(float) - 1)
    assert err.max() <= 64 * n * EPS


def test_wait_timeout_reported(P):
    """wait_limit < 0: the kernel's first wait gives up; it drains its copies and products, frees
    its tensor memory, and spi_diag_inverse returns SPI_ERR_TIMEOUT.  (The factorization waits
    nowhere: SIMT Schur complements, launches level by level.)"""
    pb = generate(scaled(SCALE, 700, seed=9))
    s = P.Solver.for_problem(pb, wait_limit=-1, force_schur=1, dag=1, diag_tc_min_pivots=1)
    s.factor(pb.values)
    with pytest.raises(P.SpiError) as e:
        s.diag_inverse()
    assert e.value.code == 6
    s = P.Solver.for_problem(pb)
    s.factor(pb.values)
    assert rel(s.diag_inverse(), oracle.OracleFactor.from_problem(pb).inv_diag()) <= 1e-10


def test_room_for_another_stream(P):
    """diag_ctas_per_sm keeps its promise: the variances then come from the SIMT kernel, whose CTAs
    leave room on every SM (the tensor-core kernel's take one each)."""
    pb = generate(scaled(SCALE, 700, seed=9))
    v = []
    for more in (dict(diag_ctas_per_sm=3), dict(diag_ctas_per_sm=3, diag_tc_min_pivots=-1)):
        s = P.Solver.for_problem(pb, rhs_block=32, **more)
        s.factor(pb.values)
        v.append(s.diag_inverse())
        assert s.info()["launches_diag"] == 1
    # the same kernel on two factorizations (whose atomics may add in another order)
    assert rel(v[0], v[1]) <= 1e-13


@pytest.mark.parametrize("block", [8, 48, 128])
def test_other_block_sizes_hold_no_packed_operands(P, block):
    """Blocks the tensor-core kernel does not take: one SIMT launch and no more device memory than
    with the kernel switched off."""
    pb = generate(scaled(SCALE, 300, seed=2))
    held = []
    for more in ({}, {"diag_tc_min_pivots": -1}):
        s = P.Solver.for_problem(pb, rhs_block=block, **more)
        s.factor(pb.values)
        s.diag_inverse()
        held.append(s.info()["device_bytes"])
        assert s.info()["launches_diag"] == 1
    assert held[0] == held[1]


@pytest.mark.parametrize("dominance", [0.1, 10.0, 300.0])
def test_accuracy_is_that_of_the_fp64_pipe(P, dominance):
    """The root mean square error against extended precision at most twice the SIMT kernel's on the
    same factor (an emulation gives 1.0 times; with six digits instead of seven 30 times or more)."""
    pb = random_spd(300, 1.0, 3, dominance=dominance)
    ref = np.diag(exact.inverse(exact.dense(pb)))
    rms = [float(np.sqrt(np.mean((v / ref - 1) ** 2))) for v in both(P, pb)]
    assert rms[0] <= 2 * max(rms[1], EPS)


@pytest.mark.parametrize("c", [3, 6, 9])
@pytest.mark.parametrize("n", [64, 130, 300])
def test_ill_conditioned_front(P, n, c):
    """A Gaussian kernel matrix plus 10^-c on the diagonal: multiplying by the tiles' inverses, the
    variances are off by no more than with substitution (both by the factorization's own error)."""
    t = np.linspace(0.0, 1.0, n)
    a = np.exp(-((t[:, None] - t) / 0.1) ** 2) + 10.0 ** -c * np.eye(n)
    pb = exact.problem(a)
    ref = np.diag(exact.inverse(a))
    err = [float(np.abs(v / ref - 1).max()) for v in both(P, pb)]
    assert err[0] <= 1.5 * err[1] + 64 * n * EPS


def test_narrow_supernodes_stay_on_the_simt_kernel(P):
    """The rule's two sides, and the option over it: many problems of order 8 against one wide front."""
    small = [random_spd(8, 1.0, i, dominance=8.0) for i in range(400)]
    wide = [random_spd(400, 1.0, 1, dominance=400.0)]
    for probs, rule in ((small, 1), (wide, 2)):
        v = {}
        for forced, launches in ((0, rule), (1, 2), (-1, 1)):
            s = P.Solver.for_problems(probs, diag_tc_min_pivots=forced)
            s.factor(np.concatenate([p.values for p in probs]))
            v[forced] = s.diag_inverse()
            assert s.info()["launches_diag"] == launches
        assert rel(v[0], v[-1]) <= 64 * 400 * EPS and rel(v[1], v[-1]) <= 64 * 400 * EPS
