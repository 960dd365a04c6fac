"""Reads and writes beside the library's buffers: every device allocation lies between 64 KB of NaN
patterns (tests/cuda_shim.c).  A value read there turns a result into NaN, a value written there is
found when the buffer is freed; both stay inside memory of the process."""
import pytest

import shim

pytestmark = pytest.mark.gpu
START = """
import numpy as np
import paper_1305_5683_gb300 as P
from spigen import BAND, SCALE, generate, generate_bands, random_spd, scaled, sky_scaled
def finite(*vs):
    for v in vs:
        assert np.isfinite(v).all()
"""
CALLS = {
    # symmetric indefinite: 1x1 and 2x2 pivots, the first of all among the 1x1 ones (its -1 is no partner)
    "pivoting": """
import test_gpu_pivoting as T
for A in (T.indefinite(20, 4, 0.3), T.indefinite(150, 5, 0.04), T.indefinite(600, 6, 0.01), T.kkt(120, 40, 2)):
    n, cp, ri, va = T.lower(A)
    s = P.Solver(n, cp, ri, pivoting=True)
    s.factor(va)
    x, v = s.solve(np.ones(n)), s.diag_inverse()
    finite(x, v)
    ref = np.diag(np.linalg.inv(A))
    assert abs(v - ref).max() <= 1e-8 * abs(ref).max()
    s.close()
""",
    "fp64": """
for pb in (generate(scaled(SCALE, 700, seed=3)), random_spd(300, 1.0, 1, dominance=300.0)):
    for kw in (dict(), dict(dag=1, diag_tc_min_pivots=1), dict(dag=2, force_schur=1, diag_tc_min_pivots=-1),
               dict(diag_unpruned=True)):
        s = P.Solver.for_problem(pb, **kw)
        s.factor(pb.values)
        finite(s.solve(pb.b), s.diag_inverse(), s.inverse_block(np.arange(0, 100, 3, dtype=np.int32)))
        finite(s.inverse_entries(np.arange(9, dtype=np.int32), np.arange(9, dtype=np.int32)[::-1].copy()))
        s.close()
""",
    "mixed": """
for pb in (generate(scaled(SCALE, 700, seed=3)), generate(sky_scaled(600, 3.0, 12))):
    for kw in (dict(), dict(dag=1, diag_tc_min_pivots=1), dict(dag=2)):
        s = P.Solver.for_problem(pb, precision=1, **kw)
        s.factor(pb.values)
        finite(s.solve(pb.b), s.diag_inverse(), s.diag_inverse_refined(np.arange(40, dtype=np.int32)))
        s.close()
""",
    "batches": """
bands = generate_bands(scaled(BAND, 400, seed=4), 3)
for precision in (0, 1):
    s = P.Solver(bands.n, bands.colptr, bands.rowind, batch=3, precision=precision)
    s.factor_batch(bands.values)
    finite(s.solve_batch(bands.b), s.diag_inverse_batch())
    s.close()
pbs = [random_spd(m, 0.3, m) for m in (1, 8, 60, 130)]
s = P.Solver.for_problems(pbs, diag_tc_min_pivots=1)
s.factor(np.concatenate([p.values for p in pbs]))
finite(s.solve(np.concatenate([p.b for p in pbs])), s.diag_inverse())
s.close()
pb = generate(scaled(SCALE, 300, seed=3), sparse_design=True)
s = P.Solver.for_problem(pb).normal_setup(pb.H)
nv, b = s.normal_assemble(pb.H.data, pb.w, pb.y)
finite(nv, b)
finite(*s.normal_update(np.arange(50, dtype=np.int32), pb.H.data, pb.w, pb.y, nv, b))
s.close()
""",
}


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1305_5683_gb300 as P
    P.build.build()
    return P


@pytest.mark.parametrize("calls", list(CALLS))
def test_buffers_keep_to_themselves(P, tmp_path, calls):
    _, log, _ = shim.run(shim.build(tmp_path), tmp_path, START + CALLS[calls], redzone=65536)
    assert len(log) == 1 and int(log[0].split()[1]) > 100, log
