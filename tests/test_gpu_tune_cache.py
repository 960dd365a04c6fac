"""What the autotuner's file may decide: its choices hold for the library's present kernels and
for problems of about the size they were timed on; and the candidates timed are what would run."""
import pytest

import shim
from spigen import SCALE, generate, scaled

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1305_5683_gb300 as P
    P.build.build()
    return P


def timed(P, cache, points):
    """Whether a context's factor and solve forms were timed (rather than read)."""
    pb = generate(scaled(SCALE, points, seed=3))
    s = P.Solver.for_problem(pb, autotune=1, tune_cache=str(cache))
    s.factor(pb.values)
    s.solve(pb.b)
    i = s.info()
    return i["tune_ms_launches"] > 0, i["tune_solve_ms_launches"] > 0


def test_forms_of_older_kernels_and_other_sizes_are_not_taken(P, tmp_path):
    import torch
    cache = tmp_path / "tune.txt"
    dev = torch.cuda.get_device_name(0).replace(" ", "_")
    old = [f"{dev} fp64 single {kind} 0 1 9.0 1.0" for kind in "DV"]  # a file of the first kernels
    cache.write_text("\n".join(old) + "\n")
    assert timed(P, cache, 400) == (True, True)
    assert timed(P, cache, 400) == (False, False)
    assert timed(P, cache, 2500) == (True, True)
    assert timed(P, cache, 2500) == (False, False)
    assert timed(P, cache, 400) == (False, False)  # the other size's lines are still there
    text = cache.read_text()
    assert all(l in text for l in old)


def test_block_step_candidate_is_timed_with_its_own_kernels(P, tmp_path):
    """FP64 panels of more than 128 pivots on the block-step chain take the tensor-core rank-128
    updates; the autotuner's candidate has to contain them (with dag = 2 nothing else does)."""
    code = """
import paper_1305_5683_gb300 as P
from spigen import random_spd
pb = random_spd(400, 1.0, 1, dominance=400.0)
P.Solver.for_problem(pb, autotune=1, dag=2).factor(pb.values)
"""
    _, kernels, _ = shim.run(shim.build(tmp_path), tmp_path, code)
    assert any("k_front_panel" in k for k in kernels) and any("k_schur_fxILi1E" in k for k in kernels)
