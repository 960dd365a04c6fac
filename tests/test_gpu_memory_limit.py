"""A device without the memory for the FP64 form's extra operands (the inverted diagonal tiles,
the packed pieces of the variances): every call still returns its results, by the kernels that
need neither.  The limit is simulated (tests/cuda_shim.c)."""
import numpy as np
import pytest

import shim

pytestmark = pytest.mark.gpu
ORDER, COUNT = 320, 12  # (the solve's wide steps pay from about here on)
CODE = f"""
import numpy as np
import paper_1305_5683_gb300 as P
from spigen import random_spd
pbs = [random_spd({ORDER}, 1.0, i, dominance={ORDER}.0) for i in range({COUNT})]
s = P.Solver.for_problems(pbs, diag_tc_min_pivots=1)
idx = np.arange(0, {ORDER}, 4, dtype=np.int32)
for scale in (1.0, 2.0):
    s.factor(np.concatenate([p.values for p in pbs]) * scale)
    x = s.solve(np.concatenate([p.b for p in pbs])) * scale
    v = s.diag_inverse() * scale
    w = s.diag_inverse(idx) * scale
    g = s.inverse_block(idx) * scale
    assert abs(np.diag(g) / w - 1).max() < 1e-12
    assert abs(w / v[idx] - 1).max() < 1e-12
    assert abs(s.solve(np.concatenate([p.b for p in pbs])) * scale / x - 1).max() < 1e-10
np.savez(OUT, x=x, v=v, g=g)
"""


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1305_5683_gb300 as P
    P.build.build()
    return P


def test_results_under_every_limit(P, tmp_path):
    so = shim.build(tmp_path)
    out = str(tmp_path / "out.npz")
    code = f"OUT = {out!r}\n" + CODE
    _, _, peak = shim.run(so, tmp_path, code)
    ref = dict(np.load(out))
    tiles = 2 * 8 * COUNT * (2 * 128 ** 2 + 64 ** 2)  # the inverses and their transposes
    pieces = COUNT * (3 * 8 + 2 * 8 + 4) * 7 * 4096    # 128 x 16 pieces of the three chunks
    for limit in (peak - 1, peak - pieces // 2, peak - pieces + 1, peak - pieces - tiles // 4,
                  peak - pieces - tiles + 4096):
        _, kernels, used = shim.run(so, tmp_path, code, limit=limit)
        assert used <= limit
        got = dict(np.load(out))
        assert np.abs(got["x"] - ref["x"]).max() <= 1e-12 * np.abs(ref["x"]).max()
        assert np.abs(got["v"] / ref["v"] - 1).max() <= 1e-12
        assert np.abs(got["g"] - ref["g"]).max() <= 1e-12 * np.abs(ref["g"]).max()
    # the last limit leaves room for neither: the tiles go when the variances' workspace needs theirs
    assert not any("k_diag_fx" in k for k in kernels) and any("k_fwd_step" in k for k in kernels)
