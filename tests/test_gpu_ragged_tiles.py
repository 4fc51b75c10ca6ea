"""The ragged batch's matvec at the edges of its loads: one, eight and nine 128-column groups a
row (a warp with no group, one, and a second behind a prefetch), rows short of a block, and many
small systems beside a large one, against the same systems solved one at a time.

Both solve to 1e-10; their charges agree to 1e-8 (the bar of the batch tests)."""
import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("cells", [
    [(4, 4), (17, 1)],                     # 128 and 136 atoms
    [(16, 8), (43, 3), (4, 4)],            # 1,024, 1,032 and 128
    [(43, 6)] + [(5, 3)] * 9,              # 2,064 beside nine of 120
])
def test_against_single_solves(cells):
    rng = np.random.default_rng(len(cells))
    ctxs, bs, want = [], [], []
    for nx, ny in cells:
        el = wl.two_sheet_electrode(nx, ny)
        c = cpm.Context(el.box, precision=cpm.CPM_PREC_FP32, rcut_dc=2.0, solver_path=1)
        c.cpm_build_E(el.xyz, el.alpha)
        b = el.chi + rng.normal(0.0, 0.3, el.n)
        q, it, rel = c.cpm_solve(b[None], tol=1e-10)
        ctxs.append(c)
        bs.append(b)
        want.append(q[0])
    batch = cpm.Batch(ctxs)
    q, it, rel = batch.solve(np.concatenate(bs), tol=1e-10)
    assert np.all(rel <= 1e-10)
    for k, (a, w) in enumerate(zip(np.split(q, np.cumsum(batch.sizes)[:-1]), want)):
        assert np.linalg.norm(a - w) <= 1e-8 * np.linalg.norm(w), k
    batch.close()
    for c in ctxs:
        c.close()
