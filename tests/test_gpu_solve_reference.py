"""Charges against the library's matrix by products that are not its own: torch's FP64 product with
the matrix of cpm_get_E, in FP64 and in float storage, and the two storages against each other.
With E64 q64 = b - r64 and E32 q32 = b - r32, the difference d = q32 - q64 satisfies
E64 d + (E32 - E64) q32 = r64 - r32: at most twice the solve's tolerance."""
import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = 1e-10


@pytest.mark.parametrize("cells,nrhs,path", [((8, 8), 1, 1), ((8, 8), 1, 2), ((11, 9), 4, 1),
                                             ((13, 11), 37, 1)])
def test_both_storages(cells, nrhs, path):
    el = wl.two_sheet_electrode(*cells)
    b = np.random.default_rng(nrhs).normal(size=(nrhs, el.n))
    bt = torch.tensor(b, device="cuda")
    mats, charges = [], []
    for precision in (cpm.CPM_PREC_FP64, cpm.CPM_PREC_BF16X6):
        ctx = cpm.Context(el.box, precision=precision, solver_path=path)
        ctx.cpm_build_E(el.xyz, el.alpha)
        e = torch.tensor(np.asarray(ctx.cpm_get_E(cpm.CPM_E_STORED), dtype=np.float64),
                         device="cuda")
        q = torch.tensor(ctx.cpm_solve(b, tol=TOL, maxit=3000)[0], device="cuda")
        ctx.close()
        r = bt - cpm.KE * (q @ e.T)
        assert (r.norm(dim=1) / bt.norm(dim=1)).max() <= 1.01 * TOL + 1e-12
        mats.append(e)
        charges.append(q)
    d = (charges[1] - charges[0]) @ mats[0].T + charges[1] @ (mats[1] - mats[0]).T
    assert (cpm.KE * d.norm(dim=1) / bt.norm(dim=1)).max() <= 2.02 * TOL + 2e-12
