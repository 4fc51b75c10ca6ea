"""A batch gives back what it holds: a thousand batches made, solved and destroyed leave the
process as large as it was.  One that keeps its page of pinned host memory leaves 4 KB each, 4 MB;
the bar is half of that."""
import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _resident_kb():
    with open("/proc/self/status") as f:
        return next(int(line.split()[1]) for line in f if line.startswith("VmRSS"))


def test_batches_leave_nothing():
    ctxs, n = [], 0
    for cells in ((3, 2), (5, 3)):
        el = wl.two_sheet_electrode(*cells)
        ctxs.append(cpm.Context(el.box, precision=cpm.CPM_PREC_FP32, rcut_dc=3.0))
        ctxs[-1].cpm_build_E(el.xyz, el.alpha)
        n += el.n
    b = np.random.default_rng(0).normal(size=n)

    def batches(count):
        for _ in range(count):
            batch = cpm.Batch(ctxs)
            batch.solve(b, tol=1e-8)
            batch.close()

    batches(100)  # what the first ones leave with the driver and the allocators
    before = _resident_kb()
    batches(1000)
    assert _resident_kb() - before < 2048
    for ctx in ctxs:
        ctx.close()
