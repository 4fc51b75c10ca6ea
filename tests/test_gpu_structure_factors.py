"""The ions' structure factors at the edges of their blocks of eight and chunks of 256, with
charges that are floats and charges that are not, few and many k-vectors: the potential in
float storage against FP64 storage (its phasors come from other tables and its sums are
plain FP64), 2e-8 of the largest entry as in the parity tests.
"""
import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("cells", [(3, 2), (9, 7)])
@pytest.mark.parametrize("n_ion,frames", [(1, 1), (7, 2), (8, 1), (9, 3), (255, 1), (264, 2),
                                          (601, 1)])
@pytest.mark.parametrize("charges", ["unit", "any"])
def test_block_edges(cells, n_ion, frames, charges):
    el = wl.two_sheet_electrode(*cells)
    rng = np.random.default_rng(n_ion + frames)
    ions = np.stack([np.column_stack([rng.uniform(0, el.box[0], n_ion),
                                      rng.uniform(0, el.box[1], n_ion),
                                      rng.uniform(3.0, 27.0, n_ion)]) for _ in range(frames)])
    q = rng.choice([-1.0, 1.0], size=(frames, n_ion))
    if charges == "any":
        q = q * rng.uniform(0.2, 1.0, q.shape)
    out = {}
    for prec in (cpm.CPM_PREC_FP64, cpm.CPM_PREC_BF16X6, cpm.CPM_PREC_FP32):
        ctx = cpm.Context(el.box, precision=prec, rcut_dc=3.0)
        ctx.cpm_build_E(el.xyz, el.alpha)
        out[prec], _ = ctx.cpm_potential(ions, q, el.chi)
        ctx.close()
    ref = out[cpm.CPM_PREC_FP64]
    for prec in (cpm.CPM_PREC_BF16X6, cpm.CPM_PREC_FP32):
        assert np.abs(out[prec] - ref).max() <= 2e-8 * np.abs(ref).max()
