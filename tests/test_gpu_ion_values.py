"""An ion coordinate that is NaN or infinite shows in the potential of its frame, in every storage
and screen mode, and nowhere else: b is NaN there, the other frame's b is that of a call without it,
and a solve of the frame breaks down."""
import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("slab", [True, False])
@pytest.mark.parametrize("precision", [cpm.CPM_PREC_FP64, cpm.CPM_PREC_FP32, cpm.CPM_PREC_BF16X6])
@pytest.mark.parametrize("cells,rcut", [((10, 6), 12.0),   # every box edge above 2 r_c
                                        ((3, 2), 12.0),    # a list of whole-box shifts
                                        ((3, 2), 30.0)])   # every image
def test_coordinate_that_is_not_finite(slab, precision, cells, rcut):
    el = wl.two_sheet_electrode(*cells)
    rng = np.random.default_rng(3)
    ions = rng.uniform(0, 1, (2, 150, 3)) * [el.box[0], el.box[1], 20.0] + [0, 0, 5.0]
    q = np.tile([1.0, -1.0], (2, 75))
    ctx = cpm.Context(el.box, precision=precision, rcut_dc=3.0, rcut_real=rcut, slab=slab)
    ctx.cpm_build_E(el.xyz, el.alpha)
    good, _ = ctx.cpm_potential(ions, q, el.chi)
    assert np.isfinite(good).all()
    for axis in range(3):
        for bad in (np.nan, np.inf, -np.inf):
            broken = ions.copy()
            broken[1, 140, axis] = bad
            b, qsol = ctx.cpm_potential(broken, q, el.chi)
            assert np.isnan(b[1]).all(), (axis, bad)
            assert np.array_equal(b[0], good[0]) and np.isfinite(qsol).all()
    with pytest.raises(cpm.CpmError) as ei:
        ctx.cpm_solve(b[1:], tol=1e-8)
    assert ei.value.status == cpm.CPM_EBREAKDOWN
    ctx.close()
