"""The forces' sums split over the grid: ion counts at the edges of the 8-ion and 32-lane
groups, one and several frames, few and many electrode atoms, against the FP64 oracle.

Tolerances: FP64 storage takes the ions' phases from 32-bit fractions of the box (rounded by
up to 1e-8 A here, forces that change on an Angstrom), so 1e-7 of the largest force; float
storage the bar of the other force tests, 1e-6 (phasors of one float ulp, 6e-8, on the tail
k-vectors).
"""
import numpy as np
import pytest

from oracle import forces as fo
from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = {"fp64": 1e-7, "bf16x6": 1e-6}
PREC = {"fp64": cpm.CPM_PREC_FP64, "bf16x6": cpm.CPM_PREC_BF16X6}


@pytest.mark.parametrize("prec", ["fp64", "bf16x6"])
@pytest.mark.parametrize("n_ion,frames,cells", [(1, 1, (3, 2)), (7, 3, (3, 2)), (9, 2, (5, 3)),
                                                (33, 1, (8, 5))])
def test_forces_at_group_edges(prec, n_ion, frames, cells):
    el = wl.two_sheet_electrode(*cells)
    rng = np.random.default_rng(100 * n_ion + frames)
    ions = np.stack([np.column_stack([rng.uniform(0, el.box[0], n_ion),
                                      rng.uniform(0, el.box[1], n_ion),
                                      rng.uniform(2.0, 28.0, n_ion)]) for _ in range(frames)])
    q_ion = rng.choice([-1.0, 1.0, 0.37], size=(frames, n_ion))
    q = rng.normal(0.0, 0.01, (frames, el.n))
    ctx = cpm.Context(el.box, rcut_dc=3.0, precision=PREC[prec])
    ctx.cpm_build_E(el.xyz, el.alpha)
    f = ctx.cpm_ion_forces(ions, q_ion, q)
    for k in range(frames):
        ref = fo.forces_on_ions(el.xyz, el.alpha, q[k], ions[k], q_ion[k], el.box, wl.G_EWALD,
                                wl.RCUT_REAL, wl.KSPACE_EPS, True)
        assert np.abs(f[k] - ref).max() <= TOL[prec] * np.abs(ref).max(), k
    ctx.close()
