"""Calls whose kernels run side by side (real-space sums beside the ions' structure factors):
calls of different sizes in turn on one context give the same bits every time, without ions the
potential is chi, and the kernels' own times are reported.

The order of every sum is fixed, so the repeats are compared exactly."""
import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

PREC = {"fp64": cpm.CPM_PREC_FP64, "bf16x6": cpm.CPM_PREC_BF16X6}


@pytest.mark.parametrize("prec", ["fp64", "bf16x6"])
@pytest.mark.parametrize("cells", [(3, 2), (9, 7)])
def test_calls_in_turn(prec, cells):
    el = wl.two_sheet_electrode(*cells)
    rng = np.random.default_rng(cells[0])
    sets = []
    for n_ion, frames in [(1, 1), (257, 3), (40, 9), (3000, 1)]:
        xyz = rng.uniform(0, 1, (frames, n_ion, 3)) * [el.box[0], el.box[1], 22.0] + [0, 0, 4.0]
        sets.append((xyz, rng.choice([-1.0, 1.0], (frames, n_ion)),
                     rng.normal(0, 0.01, (frames, el.n))))
    ctx = cpm.Context(el.box, precision=PREC[prec], rcut_dc=3.0)
    ctx.cpm_build_E(el.xyz, el.alpha)
    first = [None] * len(sets)
    for turn in range(6):
        for k, (xyz, q, qe) in enumerate(sets):
            b, qsol = ctx.cpm_potential(xyz, q, el.chi)
            got = (b.copy(), qsol.copy(), ctx.cpm_ion_forces(xyz, q, qe).copy())
            first[k] = first[k] or got
            for a, b in zip(first[k], got):
                assert np.array_equal(a, b), (turn, k)
    info = ctx.cpm_get_info()
    assert info["t_pot_sf_ms"] > 0 and info["t_pot_kspace_ms"] > 0 and info["t_pot_real_ms"] > 0
    b, qsol = ctx.cpm_potential(np.zeros((2, 0, 3)), np.zeros((2, 0)), el.chi)
    assert np.array_equal(b, np.stack([el.chi, el.chi])) and not qsol.any()
    ctx.close()
