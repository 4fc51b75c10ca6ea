"""Many ions in float storage: a frame's potential does not depend on how its ions were shared
out.  One frame (its far terms left by the shares and added in order, or its ions kept together)
against the same frame among enough copies that every warp takes all ions.

Tolerance 1e-10 of the largest entry: the float pairs and FP64 sums that are split differently
are good to ~1e-12; far sums by shares differ by up to 1e-9."""
import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("cells,n_ion,frames", [
    ((8, 5), 1201, 400),    # a list of whole-box shifts, the fewest ions kept in a chain
    ((8, 5), 3000, 400),
    ((13, 8), 4001, 160),   # every box edge above 2 r_c
    ((40, 20), 1500, 20),   # more groups than shares in a block
])
def test_one_frame_and_many(cells, n_ion, frames):
    el = wl.two_sheet_electrode(*cells)
    rng = np.random.default_rng(n_ion)
    xyz = rng.uniform(0, 1, (1, n_ion, 3)) * [el.box[0], el.box[1], 22.0] + [0, 0, 4.0]
    q = rng.choice([-1.0, 1.0], (1, n_ion))
    ctx = cpm.Context(el.box, precision=cpm.CPM_PREC_FP32, rcut_dc=3.0)
    ctx.cpm_build_E(el.xyz, el.alpha)
    one, _ = ctx.cpm_potential(xyz, q, el.chi)
    many, _ = ctx.cpm_potential(np.repeat(xyz, frames, 0), np.repeat(q, frames, 0), el.chi)
    ctx.close()
    assert np.abs(many - one).max() <= 1e-10 * np.abs(one).max()
