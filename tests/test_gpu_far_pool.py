"""Many ions in float storage, in orders and places that fill the shares' lists of far terms
unevenly: the potential of one frame (ions in shares) is that of the same frame among enough copies
that every warp takes all ions.  Ions sorted in space, as a cell-sorted simulation has them,
give one share most of an atom's terms; ions in a small ball with atoms in no order give
every warp a lane with all of them, more than the pool of the lists holds, and the sums are taken again.

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


def _one_and_many(el, xyz, q, frames):
    ctx = cpm.Context(el.box, precision=cpm.CPM_PREC_FP32, rcut_dc=3.0)
    ctx.cpm_build_E(el.xyz, el.alpha)
    one, _ = ctx.cpm_potential(xyz[None], q[None], el.chi)
    again, _ = ctx.cpm_potential(xyz[None], q[None], el.chi)
    many, _ = ctx.cpm_potential(np.repeat(xyz[None], frames, 0), np.repeat(q[None], frames, 0),
                                el.chi)
    ctx.close()
    assert np.array_equal(one, again)
    assert np.abs(many - one).max() <= 1e-10 * np.abs(one).max()


@pytest.mark.parametrize("axis", [0, 2])
@pytest.mark.parametrize("cells,n_ion,frames", [
    ((8, 5), 3000, 400),   # a list of whole-box shifts
    ((13, 8), 4001, 160),  # every box edge above 2 r_c
    ((20, 12), 5000, 64),
])
def test_sorted_ions(cells, n_ion, frames, axis):
    el = wl.two_sheet_electrode(*cells)
    rng = np.random.default_rng(n_ion + axis)
    xyz = rng.uniform(0, 1, (n_ion, 3)) * [el.box[0], el.box[1], 22.0] + [0, 0, 4.0]
    xyz = xyz[np.argsort(xyz[:, axis])]
    # charges of one sign: the far sums grow, and so do their roundings
    _one_and_many(el, xyz, np.ones(n_ion), frames)


@pytest.mark.parametrize("shuffled", [False, True])
def test_ions_in_a_ball(shuffled):
    el = wl.two_sheet_electrode(13, 8)
    rng = np.random.default_rng(7)
    if shuffled:
        order = rng.permutation(el.n)
        el.xyz[:], el.alpha[:], el.chi[:] = el.xyz[order], el.alpha[order], el.chi[order]
    xyz = rng.normal(0, 0.5, (4001, 3)) + [10.0, 10.0, 4.0]
    _one_and_many(el, xyz, rng.uniform(0.5, 1.0, 4001), 160)
