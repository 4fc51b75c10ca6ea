"""The local inverses of the PCG-DC preconditioner at the edges of their kernel: neighbourhoods of
one atom, around whole 32-element segments and up to the largest size, with and without row
exchanges (atoms 0.42 A apart: entries above the diagonal), against the FP64 oracle.

Tolerance 1e-11 of the largest entry, the bar of the parity test (refinement ends at
corrections below 1e-9, whose error is ~1e-13)."""
import numpy as np
import pytest

from oracle import precond as pc
from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _check(box, xyz, alpha, rcut):
    p_ref, nb = pc.dc_preconditioner(xyz, alpha, box, wl.G_DC, rcut)
    ctx = cpm.Context(box, rcut_dc=rcut, g_dc=wl.G_DC)
    ctx.cpm_build_E(xyz, alpha)
    off, idx, val = ctx.cpm_get_precond()
    ctx.close()
    top = np.abs(p_ref).max()
    for j in range(len(xyz)):
        cols = idx[off[j]:off[j + 1]]
        assert np.array_equal(cols, nb[j])
        np.testing.assert_allclose(val[off[j]:off[j + 1]], p_ref[j, cols], rtol=0,
                                   atol=1e-11 * top)
    return max(len(x) for x in nb)


@pytest.mark.parametrize("rcut", [0.5, 1.6, 5.1, 7.4, 8.6])
@pytest.mark.parametrize("pairs", [False, True])
def test_sheets(rcut, pairs):
    el = wl.two_sheet_electrode(8, 5)
    xyz = np.array(el.xyz)
    for a in (10, 100, 200) if pairs else ():
        xyz[a + 1] = xyz[a] + [0.42, 0.0, 0.0]
    _check(el.box, xyz, el.alpha, rcut)


def test_large_neighbourhoods():
    el = wl.stacked_electrode(np.random.default_rng(3), 9, 6, 3, spacing=6.0)
    assert 128 < _check(el.box, el.xyz, el.alpha, 8.4) <= 160
