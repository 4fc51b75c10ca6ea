"""The real-space part of the potential: every screen mode and storage, ion counts and atom
orders at the edges of the warps' groups, against the FP64 oracle and against FP64 storage.

Tolerance of b: float storage 2e-8 of the largest entry (its k-space tail is float; the
bars of the parity tests), FP64 storage 1e-11.
"""
import numpy as np
import pytest

from oracle import ewald as ew
from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

PREC = {"fp64": cpm.CPM_PREC_FP64, "bf16x6": cpm.CPM_PREC_BF16X6}
TOL = {"fp64": 1e-11, "bf16x6": 2e-8}


def _b(el, ions, q, prec, order=None, **kw):
    order = np.arange(el.n) if order is None else order
    ctx = cpm.Context(el.box, precision=PREC[prec], rcut_dc=3.0, **kw)
    ctx.cpm_build_E(el.xyz[order], el.alpha[order])
    b, qsol = ctx.cpm_potential(ions, q, el.chi[order])
    ctx.close()
    out = np.empty_like(b)
    out[:, order] = b
    return out, qsol


def _ions(rng, box, frames, n, zlo=2.0, zhi=28.0):
    return np.stack([np.column_stack([rng.uniform(-box[0], 2 * box[0], n),
                                      rng.uniform(0, box[1], n),
                                      rng.uniform(zlo, zhi, n)]) for _ in range(frames)])


@pytest.mark.parametrize("prec", ["fp64", "bf16x6"])
@pytest.mark.parametrize("cells,rcut,n_ion,frames", [
    ((10, 6), 12.0, 33, 2),   # every box edge above 2 r_c
    ((8, 5), 12.0, 1, 1),     # a list of whole-box shifts, one ion
    ((3, 2), 12.0, 70, 3),    # many shifts, 48 atoms
    ((3, 2), 30.0, 9, 1),     # more than 64 shifts: every image in FP64
])
def test_modes_against_the_oracle(prec, cells, rcut, n_ion, frames):
    el = wl.two_sheet_electrode(*cells)
    rng = np.random.default_rng(n_ion)
    ions = _ions(rng, el.box, frames, n_ion)
    ions[0, 0] = el.xyz[3] + np.array([0.05, -0.02, 0.04])  # inside the Gaussian's core
    q = rng.choice([-1.0, 1.0, 0.37], size=(frames, n_ion))
    b, qsol = _b(el, ions, q, prec, rcut_real=rcut)
    for f in range(frames):
        bs = ew.electrolyte_potential(el.xyz, el.alpha, ions[f], q[f], el.box, 0.3, rcut)
        bs = ew.neutral_form_bsol(bs, el.xyz, ions[f], q[f], el.box, 0.3)
        ref = ew.rhs_volts(el.chi, bs)
        assert np.abs(b[f] - ref).max() <= TOL[prec] * np.abs(ref).max(), f
        assert abs(qsol[f] - q[f].sum()) <= 1e-12 * n_ion


@pytest.mark.parametrize("order", ["given", "reversed", "shuffled"])
def test_atom_orders_and_dense_ions(order):
    # 1,144 atoms, 3,000 ions: full lists, several of the grid's shares; a shuffled electrode
    # has warps whose atoms span the box (no ion dropped, the wrapping screen)
    el = wl.two_sheet_electrode(13, 11)
    rng = np.random.default_rng(5)
    ions = _ions(rng, el.box, 1, 3000)
    q = np.tile([1.0, -1.0], 1500)[None]
    perm = {"given": np.arange(el.n), "reversed": np.arange(el.n)[::-1].copy(),
            "shuffled": rng.permutation(el.n)}[order]
    ref, _ = _b(el, ions, q, "fp64")
    b, _ = _b(el, ions, q, "bf16x6", perm)
    assert np.abs(b - ref).max() <= TOL["bf16x6"] * np.abs(ref).max()
