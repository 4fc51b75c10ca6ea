"""Potentials and forces where the memory for their usual scratch cannot be had: the call goes
through with less (no lists of far terms, few tabulated phasors, one share) and gives the same
result; once the workspace is released it takes the usual scratch again.

Tolerances, of the largest entry: FP64 sums in another grouping 1e-12; float storage 1e-10 (the sums
that are grouped differently are float pairs and FP64; the far chain keeps its order)."""
import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl
from paper_2111_06704_gb300.guess import LearnedGuess

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

PREC = {"fp64": cpm.CPM_PREC_FP64, "fp32": cpm.CPM_PREC_FP32, "bf16x6": cpm.CPM_PREC_BF16X6}
TOL = {"fp64": 1e-12, "fp32": 1e-10, "bf16x6": 1e-10}


class Memory:
    """Device memory from the caching allocator that refuses requests of `limit` bytes or more."""

    def __init__(self):
        self.limit, self.asked = None, []

    def alloc(self, nbytes):
        self.asked.append(nbytes)
        if self.limit is not None and nbytes >= self.limit:
            return None
        return torch.cuda.caching_allocator_alloc(nbytes)


def _ions(el, frames, n_ion):
    rng = np.random.default_rng(n_ion)
    xyz = rng.uniform(0, 1, (frames, n_ion, 3)) * [el.box[0], el.box[1], 22.0] + [0, 0, 4.0]
    return xyz, rng.choice([-1.0, 1.0], (frames, n_ion)), rng.normal(0, 0.01, (frames, el.n))


def _less_memory(prec, cells, call, **kw):
    el = wl.two_sheet_electrode(*cells)
    mem = Memory()
    ctx = cpm.Context(el.box, precision=PREC[prec],
                      allocator=(mem.alloc, torch.cuda.caching_allocator_delete), **kw)
    ctx.cpm_build_E(el.xyz, el.alpha)
    mem.asked.clear()
    ref = call(ctx, el).copy()
    most = max(mem.asked)  # the scratch: larger than the staged arrays
    ctx.cpm_release_workspace()
    mem.limit = most
    for _ in range(2):  # the size is not asked for again while it is known to be refused
        mem.asked.clear()
        got = call(ctx, el).copy()
        assert np.abs(got - ref).max() <= TOL[prec] * np.abs(ref).max()
    assert most not in mem.asked
    mem.limit = None
    ctx.cpm_release_workspace()
    mem.asked.clear()
    assert np.array_equal(call(ctx, el), ref) and most in mem.asked
    ctx.close()


@pytest.mark.parametrize("prec,cells,n_ion,frames,kw", [
    ("fp64", (8, 8), 3000, 24, {}),       # whole frames' phasors at a time
    ("fp64", (8, 5), 40011, 1, {}),       # a frame's ions in parts
    ("fp32", (20, 12), 5000, 2, {}),      # far terms in lists
    ("bf16x6", (20, 12), 300, 3, {"stream_operand": 1}),  # shares of the direct sum
])
def test_potential(prec, cells, n_ion, frames, kw):
    def call(ctx, el):
        xyz, q, _ = _ions(el, frames, n_ion)
        return ctx.cpm_potential(xyz, q, el.chi)[0]

    _less_memory(prec, cells, call, **kw)


@pytest.mark.parametrize("cells,n_ion,frames,kw", [
    ((8, 8), 3000, 24, {}),
    ((8, 5), 40011, 1, {}),  # one frame's ions in parts
    ((26, 20), 7000, 3, {}),  # the electrode's atoms in parts
])
def test_forces(cells, n_ion, frames, kw):
    def call(ctx, el):
        xyz, q, qe = _ions(el, frames, n_ion)
        return ctx.cpm_ion_forces(xyz, q, qe)

    _less_memory("fp64", cells, call, **kw)


def test_gradient():
    # blocks' shares of 84 KB each: as many blocks as the memory allows, the same sums to float
    # rounding of the tiles' (1e-5 of a layer's largest entry: the bar of the gradient's tests)
    el = wl.two_sheet_electrode(3, 2)
    mem = Memory()
    ctx = cpm.Context(el.box, rcut_dc=3.0,
                      allocator=(mem.alloc, torch.cuda.caching_allocator_delete))
    g = LearnedGuess(ctx, seed=3)
    gen = torch.Generator(device="cuda").manual_seed(1)
    feat = torch.randn((30000, 32), generator=gen, device="cuda")
    target = torch.randn(30000, generator=gen, device="cuda")
    loss = g.gradient(feat, target)
    ref = g.grad.clone()
    ctx.cpm_release_workspace()
    for mem.limit in (1 << 20, 100 << 10):
        assert abs(g.gradient(feat, target) - loss) <= 1e-5 * loss
        at = 0
        for n in (2048, 64, 4096, 64, 4096, 64, 64, 1):
            a, b = g.grad[at:at + n], ref[at:at + n]
            assert (a - b).abs().max() <= 1e-5 * b.abs().max()
            at += n
        ctx.cpm_release_workspace()
    ctx.close()


def test_no_lists_where_images_are_not_listed():
    # a box so small that every image of a pair is summed in FP64: no far terms, no pool for them
    # (2,000 ions' records and factors are 0.3 MB; a pool was 30 MB)
    el = wl.two_sheet_electrode(3, 2)
    mem = Memory()
    ctx = cpm.Context(el.box, precision=cpm.CPM_PREC_FP32, rcut_dc=3.0, rcut_real=30.0,
                      allocator=(mem.alloc, torch.cuda.caching_allocator_delete))
    ctx.cpm_build_E(el.xyz, el.alpha)
    mem.asked.clear()
    xyz, q, _ = _ions(el, 1, 2000)
    ctx.cpm_potential(xyz, q, el.chi)
    assert max(mem.asked) < 2 << 20
    ctx.close()
