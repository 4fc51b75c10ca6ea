"""The solver's tuner compares the two paths' solves, not what their first use costs: reservations
(here a device allocator that takes 20 ms an allocation) and the loading of kernels are in neither
time, so the path chosen after a cold first solve is the one that is faster warm."""
import time

import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _warm_time(el, b, path):
    ctx = cpm.Context(el.box, solver_path=path)
    ctx.cpm_build_E(el.xyz, el.alpha)
    best = np.inf
    for _ in range(5):
        t = time.perf_counter()
        ctx.cpm_solve(b, tol=1e-8)
        best = min(best, time.perf_counter() - t)
    ctx.close()
    return best


def _alloc(nbytes):
    time.sleep(0.02)
    return torch.cuda.caching_allocator_alloc(nbytes)


@pytest.mark.parametrize("release", [False, True])
@pytest.mark.parametrize("cells,nrhs", [((25, 20), 1), ((25, 20), 20), ((20, 12), 40)])
def test_cold_and_warm_choose_alike(cells, nrhs, release):
    el = wl.two_sheet_electrode(*cells)
    b = np.random.default_rng(nrhs).normal(size=(nrhs, el.n))
    kernels, cluster = _warm_time(el, b, 1), _warm_time(el, b, 2)
    assert kernels < 0.8 * cluster  # sizes where the choice is plain
    ctx = cpm.Context(el.box, allocator=(_alloc, torch.cuda.caching_allocator_delete))
    ctx.cpm_build_E(el.xyz, el.alpha)
    for _ in range(3):
        ctx.cpm_solve(b, tol=1e-8)
        path = ctx.cpm_get_info()["solve_path"]
        if release:
            ctx.cpm_release_workspace()
    assert path == 1
    ctx.close()
