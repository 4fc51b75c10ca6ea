"""What cpm_release_workspace costs the next call: the device memory again (from the caching
allocator here, a cached block, some 10 us), but not the context's page of pinned host memory: with
that pinned anew, a small potential after a release took nine times as long (390 us for 44).  Less
than twice a call without a release."""
import time

import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _median(f):
    times = []
    for _ in range(51):
        t = time.perf_counter()
        f()
        times.append(time.perf_counter() - t)
    return float(np.median(times))


def test_no_pinning_after_a_release():
    el = wl.two_sheet_electrode(8, 8)
    rng = np.random.default_rng(0)
    ions = rng.uniform(0, 1, (1, 200, 3)) * [el.box[0], el.box[1], 20.0] + [0, 0, 5.0]
    ions = torch.tensor(ions, device="cuda")
    q = torch.ones((1, 200), dtype=torch.float64, device="cuda")
    chi = torch.tensor(el.chi, device="cuda")
    b = torch.zeros((1, el.n), dtype=torch.float64, device="cuda")
    ctx = cpm.Context(el.box, allocator=(torch.cuda.caching_allocator_alloc,
                                         torch.cuda.caching_allocator_delete))
    ctx.cpm_build_E(el.xyz, el.alpha)

    def call():
        ctx.cpm_potential(ions, q, chi, b)

    def released():
        ctx.cpm_release_workspace()
        call()

    for f in (call, released):
        f()
    assert _median(released) < 2.0 * _median(call)
    ctx.close()
