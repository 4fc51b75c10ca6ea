"""The network's gradient over many tiles a block (1,000), on samples that are all alike, so that
the roundings of a sum do not cancel: against 64-bit autograd of one sample, whose gradient is that
of the mean.

Tolerance, of a layer's largest entry: 1e-5 for the activations and the tiles' sums (the bar of the
gradient's other tests) and 256 roundings of a sum that grows to 256 terms, 256 x 2^-25 = 7.6e-6."""
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl
from paper_2111_06704_gb300.guess import LearnedGuess
from tests.test_gpu_grad_tiles import SHAPES, _reference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = 1e-5 + 256 * 2.0 ** -25


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_samples_alike(seed):
    el = wl.two_sheet_electrode(3, 2)
    ctx = cpm.Context(el.box, rcut_dc=3.0)
    g = LearnedGuess(ctx, seed=seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    row = torch.randn((1, 32), generator=gen, device="cuda")
    samples = 152 * 128 * 1000
    feat = row.expand(samples, 32).contiguous()
    target = torch.full((samples,), 0.7, device="cuda")
    g.norm.copy_(torch.cat([torch.full((32,), 0.1), torch.full((32,), 0.8)]))
    loss, ref = _reference(g.params, g.norm, row, target[:1], g.bf16)
    assert abs(g.gradient(feat, target) - loss) <= 1e-5 * loss
    at = 0
    for i, o in SHAPES:
        for n in (i * o, o):
            a, b = g.grad[at:at + n].double(), ref[at:at + n]
            assert (a - b).abs().max() <= TOL * b.abs().max()
            at += n
    ctx.close()
