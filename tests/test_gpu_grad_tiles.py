"""The network's gradient at the edges of its 128-sample tiles and of the blocks' shares of
them, with and without BF16 weights, against 64-bit torch autograd of the same network, and
the training step against the gradient call followed by the Adam call.

Tolerance: float products and sums of 128-sample tiles and an activation of ~1e-6 relative
error: 1e-5 of the largest gradient entry of a layer.
"""
import ctypes

import numpy as np
import pytest

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl
from paper_2111_06704_gb300.guess import LearnedGuess

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

SHAPES = ((32, 64), (64, 64), (64, 64), (64, 1))


def _reference(p, norm, feat, target, bf16):
    w = (p.to(torch.bfloat16) if bf16 else p).double().requires_grad_(True)
    h = (feat.double() - norm[:32].double()) * norm[32:].double()
    at = 0
    for k, (i, o) in enumerate(SHAPES):
        a = w[at:at + i * o].reshape(o, i)
        b = w[at + i * o:at + i * o + o]
        at += i * o + o
        h = h @ a.T + b
        if k < 3:
            h = h * torch.sigmoid(h)
    loss = ((h[:, 0] - target.double()) ** 2).mean()
    loss.backward()
    return float(loss.detach()), w.grad


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("samples", [1, 127, 128, 129, 152 * 128, 152 * 128 + 1, 50000])
def test_gradient_and_step(samples, bf16):
    el = wl.two_sheet_electrode(3, 2)
    ctx = cpm.Context(el.box, rcut_dc=3.0)
    g = LearnedGuess(ctx, seed=3, bf16=bf16)
    gen = torch.Generator(device="cuda").manual_seed(samples)
    feat = torch.randn((samples, 32), generator=gen, device="cuda")
    target = torch.randn(samples, generator=gen, device="cuda")
    g.norm.copy_(torch.cat([torch.full((32,), 0.1), torch.full((32,), 0.8)]))
    loss, ref = _reference(g.params, g.norm, feat, target, bf16)
    got = g.gradient(feat, target)
    assert abs(got - loss) <= 1e-5 * loss
    grad = g.grad.clone()
    at = 0
    for i, o in SHAPES:
        for n in (i * o, o):
            a, b = grad[at:at + n].double(), ref[at:at + n]
            assert (a - b).abs().max() <= 1e-5 * b.abs().max() + 1e-12
            at += n
    p0, m0, v0 = g.params.clone(), g.m.clone(), g.v.clone()
    g.adam(1e-3)
    p1 = g.params.clone()
    g.params.copy_(p0)
    g.m.copy_(m0)
    g.v.copy_(v0)
    g.step = 0
    g.train_step(feat, target, 1e-3)
    assert torch.equal(g.params, p1) and torch.equal(g.grad, grad)
    ctx.close()
