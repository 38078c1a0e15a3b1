"""Scatter-network inputs that the forward pass rounds itself (csrc/mlp.cu): rows
that start on 16 bytes and rows that do not, row counts at the edges of its
128-row tiles and of a second tile per group, outputs written over the inputs,
and the gradient, whose forward pass rounds them beforehand.  The rounding is
the same, so the outputs are the same bits."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_17111_gb300 as lm  # noqa: E402
from paper_2305_17111_gb300 import _native as nat  # noqa: E402


def _forward(net, x_ptr, n, out_ptr):
    rc = nat.load().lm_surrogate_forward(net._s, ctypes.c_void_p(x_ptr), n,
                                         ctypes.c_void_p(out_ptr), None)
    assert rc == 0
    torch.cuda.synchronize()


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 * 3 + 5, 100_001])
def test_forward_rounds_rows_of_any_alignment(n):
    net = lm.Surrogate(seed=3)
    flat = torch.from_numpy(np.random.default_rng(n).normal(size=n * 32 + 1).astype(np.float32)).cuda()
    x = flat[1:].clone()                       # on 16 bytes; flat[1:] itself is not
    assert x.data_ptr() % 16 == 0 and flat[1:].data_ptr() % 16 == 4
    a = torch.full((n,), float("nan"), device="cuda")
    b = torch.full((n,), float("nan"), device="cuda")
    _forward(net, x.data_ptr(), n, a.data_ptr())
    _forward(net, flat[1:].data_ptr(), n, b.data_ptr())
    assert torch.isfinite(a).all() and torch.equal(a, b)
    # rows already in BF16 round to themselves
    _forward(net, x.bfloat16().float().data_ptr(), n, b.data_ptr())
    assert torch.equal(a, b)
    # outputs over the first inputs
    _forward(net, x.data_ptr(), n, x.data_ptr())
    assert torch.equal(x[:n], a)


@pytest.mark.parametrize("n", [1, 127, 129, 1000])
@pytest.mark.parametrize("weighted", [False, True])
def test_gradient_rounds_its_inputs(n, weighted):
    """FP32 inputs give what inputs already in BF16 give, with the loss, also where
    the scratch has grown since a smaller call and is larger than the call needs."""
    net = lm.Surrogate(seed=4)
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn(n, 32, generator=g, device="cuda")
    t = torch.randn(n, generator=g, device="cuda")
    w = torch.rand(n, generator=g, device="cuda") + 0.5 if weighted else None
    rounded = x.bfloat16().float()
    first = net.gradient(x, t, w)
    again = net.gradient(rounded, t, w)
    big = torch.randn(3001, 32, generator=g, device="cuda")
    net.gradient(big, torch.randn(3001, generator=g, device="cuda"))     # the scratch grows
    later = net.gradient(x, t, w)
    assert torch.isfinite(first[0]).all() and first[1] > 0.0
    for other in (again, later):
        assert torch.equal(first[0], other[0]) and first[1] == other[1]
    net.close()
