"""Real factors of lattice_expr trees that are not plain numbers: each call reads the value that the
factor has then."""
import numpy as np
import pytest
import torch

import paper_1710_09409_gb300 as su3s
from paper_1710_09409_gb300 import autograd
from paper_1710_09409_gb300.autograd import _program

L0, L1 = ("leaf", 0), ("leaf", 1)


class Coefficient:
    value = 0.5

    def __float__(self):
        return self.value


def test_a_changed_factor_is_read_again():
    c, o = torch.tensor(0.5), Coefficient()
    tc, to = ("scale", c, L0), ("add", ("scale", o, L0), L1)
    assert list(_program(tc, (0,)).scalars) == [0.5] and list(_program(to, (0, 0)).scalars) == [0.5]
    c.mul_(4)
    o.value = -1.25
    assert list(_program(tc, (0,)).scalars) == [2.0] and list(_program(to, (0, 0)).scalars) == [-1.25]
    i = torch.tensor(0)
    t = ("mul", ("leaf", i), L1)
    assert list(_program(t, (0, 0)).prog) == [0, 0, 0, 1, 1, 0]
    i.add_(1)
    assert list(_program(t, (0, 0)).prog) == [0, 1, 0, 1, 1, 0]
    # equal plain numbers share a program, and nothing else is kept
    assert _program(("scale", 2, L0), (0,)) is _program(("scale", 2.0, L0), (0,))
    assert list(_program(("scale", np.float64(2.0), L0), (0,)).scalars) == [2.0]
    assert not any(x is c or x is o or x is i for k in autograd._programs for x in _flat(k))


def _flat(x):
    return [y for z in x for y in _flat(z)] if isinstance(x, tuple) else [x]


@pytest.mark.gpu
def test_values_and_gradients_follow_the_factor(gpu_lib):
    lat = su3s.Lattice((4, 4, 4, 4))
    f = su3s.Field(lat)
    f.pack(torch.randn(f.canonical_shape, dtype=torch.float64, device="cuda"))
    a = f.tensor.clone().requires_grad_(True)
    w = torch.ones_like(a)
    c = torch.tensor(0.5)
    product, tensors = ("mul", ("mul", L0, L1), ("leaf", 2)), [f.tensor, f.tensor, f.tensor, a]
    tree = ("add", product, ("scale", c, ("leaf", 3)))
    for value in (0.5, 2.0):
        c.fill_(value)
        z = su3s.lattice_expr(tree, lat, tensors)
        (g,) = torch.autograd.grad(z, a, w)
        ref = su3s.lattice_expr(("add", product, ("scale", value, ("leaf", 3))), lat, tensors)
        (gr,) = torch.autograd.grad(ref, a, w)
        assert torch.equal(z, ref) and torch.equal(g, gr)
        assert (g == value).all()
