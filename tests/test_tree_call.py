"""Trees over device buffers in one call (su3s_tree_*, the autograd bridge): what a program may
be (no GPU), and that the results are those of the calls it stands for (GPU)."""
import ctypes
import threading

import pytest
import torch

import paper_1710_09409_gb300 as su3s
from paper_1710_09409_gb300.autograd import _Program, _program

FAKE = 1 << 40  # 16-byte aligned, never dereferenced
L0, L1 = ("leaf", 0), ("leaf", 1)


def call(prog, scalars=(), kinds=(0, 0), ptr=FAKE, nbytes=1 << 20, dest=FAKE, math=0):
    L = su3s.load(build_if_missing=True)
    lat = su3s.Lattice((2, 2, 2, 2))
    n = len(kinds)
    keep = [(ctypes.c_int32 * max(1, len(prog)))(*prog), (ctypes.c_double * 4)(*scalars),
            (ctypes.c_int * n)(*kinds), (ctypes.c_void_p * n)(*[ptr] * n), (ctypes.c_size_t * n)(*[nbytes] * n)]
    t = su3s._Tree(lat._h, *[ctypes.addressof(k) for k in keep], len(prog) // 2, len(scalars), n, 1, 0, 0)
    rc = L.su3s_tree_eval(ctypes.byref(t), dest, nbytes, math, None)
    return rc, L.su3s_last_error().decode()


@pytest.mark.parametrize("prog,scalars,kinds,code", [
    ((1, 0), (), (0, 0), 1),                       # a product of nothing
    ((0, 0, 0, 1), (), (0, 0), 1),                 # two values left
    ((0, 2), (), (0, 0), 1), ((0, -1), (), (0, 0), 1), ((7, 0), (), (0, 0), 1), ((0, 0, 6, 0), (), (0, 0), 1),
    ((0, 0, 4, 1), (2.0,), (0, 0), 1), ((0, 0, 4, -1), (2.0,), (0, 0), 1),
    ((0, 1, 0, 0, 1, 0), (), (0, 1), 2),           # vector times matrix
    ((0, 0, 0, 1, 2, 0), (), (0, 1), 2),           # matrix plus vector
    ((0, 1, 5, 0), (), (0, 1), 2),                 # adjoint of a vector
    ((), (), (0, 0), 1)])
def test_bad_programs_are_refused(prog, scalars, kinds, code):
    rc, msg = call(prog, scalars, kinds)
    assert rc == code and msg


def test_bad_buffers_are_refused():
    ok = (0, 0, 0, 1, 1, 0)
    assert call(ok, ptr=FAKE + 8)[0] == 1          # not 16-byte aligned
    assert call(ok, ptr=None)[0] == 1
    assert call(ok, nbytes=16)[0] == 3             # smaller than the field
    assert call(ok, dest=None)[0] == 1
    assert call(ok, math=9)[0] == 1


def test_programs():
    p = _Program(("sub", ("mul", ("adj", L0), L1), ("scale", 2.5, ("leaf", -1))), (0, 0))
    assert list(p.prog) == [0, 0, 5, 0, 0, 1, 1, 0, 0, 1, 4, 0, 3, 0]
    assert list(p.scalars) == [2.5] and p.reads == {0, 1} and p.kind == su3s.MATRIX
    with pytest.raises(IndexError):
        _Program(("leaf", 2), (0, 0))
    with pytest.raises(ValueError):
        _Program(("pow", L0, L1), (0, 0))
    # zeros of either sign are equal keys with different programs
    assert str(list(_program(("scale", 0.0, L0), (0,)).scalars)) == "[0.0]"
    assert str(list(_program(("scale", -0.0, L0), (0,)).scalars)) == "[-0.0]"
    # a tree with lists in it has no key
    assert list(_program(["mul", L0, L1], (0, 0)).prog) == [0, 0, 0, 1, 1, 0]


def fields(lat, n, kind=su3s.MATRIX):
    g = torch.Generator(device="cuda").manual_seed(5)
    f = [su3s.Field(lat, kind) for _ in range(n)]
    for x in f:
        x.pack(torch.randn(x.canonical_shape, dtype=torch.float64, device="cuda", generator=g))
    return f


@pytest.mark.gpu
@pytest.mark.parametrize("needs", [(True, True), (True, False), (False, True)])
def test_autograd_equals_the_calls_it_stands_for(gpu_lib, needs):
    lat = su3s.Lattice((5, 6, 7, 3))
    a, b, w = fields(lat, 3)
    ta, tb = a.tensor.clone().requires_grad_(needs[0]), b.tensor.clone().requires_grad_(needs[1])
    z = su3s.lattice_expr(("add", ("mul", L0, L1), ("scale", 0.5, L0)), lat, [ta, tb])
    ref = a.like()
    su3s.evaluate(ref, a * b + 0.5 * a)
    assert torch.equal(z.detach(), ref.tensor)
    z2 = su3s.lattice_expr(("mul", L0, ("leaf", -1)), lat, [ta, tb])
    z2.backward(w.tensor)
    ga, gb = a.like(), a.like()
    su3s.eval_adjoint(a * b, w, [ga, gb])
    for t, g, need in ((ta, ga, needs[0]), (tb, gb, needs[1])):
        assert (t.grad is not None) == need
        assert not need or torch.equal(t.grad, g.tensor)
    with pytest.raises(ValueError):
        su3s.lattice_expr(("mul", L0, L1), lat, [ta.detach()[::2], tb])


@pytest.mark.gpu
def test_fields_of_a_new_thread_and_stream(gpu_lib):
    """A thread that has made no call yet gets the same kernels and results, on its own stream."""
    lat = su3s.Lattice((8, 8, 8, 4))
    a, b = fields(lat, 2)
    want = a.like()
    su3s.evaluate(want, a * b)
    torch.cuda.synchronize()
    got = {}

    def work():
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            x, y = (su3s.Field(lat, tensor=t) for t in (a.tensor, b.tensor))
            z = x.like()
            su3s.evaluate(z, x * y)
            g = su3s.lattice_expr(("mul", L0, L1), lat, [a.tensor, b.tensor])
            s.synchronize()
            got["z"], got["g"] = z.tensor, g

    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert torch.equal(got["z"], want.tensor) and torch.equal(got["g"], want.tensor)


@pytest.mark.gpu
def test_one_leaf_node_serves_every_tree(gpu_lib):
    lat = su3s.Lattice((4, 4, 4, 4))
    a, b = fields(lat, 2)
    z, ref = a.like(), a.like()
    e = a * b
    del b
    su3s.evaluate(z, e + e)
    su3s.evaluate(ref, 2.0 * e)
    assert torch.equal(z.tensor, ref.tensor)
    su3s.evaluate(z, a, su3s.MATH_F64)   # a copy (the pair arithmetic holds 48 bits)
    assert torch.equal(z.tensor, a.tensor)
    with pytest.raises(TypeError):
        a * "b"
    with pytest.raises(su3s.Su3sError):
        a + su3s.Field(lat, su3s.VECTOR)
