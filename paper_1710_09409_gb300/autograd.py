"""torch.autograd bridge: differentiable evaluation of lattice expressions.

Forward runs the fused evaluation kernel; backward runs the hand-written
reverse-mode kernel (for z = a*b: dA = G B^dagger, dB = A^dagger G; sums,
real factors and adjoints by the chain rule), both through the C ABI.  Tensors
are FP64 fields in a device layout (flat float64 CUDA tensors of the field's
size); the gradient convention is the one PyTorch uses for real tensors, i.e.
dL/dRe and dL/dIm per stored real, which for complex entries is
dL/dRe + i dL/dIm.
"""
import ctypes

import numpy as np
import torch

from . import F64, MATH_DEFAULT, MATRIX, SOA, _check, _stream, _Tree, load

_OPS = {"mul": 1, "add": 2, "sub": 3}
_FIXED = (int, float, bool, np.float64)   # number types whose objects never change


def _result_kind(tree, kinds):
    op = tree[0]
    if op == "leaf":
        return kinds[tree[1]]
    if op in ("mul", "scale"):
        return _result_kind(tree[2], kinds)
    if op in ("add", "sub"):
        return _result_kind(tree[1], kinds)
    return MATRIX


class _Program:
    """A tree in postfix order for su3s_tree: (operation, argument) pairs, the real factors, the
    leaf kinds, and which tensors it reads."""

    def __init__(self, tree, kinds):
        prog, scalars, self.reads = [], [], set()
        n = len(kinds)
        given = list(kinds)   # the values the tree is made of

        def walk(t):
            op = t[0]
            if op == "leaf":
                given.append(t[1])
                i = range(n)[t[1]]
                self.reads.add(i)
                prog.extend((0, i))
            elif op in _OPS:
                walk(t[1])
                walk(t[2])
                prog.extend((_OPS[op], 0))
            elif op == "scale":
                given.append(t[1])
                scalars.append(float(t[1]))
                k = len(scalars) - 1
                walk(t[2])
                prog.extend((4, k))
            elif op == "adj":
                walk(t[1])
                prog.extend((5, 0))
            else:
                raise ValueError(op)

        walk(tree)
        self.prog = (ctypes.c_int32 * len(prog))(*prog)
        self.scalars = (ctypes.c_double * max(1, len(scalars)))(*scalars)
        self.kinds = (ctypes.c_int * n)(*kinds)
        self.kind = _result_kind(tree, kinds)
        self.nprog, self.nscalar, self.nleaf = len(prog) // 2, len(scalars), n
        # Equal keys have equal programs, now and later: not so for zeros (0.0 == -0.0), nor for
        # objects that can change under the same key (a 0-d tensor as a factor, updated in place).
        self.keep = all(type(x) in _FIXED for x in given) and all(s != 0.0 for s in scalars)


_programs = {}


def _program(tree, kinds):
    key = (tree, kinds)
    try:
        p = _programs.get(key)
    except TypeError:      # a tree with lists in it
        return _Program(tree, kinds)
    if p is None:
        p = _Program(tree, kinds)
        if p.keep:
            if len(_programs) >= 256:
                _programs.clear()
            _programs[key] = p
    return p


def _tree_call(prog, spec, tensors):
    """The su3s_tree of a call; the arrays it points to are kept alive by the returned list."""
    _, lattice, _, nmu, layout, block, _ = spec
    for t in tensors:
        if not t.is_cuda or not t.is_contiguous():
            raise ValueError("field storage must be a contiguous CUDA tensor")
    n = prog.nleaf
    ptrs = (ctypes.c_void_p * n)(*[t.data_ptr() for t in tensors])
    sizes = (ctypes.c_size_t * n)(*[t.numel() * t.element_size() for t in tensors])
    tree = _Tree(lattice._h, ctypes.addressof(prog.prog), ctypes.addressof(prog.scalars),
                 ctypes.addressof(prog.kinds), ctypes.addressof(ptrs), ctypes.addressof(sizes),
                 prog.nprog, prog.nscalar, n, nmu, layout, block)
    return tree, [ptrs, sizes]


def _field_tensor(spec, kind):
    _, lattice, _, nmu, layout, block, _ = spec
    nb = ctypes.c_size_t()
    _check(load().su3s_field_bytes(lattice._h, kind, nmu, F64, layout, block, ctypes.byref(nb)))
    return torch.empty(nb.value // 8, dtype=torch.float64, device="cuda")


class LatticeFunction(torch.autograd.Function):
    """apply(spec, *tensors); spec = (tree, lattice, kinds, nmu, layout, block, math)."""

    @staticmethod
    def forward(ctx, spec, *tensors):
        prog = _program(spec[0], tuple(spec[2][i] for i in range(len(tensors))))
        tree, keep = _tree_call(prog, spec, tensors)
        dest = _field_tensor(spec, prog.kind)
        _check(load().su3s_tree_eval(ctypes.byref(tree), dest.data_ptr(), dest.numel() * 8, spec[6],
                                     _stream(None)))
        ctx.spec = spec
        ctx.prog = prog
        ctx.save_for_backward(*tensors)
        return dest

    @staticmethod
    def backward(ctx, grad):
        spec, prog, tensors = ctx.spec, ctx.prog, ctx.saved_tensors
        tree, keep = _tree_call(prog, spec, tensors)
        g = grad.detach().contiguous()
        if not g.is_cuda:
            raise ValueError("field storage must be a contiguous CUDA tensor")
        grads = [_field_tensor(spec, prog.kinds[i]) if i in prog.reads and ctx.needs_input_grad[1 + i]
                 else None for i in range(prog.nleaf)]
        out = (ctypes.c_void_p * prog.nleaf)(*[None if t is None else t.data_ptr() for t in grads])
        _check(load().su3s_tree_adjoint(ctypes.byref(tree), g.data_ptr(), g.numel() * g.element_size(), out,
                                        spec[6], _stream(None)))
        return (None,) + tuple(grads)


def lattice_expr(tree, lattice, tensors, kinds=None, nmu=1, layout=SOA, block=64,
                 math=MATH_DEFAULT):
    """Differentiable dest = tree(tensors) for FP64 fields in a device layout.

    `tree` is a nested tuple ("leaf", i) | ("mul", x, y) | ("add", x, y) |
    ("sub", x, y) | ("scale", s, x) | ("adj", x) with leaf i = tensors[i]."""
    kinds = tuple(kinds) if kinds is not None else (MATRIX,) * len(tensors)
    spec = (tree, lattice, kinds, nmu, layout, block, math)
    return LatticeFunction.apply(spec, *tensors)
