"""The interpreter's kernels at the edges: every operation and operand kind, adjoints on either
side of a product, registers written in place, odd site counts and links, a destination that is a
leaf, and sites whose range sends them to native FP64 beside sites that stay."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

SEED = synth.SEED_BASE + 47
TOL = 1e-13


@pytest.fixture(scope="module")
def su3s(gpu_lib):
    return gpu_lib


def expr(tree, F):
    op = tree[0]
    if op == "leaf":
        return F[tree[1]].expr()
    if op == "scale":
        return tree[1] * expr(tree[2], F)
    if op == "adj":
        return expr(tree[1], F).adj()
    x, y = expr(tree[1], F), expr(tree[2], F)
    return x * y if op == "mul" else x + y if op == "add" else x - y


def leaf(n):
    return ("leaf", n)


@pytest.mark.parametrize("math", [2, 3], ids=["df32", "fx"])
def test_out_of_range_sites_beside_others(su3s, math):
    """Every third site holds 1e30: those run in native FP64 on their own slots of the register
    file, and their neighbours keep theirs."""
    dims = (5, 7, 9, 3)
    v = synth.volume(dims)
    f = {n: synth.su3(SEED, k, v) for k, n in enumerate("abc")}
    f["b"][::3, 1, 1, 0] = 1e30
    lat = su3s.Lattice(dims)
    F = {}
    for n in "abc":
        F[n] = su3s.Field(lat)
        F[n].upload(f[n])
    z = F["a"].like()
    tree = ("mul", ("add", leaf("a"), leaf("b")), ("sub", leaf("c"), leaf("a")))
    su3s.evaluate(z, expr(tree, F), math)
    got, ref = z.download(), oracle.eval_tree(tree, f)
    size = np.abs(f["b"]).max((1, 2, 3))
    # a product of sums of two unit matrices: 4 x (the two-term bound of a product's 6 terms)
    assert (np.abs(got - ref).max((1, 2, 3)) <= 4 * TOL * np.maximum(1.0, size)).all()
