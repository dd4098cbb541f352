"""Interpreted trees in which a field occurs again while an operation still waits for its first
occurrence, against the oracle: the forms that showed wrong registers, and random trees."""
import random

import numpy as np
import pytest

import oracle
import synth
from test_gpu_interp import expr, leaf, make, M, R, TOL, V

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def su3s(gpu_lib):
    return gpu_lib


a, b, c, r, s, v, w = (leaf(x) for x in "abcrsvw")


def mul(x, y):
    return ("mul", x, y)


def add(x, y):
    return ("add", x, y)


def sub(x, y):
    return ("sub", x, y)


TREES = [
    (M, add(a, ("scale", 0.5, a))),
    (M, mul(a, add(a, b))),
    (M, sub(a, add(a, b))),
    (M, mul(a, mul(add(a, b), c))),
    (M, mul(("adj", a), mul(b, a))),
    (M, mul(a, mul(b, a))),
    (M, mul(("adj", a), sub(a, b))),
    (M, add(a, add(mul(a, b), c))),
    (M, sub(a, mul(mul(b, a), c))),
    (M, sub(a, mul(b, ("scale", 0.25, a)))),
    (M, add(a, ("adj", mul(a, a)))),
    (V, add(v, ("scale", -0.5, v))),
    (V, mul(a, mul(("adj", a), v))),
    (V, sub(v, mul(a, mul(b, v)))),
    (R, mul(r, add(r, s))),
    (R, sub(r, mul(s, ("scale", 0.75, r)))),
]


def random_tree(rng, uses, kind):
    """A tree of `uses` leaf nodes over three matrices, two vectors and two reals."""
    k = rng.randrange(6)
    if k == 0 and kind == M:
        return ("adj", random_tree(rng, uses, kind))
    if k == 1:
        return ("scale", rng.choice([0.5, -0.75, 1.25]), random_tree(rng, uses, kind))
    if uses == 1:
        return leaf(rng.choice({M: "abc", V: "vw", R: "rs"}[kind]))
    left, op = rng.randrange(1, uses), rng.choice(["mul", "add", "sub"])
    return (op, random_tree(rng, left, M if op == "mul" and kind == V else kind), random_tree(rng, uses - left, kind))


def scalars(t):
    return (t[0] == "scale") + sum(scalars(x) for x in t[1:] if isinstance(x, tuple))


def random_trees(seed, n):
    rng, out = random.Random(seed), []
    while len(out) < n:
        kind = rng.choice([M, M, V, R])
        t = random_tree(rng, rng.randrange(3, 7), kind)
        if scalars(t) <= 4 and len(oracle.leaf_names(t)) <= 6:
            out.append((kind, t))
    return out


def steps(t):
    """Arithmetic steps of a tree: the terms its error bound adds up."""
    return 1 + sum(steps(x) for x in t[1:] if isinstance(x, tuple))


def magnitude(t, size):
    """Bound on the largest real of a tree's value and of everything in it."""
    op = t[0]
    if op == "leaf":
        return size[t[1]]
    if op == "scale":
        return max(1.0, abs(t[1])) * magnitude(t[2], size)
    x = [magnitude(u, size) for u in t[1:]]
    return max(x[0], 6.0 * x[0] * x[1]) if op == "mul" else sum(x)


# 300,000 sites is where the pair arithmetic takes two sites per thread
@pytest.mark.parametrize("dims", [(9, 8, 7, 6), (31, 37, 41, 7)])
@pytest.mark.parametrize("math", [1, 2, 3], ids=["f64", "df32", "fx"])
def test_fields_that_occur_again(su3s, dims, math):
    lat = su3s.Lattice(dims)
    h, F = {}, {}
    for name in "abcrsvw":
        h1, F1 = make(su3s, lat, ["v" if name == "w" else name], 1, 0, 64)
        (h[name],), (F[name],) = h1.values(), F1.values()
    h["w"] = np.ascontiguousarray(h["v"][::-1])
    F["w"].upload(h["w"])
    size = {n: max(1.0, np.abs(h[n]).max()) for n in h}
    z = {k: F[n].like() for k, n in ((M, "a"), (V, "v"), (R, "r"))}
    for kind, tree in TREES + random_trees(synth.SEED_BASE + 51, 24):
        su3s.evaluate(z[kind], expr(tree, F), math)
        ref = oracle.eval_tree(tree, {n: h[n] for n in oracle.leaf_names(tree)})
        # every step within a product's bound, of the largest value that can occur
        tol = TOL * steps(tree) * magnitude(tree, size)
        err = np.abs(z[kind].download() - ref).max()
        assert err <= tol, (tree, err, tol)
