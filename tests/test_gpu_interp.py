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


M, V, R = "matrix", "vector", "real"
TREES = {
    "a (b + c) - d": (M, ("sub", ("mul", leaf("a"), ("add", leaf("b"), leaf("c"))), leaf("d"))),
    "adjoint of the left product": (M, ("mul", ("adj", ("mul", leaf("a"), leaf("b"))), leaf("c"))),
    "adjoints on both sides": (M, ("mul", ("adj", ("add", leaf("a"), leaf("b"))), ("adj", leaf("c")))),
    "adjoint twice": (M, ("mul", ("adj", ("adj", ("sub", leaf("a"), leaf("b")))), leaf("c"))),
    "adjoint at the root": (M, ("adj", ("add", ("mul", leaf("a"), leaf("b")), leaf("c")))),
    "a leaf used again": (M, ("add", ("mul", leaf("a"), ("sub", leaf("b"), leaf("a"))),
                              ("mul", leaf("a"), leaf("a")))),
    "scales": (M, ("sub", ("scale", 0.75, ("mul", ("scale", -2.0, leaf("a")), leaf("b"))),
                   ("scale", 1.5, leaf("a")))),
    "same leaf twice in a sum": (M, ("add", ("add", leaf("a"), leaf("a")), ("scale", 3.0, leaf("a")))),
    "vector": (V, ("add", ("mul", ("adj", ("add", leaf("a"), leaf("b"))), leaf("v")),
                   ("scale", -0.5, leaf("v")))),
    "real": (R, ("sub", ("mul", ("mul", leaf("r"), leaf("s")), leaf("r")), ("scale", 2.0, leaf("s")))),
}


def make(su3s, lat, names, nmu, layout, block):
    n = lat.volume * nmu
    h, F = {}, {}
    for name in names:
        k = sum(map(ord, name))
        kind = V if name == "v" else R if name in "rs" else M
        h[name] = (synth.gauss_vector(SEED, k, n) if kind == V else synth.uniform_real(SEED, k, n)
                   if kind == R else synth.su3(SEED, k, n))
        F[name] = su3s.Field(lat, {M: su3s.MATRIX, V: su3s.VECTOR, R: su3s.REAL}[kind], nmu, su3s.F64,
                             layout, block)
        F[name].upload(h[name])
    return h, F


# 64 and 128 sites are half and one run of a block's pairs; 30 pads to 64, 129 to 192
@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (30, 1, 1, 1), (43, 3, 1, 1), (9, 8, 7, 6)])
@pytest.mark.parametrize("nmu,layout,block", [(1, 0, 64), (3, 0, 64), (1, 1, 4), (2, 1, 32)])
@pytest.mark.parametrize("math", [1, 2, 3], ids=["f64", "df32", "fx"])
def test_trees_match_oracle(su3s, dims, nmu, layout, block, math):
    lat = su3s.Lattice(dims)
    cat = {s for (_, s, _, _) in su3s.catalogue()}
    for name, (kind, tree) in TREES.items():
        names = oracle.leaf_names(tree)
        h, F = make(su3s, lat, names, nmu, layout, block)
        e = expr(tree, F)
        assert e.signature() not in cat, name
        z = F[{M: "a", V: "v", R: "r"}[kind]].like()
        su3s.evaluate(z, e, math)
        ref = oracle.eval_tree(tree, h)
        # products of up to three factors and sums of them: 4 x the two-term product's bound
        tol = 4 * TOL * max(1.0, np.abs(ref).max())
        assert np.abs(z.download() - ref).max() < tol, name
        if kind == M:   # a destination that is a leaf
            su3s.evaluate(F["a"], e, math)
            assert np.abs(F["a"].download() - ref).max() < tol, name


# more sites than one wave of threads takes: two sites per thread for programs of three registers,
# an odd number of 32-site runs; 300,000 sites is where that begins
@pytest.mark.parametrize("dims", [(300000 - 64, 1, 1, 1), (300000, 1, 1, 1), (31, 37, 41, 15)])
def test_large_lattices_match_oracle(su3s, dims):
    lat = su3s.Lattice(dims)
    h, F = make(su3s, lat, "abcvrs", 1, 0, 64)
    h["d"], F["d"] = h["c"], F["c"]
    for x in "abc":                    # one site in 997 out of range
        h[x][::997, 2, 0, 1] = 1e30
        F[x].upload(h[x])
    for name, (kind, tree) in TREES.items():
        z = F[{M: "a", V: "v", R: "r"}[kind]].like()
        su3s.evaluate(z, expr(tree, F))
        names = oracle.leaf_names(tree)
        ref = oracle.eval_tree(tree, {n: h[n] for n in names})
        # per site: products of up to three factors of the site's largest magnitude
        size = np.max([np.abs(h[n]).reshape(lat.volume, -1).max(1) for n in names], 0)
        tol = 24 * TOL * np.maximum(1.0, size) ** 3
        err = np.abs(z.download() - ref).reshape(lat.volume, -1).max(1)
        assert (err <= tol).all(), name


def test_program_limits_stand(su3s):
    """What the interpreter refused for its size before registers were reused is refused still."""
    lat = su3s.Lattice((4, 4, 1, 1))
    F = [su3s.Field(lat) for _ in range(2)]

    def full(depth):   # a balanced tree of sums holds a register per level and leaf
        if depth == 0:
            return F[0].expr()
        return full(depth - 1).adj() * full(depth - 1)

    z = F[0].like()
    with pytest.raises(su3s.Su3sError) as err:
        su3s.evaluate(z, full(5))
    assert err.value.code == 6
