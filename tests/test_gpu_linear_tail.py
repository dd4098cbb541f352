"""a*b*c + s*d in the fixed-point and the pair arithmetic, whose last term is added in FP64: every data
movement and a batch give the same bits, and the result is within the product's own error and the
rounding of the sum, with elements of d far above and far below the rest of their object and of the
product."""
import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import lattice_fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def su3s(gpu_lib):
    return gpu_lib


@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (31, 1, 1, 1), (33, 1, 1, 1), (6, 5, 7, 3)])
@pytest.mark.parametrize("s", [0.5, -1.0 / 3.0, 0.0, 2.0 ** -70, 2.0 ** 30])
@pytest.mark.parametrize("layout,block", [("SOA", 64), ("AOSOA", 32)])
@pytest.mark.parametrize("math,err", [("MATH_FX", 1.7e-15), ("MATH_DF32", 6e-14)])
def test_linear_last_term(su3s, dims, s, layout, block, math, err):
    lat = su3s.Lattice(dims)
    f = lattice_fields(dims, synth.SEED_BASE + 31, names=("a", "b", "c", "d"))
    rng = np.random.default_rng(41)
    f["d"] = f["d"] * 2.0 ** rng.integers(-60, 37, f["d"].shape)
    x = {}
    for k in "abcd":
        x[k] = su3s.Field(lat, layout=getattr(su3s, layout), block=block)
        x[k].upload(f[k])
    tree = lambda: x["a"] * x["b"] * x["c"] + s * x["d"].expr()
    got = []
    for pipe in range(-1, 5):
        z = x["a"].like()
        su3s.set_pipeline(pipe)
        try:
            su3s.evaluate(z, tree(), getattr(su3s, math))
        finally:
            su3s.set_pipeline(-1)
        got.append(z.download())
    batch, z = su3s.Batch(), x["a"].like()
    batch.add(z, tree())
    batch.build(getattr(su3s, math))
    batch.launch()
    torch.cuda.synchronize()
    got.append(z.download())
    assert all(np.array_equal(g, got[0]) for g in got[1:])
    # the product alone is within 1.6e-15 (fixed point) or 5.7e-14 (pairs) for unitary factors (the
    # error study); then its conversion and the rounding of the sum.  The expected sum is formed in extended precision: the oracle would
    # round s*d and the sum, by up to 2^-52 |s d| itself
    ref = oracle.eval_tree(("mul", ("mul", ("leaf", "a"), ("leaf", "b")), ("leaf", "c")), f)
    ref = ref + np.longdouble(s) * f["d"].astype(np.longdouble)
    assert (np.abs(got[0] - ref) <= err + 2.0 ** -52 * np.abs(s * f["d"])).all()
