"""What tuning the reverse mode of a sum of two products reports: the one-launch form (variant 15)
only where such a launch can run."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def su3s(gpu_lib):
    return gpu_lib


def tuned(su3s, dims, make, math=0):
    lat = su3s.Lattice(dims)
    g = torch.Generator(device="cuda").manual_seed(19)
    f = [su3s.Field(lat) for _ in range(9)]
    for x in f[:5]:
        x.pack(torch.randn(x.canonical_shape, dtype=torch.float64, device="cuda", generator=g))
    return su3s.tune_adjoint(make(*f[:4]), f[4], f[5:], math)


SUM = {"sum": lambda a, b, c, d: a * b + c * d}
OTHER = {"difference": lambda a, b, c, d: a * b - c * d, "scaled": lambda a, b, c, d: 2.0 * (a * b) + 0.5 * (c * d)}


@pytest.mark.parametrize("tree", list(OTHER))
@pytest.mark.parametrize("x", range(17, 23))
def test_no_such_kernel_for_other_trees(su3s, tree, x):
    assert tuned(su3s, (x, 16, 16, 16), OTHER[tree])[2] != 15


@pytest.mark.parametrize("x,math", [(5, 0), (6, 0), (7, 0), (8, 0), (9, 0), (10, 0), (18, 1), (19, 3)])
def test_not_below_its_size_or_in_other_arithmetics(su3s, x, math):
    assert tuned(su3s, (x, 8, 8, 16) if math == 0 else (x, 16, 16, 16), SUM["sum"], math)[2] != 15


def test_where_it_runs(su3s):
    th, bps, variant, ms = tuned(su3s, (24, 24, 24, 24), SUM["sum"])
    assert variant < 15 or (variant, th, bps) == (15, 256, 1)
    assert ms > 0
