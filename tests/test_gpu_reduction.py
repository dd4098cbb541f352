"""The field reduction at the edges of its grid: fewer sites than a block, a site more than a wave of
blocks, padded tiles that must not count, several links, every field kind, both layouts; and the same
result under stream capture."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def su3s(gpu_lib):
    return gpu_lib


@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (3, 5, 7, 2), (256, 1, 1, 1), (257, 1, 1, 1),
                                  (77825, 1, 1, 1), (31, 33, 8, 35)])
@pytest.mark.parametrize("kind,nmu", [("MATRIX", 1), ("MATRIX", 3), ("VECTOR", 1), ("VECTOR", 8), ("REAL", 1)])
@pytest.mark.parametrize("layout,block", [("SOA", 64), ("AOSOA", 32)])
def test_reduction_edges(su3s, dims, kind, nmu, layout, block):
    lat = su3s.Lattice(dims)
    rng = np.random.default_rng(17)
    x = su3s.Field(lat, getattr(su3s, kind), nmu, su3s.F64, getattr(su3s, layout), block)
    y = x.like()
    h = [rng.standard_normal(x.canonical_shape) for _ in range(2)]
    for f, v in zip((x, y), h):
        f.upload(v)
    ones = x.like()
    ones.upload(np.ones(x.canonical_shape))
    for f in (x, y):
        f.tensor[ones.tensor == 0] = float("nan")
    prod = (h[0] * h[1]).ravel()
    # every sum is a chain: a thread's products (9 fused terms per site), 5 + 7 block steps, 3 + 12
    # steps of the final block; 64 more for the expected value's own pairwise sum
    per_thread = 9 * -(-lat.volume // (256 * (304 // nmu)))
    bound = 2.0 ** -53 * (per_thread + 96) * float(np.sum(np.abs(prod)))
    got = su3s.redot(x, y).item()
    assert abs(got - float(np.sum(prod))) <= bound
    assert su3s.redot(x, y).item() == got
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        su3s.redot(x, y, out)
    g.replay()
    torch.cuda.synchronize()
    assert out.item() == got
