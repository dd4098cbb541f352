"""Default launches around the sizes where their shape changes: the staged result equals the
plain-load kernel's, value by value, on every site (pair arithmetic, FP64 storage)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def su3s(gpu_lib):
    return gpu_lib


def trees(f):
    a, b, c, d = f
    return {"commutator": lambda: a * b - b * a,
            "anticommuting adjoint": lambda: a.adj() * b - b * a.adj(),
            "sum": lambda: a * b + c * d,
            "nested": lambda: a * b * c + 0.5 * d}


def tiles():
    """Counts of 32-site tiles: around one warp, one block and one wave of blocks per SM, and
    around the 40 and 96 tiles per SM of the default shapes."""
    return [1, 2, "1sm-1", "1sm", "1sm+1", "2sm+1", "4sm-1", "8sm+1", "40sm-1", "40sm", "96sm-1", "96sm"]


@pytest.mark.parametrize("count", tiles())
def test_default_launch_equals_plain_loads(su3s, count):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if isinstance(count, str):
        k, rest = count.split("sm")
        count = int(k) * sms + int(rest or 0)
    lat = su3s.Lattice((31 if count == 1 else 32, count, 1, 1))   # 31: a ragged tail
    g = torch.Generator(device="cuda").manual_seed(11)
    f = [su3s.Field(lat) for _ in range(4)]
    for x in f:
        x.pack(torch.randn(x.canonical_shape, dtype=torch.float64, device="cuda", generator=g))
    z, ref = f[0].like(), f[0].like()
    for name, make in trees(f).items():
        z.tensor.fill_(float("nan"))
        su3s.evaluate(z, make())
        su3s.set_pipeline(su3s.PIPE_PLAIN)
        try:
            su3s.evaluate(ref, make())
        finally:
            su3s.set_pipeline(su3s.PIPE_AUTO)
        assert torch.equal(z.tensor, ref.tensor), name
    assert su3s.device_error() == 0


def test_commutator_in_place(su3s):
    """The destination is a leaf, with many tiles per warp of the queue."""
    lat = su3s.Lattice((32, 30, 20, 26))
    g = torch.Generator(device="cuda").manual_seed(12)
    a, b = su3s.Field(lat), su3s.Field(lat)
    for x in (a, b):
        x.pack(torch.randn(x.canonical_shape, dtype=torch.float64, device="cuda", generator=g))
    z = a.like()
    su3s.evaluate(z, a.adj() * b - b * a.adj())
    su3s.evaluate(a, a.adj() * b - b * a.adj())
    assert torch.equal(a.tensor, z.tensor)
