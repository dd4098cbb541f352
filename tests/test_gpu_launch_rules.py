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


@pytest.mark.parametrize("tiles,nmu,layout,block", [(2431, 1, 0, 64), (2432, 1, 0, 64), (2433, 1, 1, 32),
                                                    (4865, 1, 0, 64), (811, 3, 0, 64)])
@pytest.mark.parametrize("skip", [None, 0, 3])
def test_reverse_mode_of_a_sum_in_one_launch(su3s, tiles, nmu, layout, block, skip):
    """Both products side by side (from 8 units of two tiles per SM on): the
    gradients of the fused pass, an odd number of tiles and gradients that are not wanted among
    them."""
    lat = su3s.Lattice((32, tiles, 1, 1))
    g = torch.Generator(device="cuda").manual_seed(13)
    f = [su3s.Field(lat, su3s.MATRIX, nmu, su3s.F64, layout, block) for _ in range(5)]
    for x in f:
        x.pack(torch.randn(x.canonical_shape, dtype=torch.float64, device="cuda", generator=g))
    a, b, c, d, w = f
    got = {}
    for mode in (-1, 0):
        out = [a.like() for _ in range(4)]
        for x in out:
            x.tensor.fill_(7.0)
        su3s.set_adjoint_split(mode)
        try:
            su3s.eval_adjoint(a * b + c * d, w, [None if k == skip else x for k, x in enumerate(out)])
        finally:
            su3s.set_adjoint_split(-1)
        got[mode] = out
    for k in range(4):
        if k == skip:
            assert got[-1][k].tensor.eq(7.0).all()
        else:
            assert torch.equal(got[-1][k].unpack(), got[0][k].unpack()), k
    assert su3s.device_error() == 0
