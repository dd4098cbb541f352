"""Canonical array <-> field on the GPU (tiles of sites through shared memory): every count of
elements per site, ragged tiles, pads and arrays that are only 8-byte aligned, bit for bit; and
the projection to SU(3) at the edges of its fast path, against the CPU oracle."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

SEED = synth.SEED_BASE + 41


@pytest.fixture(scope="module")
def su3s(gpu_lib):
    return gpu_lib


def in_field_order(x, f):
    """Canonical (V, nmu, ncomp, 2) values in the field's order, pads zero."""
    v, nmu, nc, _ = x.shape
    n = f.tensor.numel() // (nmu * nc * 2)
    p = torch.zeros((n, nmu, nc, 2), dtype=x.dtype, device=x.device)
    p[:v] = x
    b = f.block if f.block else n
    return p.view(n // b, b, nmu, nc, 2).permute(0, 2, 3, 1, 4).reshape(-1)


@pytest.mark.parametrize("layout,block", [(0, 0), (1, 4), (1, 32), (1, 1024)])
@pytest.mark.parametrize("kind,nmu", [("matrix", 1), ("matrix", 3), ("matrix", 4), ("matrix", 8),
                                      ("vector", 1), ("vector", 4), ("real", 1), ("real", 3)])
@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (31, 1, 1, 1), (4, 4, 2, 1), (11, 3, 1, 1),
                                  (257, 1, 1, 1), (7, 5, 3, 4)])
def test_tiles_are_exact(su3s, dims, kind, nmu, layout, block):
    lat = su3s.Lattice(dims)
    K = {"matrix": su3s.MATRIX, "vector": su3s.VECTOR, "real": su3s.REAL}[kind]
    f = su3s.Field(lat, K, nmu, su3s.F64, layout, block or 64)
    n = int(np.prod(f.canonical_shape))
    g = torch.Generator(device="cuda").manual_seed(7)
    buf = torch.randn(n + 1, dtype=torch.float64, device="cuda", generator=g)
    for off in (0, 1):   # 16-byte aligned, and 8-byte aligned only
        x = buf[off:off + n].view(f.canonical_shape)
        f.tensor.fill_(float("nan"))
        f.pack(x)
        w = {"matrix": 9, "vector": 3}.get(kind)
        if w:
            assert torch.equal(f.tensor, in_field_order(x.reshape(-1, nmu, w, 2), f))
        assert torch.equal(f.unpack(), x)
        out = torch.full((n + 2,), 5.0, dtype=torch.float64, device="cuda")
        rc = su3s.load().su3s_field_unpack(f._h, ctypes.c_void_p(out[off:].data_ptr()),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        assert torch.equal(out[off:off + n], x.reshape(-1))
        assert out[n + off:].eq(5.0).all() and out[:off].eq(5.0).all()


def test_projection_at_the_edges_of_the_fast_path(su3s):
    """Scales whose squares overflow or vanish, negative real determinants (the cube root's branch
    cut), nearly dependent rows, and matrices without a projection (zero, NaN)."""
    n = 64
    u = synth.su3(SEED, 0, n) + 0.05 * synth.gauss_matrix(SEED, 1, n)
    q = np.linalg.qr(np.random.default_rng(3).standard_normal((n, 3, 3)))[0]
    q *= -np.sign(np.linalg.det(q))[:, None, None]          # real, determinant -1
    real = np.stack([q, np.zeros_like(q)], -1)
    close = u.copy()
    close[:, 1] = close[:, 0] + 1e-3 * close[:, 1]
    cases = {"unit": u, "2^120": u * 2.0 ** 120, "2^-120": u * 2.0 ** -120, "2^480": u * 2.0 ** 480,
             "2^-480": u * 2.0 ** -480, "det -1": real, "close rows": close}
    lat = su3s.Lattice((4, 4, 4, 1))
    for name, x in cases.items():
        f = su3s.Field(lat)
        f.upload(x)
        su3s.reunitarize(f, f)                              # in place
        # rows 1e-3 apart: the rounding of the inputs' difference, times 1e3
        tol = 1e-12 if name == "close rows" else 1e-14
        assert np.abs(f.download() - oracle.reunitarize(x)).max() < tol, name
    x = u.copy()
    x[5] = 0.0
    x[9, 2, 1, 0] = np.nan
    f = su3s.Field(lat)
    f.upload(x)
    su3s.reunitarize(f, f)
    got, ref = f.download(), oracle.reunitarize(x)
    assert np.array_equal(np.isnan(got).any((1, 2, 3)), np.isnan(ref).any((1, 2, 3)))
    fine = ~np.isnan(ref).any((1, 2, 3))
    assert np.abs(got - ref)[fine].max() < 1e-14


@pytest.mark.parametrize("ratio", [0.0, 0.24, 0.2499, 0.2501, 0.26, 1.0, 1e3, 1e6])
def test_projection_with_rows_near_each_other(su3s, ratio):
    """Row 1 = ratio (a phase of row 0) + a unit row orthogonal to it, around the part from which a
    second sweep is taken (a quarter in norm) and far past it: special unitary to rounding, and the
    rows of the definition to the rounding of the input, which the ratio magnifies."""
    rng = np.random.default_rng(23)
    n = 700
    q = np.linalg.qr(rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3)))[0]
    ph = np.exp(2j * np.pi * rng.random((n, 1)))
    m = np.stack([3.0 * q[:, :, 0], 0.5 * (q[:, :, 1] + ratio * ph * q[:, :, 0]),
                  q[:, :, 2] + 0.3 * q[:, :, 0] - 0.2j * q[:, :, 1]], 1)
    x = np.stack([m.real, m.imag], -1)
    f = su3s.Field(su3s.Lattice((n, 1, 1, 1)))
    f.upload(x)
    su3s.reunitarize(f, f)
    got = f.download()
    u = got[..., 0] + 1j * got[..., 1]
    # 2^-53 times: norms and products of 3 complex terms (16), the phase (8), twice for two rows
    eps = 2.0 ** -53 * 48
    assert np.abs(u @ np.conj(np.swapaxes(u, 1, 2)) - np.eye(3)).max() < eps
    assert np.abs(np.linalg.det(u) - 1).max() < 2 * eps
    assert np.abs(got - oracle.reunitarize(x)).max() < eps * (1 + ratio)
