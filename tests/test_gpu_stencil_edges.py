"""Neighbour terms at the edges of their kernels: out-of-range and non-finite inputs (the site is
computed in native FP64 then, so it equals that arithmetic's kernel), blocks with a ragged tail,
extents of 1 and 2 (a site that is its own neighbour), and mixed layouts of the fields."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

SEED = synth.SEED_BASE + 43
SPECIALS = [np.nan, np.inf, -np.inf, 1e40, -3e300, 2.0 ** 59, -(2.0 ** 57), 1e-40, 5e-324, -0.0]


@pytest.fixture(scope="module")
def su3s(gpu_lib):
    return gpu_lib


def plant(arr, first, stride):
    flat = arr.reshape(arr.shape[0], -1)
    for k, val in enumerate(SPECIALS):
        flat[(first + stride * k) % arr.shape[0], (5 * k + 1) % flat.shape[1]] = val


def field(su3s, lat, kind, nmu, arr, layout=0, block=64):
    f = su3s.Field(lat, kind, nmu, su3s.F64, layout, block)
    f.upload(arr)
    return f


def assert_like_native(got, ref, tol):
    """The same NaNs and infinities, finite values within tol of max(1, |ref|)."""
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(got[inf], ref[inf])
    fin = np.isfinite(ref)
    with np.errstate(invalid="ignore", over="ignore"):
        assert (np.abs(got - ref)[fin] <= tol * np.maximum(1.0, np.abs(ref[fin]))).all()


def test_dslash_with_special_inputs(su3s):
    dims = (6, 5, 7, 9)
    v = synth.volume(dims)
    u, x = synth.su3(SEED, 0, 4 * v), synth.gauss_vector(SEED, 1, 4 * v)
    plant(u, 40, 401)
    plant(x, 333, 577)
    lat = su3s.Lattice(dims)
    U = field(su3s, lat, su3s.MATRIX, 4, u)
    P = field(su3s, lat, su3s.VECTOR, 4, x)
    z, zf = P.like(), P.like()
    su3s.dslash(z, U, P, su3s.MATH_DF32)
    su3s.dslash(zf, U, P, su3s.MATH_F64)
    # inputs up to 2^57 beside normal ones: the pair arithmetic's 1.6e-12 of unit
    # operands, times the largest of the site (within a site's outputs)
    assert_like_native(z.download().reshape(v, -1), zf.download().reshape(v, -1), 1.6e-12 * 64)


@pytest.mark.parametrize("dims", [(2, 1, 3, 43), (5, 51, 1, 1), (127, 1, 1, 1), (129, 2, 1, 1),
                                  (4, 4, 4, 8)])
def test_dslash_ragged_blocks_and_mixed_layouts(su3s, dims):
    v = synth.volume(dims)
    u = synth.su3(SEED, 2, 4 * v)
    x = synth.gauss_vector(SEED, 3, 4 * v)
    x /= np.abs(x).max()
    lat = su3s.Lattice(dims)
    U = field(su3s, lat, su3s.MATRIX, 4, u, su3s.AOSOA, 32)
    P = field(su3s, lat, su3s.VECTOR, 4, x)
    z = su3s.Field(lat, su3s.VECTOR, 4, su3s.F64, su3s.AOSOA, 4)
    su3s.dslash(z, U, P)
    ref = oracle.dslash(u, x.reshape(v, 4, 3, 2), dims).reshape(4 * v, 3, 2)
    assert np.abs(z.download() - ref).max() < 1.6e-12


def test_vector_hop_with_special_inputs(su3s):
    dims = (6, 5, 7, 9)
    v = synth.volume(dims)
    u, x = synth.su3(SEED, 4, 4 * v), synth.gauss_vector(SEED, 5, v)
    plant(u, 40, 401)
    plant(x, 333, 137)
    lat = su3s.Lattice(dims)
    U = field(su3s, lat, su3s.MATRIX, 4, u)
    X = field(su3s, lat, su3s.VECTOR, 1, x)
    z, zf = X.like(), X.like()
    su3s.hop(z, U, X, su3s.MATH_DF32)
    su3s.hop(zf, U, X, su3s.MATH_F64)
    # 8 products of unit operands within 8e-13; operands up to 6 in size beside the planted ones
    assert_like_native(z.download(), zf.download(), 8e-13 * 64)


@pytest.mark.parametrize("dims", [(2, 1, 3, 43), (5, 51, 1, 1), (127, 1, 1, 1), (129, 2, 1, 1)])
def test_vector_hop_ragged_blocks_and_mixed_layouts(su3s, dims):
    v = synth.volume(dims)
    u, x = synth.su3(SEED, 6, 4 * v), synth.gauss_vector(SEED, 7, v)
    x /= np.abs(x).max()
    lat = su3s.Lattice(dims)
    U = field(su3s, lat, su3s.MATRIX, 4, u, su3s.AOSOA, 32)
    X = field(su3s, lat, su3s.VECTOR, 1, x)
    z = su3s.Field(lat, su3s.VECTOR, 1, su3s.F64, su3s.AOSOA, 4)
    su3s.hop(z, U, X)
    assert np.abs(z.download() - oracle.hop(u, x, dims)).max() < 8e-13


@pytest.mark.parametrize("dims", [(16, 16, 16, 32), (17, 16, 32, 48), (96, 64, 32, 33)])
@pytest.mark.parametrize("math", ["MATH_F64", "MATH_DF32", "MATH_FX"])
def test_neighbour_terms_over_the_waves_of_a_launch(su3s, dims, math):
    """One wave of blocks, several, and more sites than 32 waves take (threads then take several):
    the hopping terms on vectors and matrices at sites spread over the lattice against their sums in
    FP64, and the Wilson term on every site against another arithmetic's launch."""
    lat = su3s.Lattice(dims)
    g = torch.Generator(device="cuda").manual_seed(29)
    fill = lambda f: f.tensor.copy_(torch.rand(f.tensor.shape, dtype=torch.float64, device="cuda", generator=g) - 0.5)
    U = su3s.Field(lat, su3s.MATRIX, 4)
    fill(U)
    lx, ly, lz, lt = dims
    V = lx * ly * lz * lt
    rng = np.random.default_rng(5)
    sites = np.unique(np.r_[0, V - 1, V // 2, rng.integers(0, V, 200)])
    crd = np.stack([sites % lx, sites // lx % ly, sites // (lx * ly) % lz, sites // (lx * ly * lz)], 1)

    def at(field, index, mu=0):   # (n, rows, cols) complex of a structure-of-arrays field
        nc = {su3s.MATRIX: 9, su3s.VECTOR: 3}[field.kind]
        t = field.tensor.view(field.nmu * nc, -1, 2)[mu * nc:(mu + 1) * nc, torch.as_tensor(index, device="cuda")]
        return torch.view_as_complex(t.contiguous()).T.cpu().numpy().reshape(len(index), 3, nc // 3)

    def neighbour(mu, sign):
        c = crd.copy()
        c[:, mu] = (c[:, mu] + sign) % dims[mu]
        return c[:, 0] + lx * (c[:, 1] + ly * (c[:, 2] + lz * c[:, 3]))

    for kind in (su3s.VECTOR, su3s.MATRIX):
        v = su3s.Field(lat, kind)
        fill(v)
        z = v.like()
        su3s.hop(z, U, v, getattr(su3s, math))
        ref = 0
        for mu in range(4):
            n, p = neighbour(mu, 1), neighbour(mu, -1)
            ref = ref + at(U, sites, mu) @ at(v, n) + np.conj(np.swapaxes(at(U, p, mu), 1, 2)) @ at(v, p)
        # 5.7e-14 is the pair arithmetic's error for 6 real products of unit size; here 48 below 1/4
        assert np.abs(at(z, sites) - ref).max() < 1.2e-13
    # the Wilson term (48 real products below 1/2) against native FP64's launch
    psi = su3s.Field(lat, su3s.VECTOR, 4)
    fill(psi)
    z, w = psi.like(), psi.like()
    su3s.dslash(z, U, psi, getattr(su3s, math))
    su3s.dslash(w, U, psi, su3s.MATH_DF32 if math == "MATH_F64" else su3s.MATH_F64)
    assert ((z.tensor - w.tensor).view(12, -1, 2)[:, :V].abs().max() < 2.4e-13).item()
