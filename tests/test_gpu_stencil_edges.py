"""Neighbour terms at the edges of their kernels: out-of-range and non-finite inputs (the site is
computed in native FP64 then, so it equals that arithmetic's kernel), blocks with a ragged tail,
extents of 1 and 2 (a site that is its own neighbour), and mixed layouts of the fields."""
import numpy as np
import pytest

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
