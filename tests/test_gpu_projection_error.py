"""Rounding error of the projection to SU(3) against extended precision, by kind of input: no larger
than that of Gram-Schmidt's two sweeps in FP64, which it stands for."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

# rms error of the two sweeps with fused multiply-adds, 65,536 matrices of each kind
SWEEPS = {"projected, rounded to FP32": 4.31e-17, 1e-6: 4.48e-17, 1e-4: 4.49e-17, 1e-3: 4.49e-17, 1e-2: 4.50e-17,
          0.1: 4.52e-17}


def project(x):
    """The definition in extended precision."""
    m = x.astype(np.longdouble)
    m, rows = m[..., 0] + 1j * m[..., 1], []
    for i in range(3):
        r = m[:, i]
        for _ in range(3):
            for p in rows:
                r = r - (np.conj(p) * r).sum(1, keepdims=True) * p
        rows.append(r / np.sqrt((np.abs(r) ** 2).sum(1, keepdims=True)))
    det = (rows[0] * np.cross(rows[1], rows[2])).sum(1)
    phase = np.arctan2(det.imag, det.real) / 3
    z = np.stack(rows, 1) * (np.cos(phase) - 1j * np.sin(phase))[:, None, None]
    return np.stack([z.real, z.imag], -1)


@pytest.mark.parametrize("noise", list(SWEEPS), ids=str)
def test_error_of_the_projection(gpu_lib, noise):
    su3s, dims = gpu_lib, (16, 16, 16, 4)
    v = synth.volume(dims)
    u = synth.su3(synth.SEED_BASE + 61, 0, v)
    if isinstance(noise, str):
        x = u.astype(np.float32).astype(np.float64)
    else:
        x = u + noise * np.random.default_rng(61).standard_normal(u.shape)
    f = su3s.Field(su3s.Lattice(dims))
    f.upload(x)
    su3s.reunitarize(f, f)
    err = np.sqrt(((f.download() - project(x)) ** 2).mean())
    # 16,384 matrices: the rms of so many is within 0.3% of that of many more
    assert err <= 1.003 * SWEEPS[noise], err
