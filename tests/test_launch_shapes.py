"""Launch shapes that are plain host arithmetic, and what runs with them."""
import os
import shutil
import subprocess

import pytest
import torch

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PAIR_SUM = r"""
#include <stdio.h>
#include "internal.h"
int main() {
  for (int sms = 2; sms <= 264; ++sms)
    for (int nmu = 1; nmu <= 8; ++nmu) printf("%d %d %d\n", sms, nmu, su3s::pair_sum_blocks(sms, nmu));
  return 0;
}
"""


def test_one_block_per_sm_for_two_products_in_one_launch(tmp_path):
    """Every block of the one-launch reverse mode has an SM to itself (as far as two blocks per link,
    one for each product, allow), and no more than two SMs per link stay without one."""
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if cxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    src, exe = tmp_path / "shapes.cpp", str(tmp_path / "shapes")
    src.write_text(PAIR_SUM)
    subprocess.check_call([cxx, "-std=c++17", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_1710_09409_gb300", "csrc"),
                           "-I", os.path.join(cuda, "include"), str(src), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    for sms, nmu, nb in (map(int, line.split()) for line in out.splitlines()):
        assert nb >= 2 and nb % 2 == 0
        assert nb * nmu <= max(sms, 2 * nmu)
        assert sms - nb * nmu < 2 * nmu


@pytest.mark.gpu
@pytest.mark.parametrize("nmu,tiles", [(2, 1217), (5, 487), (8, 305)])
@pytest.mark.parametrize("skip", [None, 1])
def test_reverse_mode_of_a_sum_of_several_links(gpu_lib, nmu, tiles, skip):
    """Link counts that do not divide the SMs: the gradients of the fused pass."""
    su3s = gpu_lib
    lat = su3s.Lattice((32, tiles, 1, 1))
    g = torch.Generator(device="cuda").manual_seed(17)
    f = [su3s.Field(lat, su3s.MATRIX, nmu) for _ in range(5)]
    for x in f:
        x.pack(torch.randn(x.canonical_shape, dtype=torch.float64, device="cuda", generator=g))
    a, b, c, d, w = f
    got = []
    for mode in (-1, 0):
        out = [a.like() for _ in range(4)]
        su3s.set_adjoint_split(mode)
        try:
            su3s.eval_adjoint(a * b + c * d, w, [None if k == skip else x for k, x in enumerate(out)])
        finally:
            su3s.set_adjoint_split(-1)
        got.append(out)
    for k in range(4):
        assert k == skip or torch.equal(got[0][k].unpack(), got[1][k].unpack()), k
    assert su3s.device_error() == 0
