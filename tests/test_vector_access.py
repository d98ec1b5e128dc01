"""Which vectors of a caller the H_eff.psi kernels use in place, and that the others give the same
result: the rule is host code (a small program compiled from its header), the calls run on a GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_1605_02611_gb300 as G
from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, require_gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1605_02611_gb300", "csrc")

# address, bytes, device memory, base and size of the allocation, used in place
RULE = [
    (4096, 800, 1, 4096, 800, 1),      # the whole allocation
    (4104, 792, 1, 4096, 800, 1),      # its tail
    (4104, 800, 1, 4096, 800, 0),      # 8 bytes too short
    (4100, 400, 1, 4096, 800, 0),      # not aligned to 8 bytes
    (4097, 400, 1, 4096, 800, 0),
    (4096, 400, 0, 4096, 800, 0),      # host memory, or another device's
    (4088, 400, 1, 4096, 800, 0),      # starts before the allocation
    (4896, 0, 1, 4096, 800, 1),        # an empty vector
    (4096, 1 << 63, 1, 4096, 800, 0),  # more than there is
]


def test_rule(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text('#include "vector_access.hpp"\n#include <cstdio>\nint main() {\n' + "".join(
        f'  std::printf("%d\\n", (int)gbdmrg::direct_vector({a}ULL, {b}ULL, {d}, {base}ULL, {size}ULL));\n'
        for a, b, d, base, size, _ in RULE) + "}\n")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout.split()
    assert [int(x) for x in out] == [r[-1] for r in RULE]


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 5])
def test_sigma_of_vectors_that_are_copied(precision):
    """Vectors at 4-byte boundaries and overlapping ones give what aligned device vectors give (FP64:
    the same sums; tensor cores: at most about 100 FP32 additions of 6e-8 per element in another
    order from call to call).  Host memory gives that or an error, as the copy has it."""
    torch = require_gpu()
    K, M, k = 8, 60, 3
    h, eri = synth.integrals(K, 31)
    bonds, T = synth.random_isometric_mps(K, K, 0, M, 32, k)
    ctx = context_with_mps(h, eri, K, 0, bonds, T)
    ctx.set_precision(precision)
    ctx.prepare(k)
    n = ctx.nnz
    v = torch.tensor(np.random.default_rng(33).normal(size=n), device="cuda")
    y = torch.empty_like(v)
    torch.cuda.synchronize()
    ctx.sigma_device(v.data_ptr(), y.data_ptr())
    ref = y.cpu().numpy()
    tol = 0.0 if precision == 0 else 1e-5 * np.abs(ref).max()

    def odd(t):  # the vector at an address that is 4 modulo 8
        b = torch.zeros(2 * n + 1, dtype=torch.float32, device="cuda")
        b[1:] = t.view(torch.float32)
        return b

    xo, yo = odd(v), odd(torch.zeros_like(v))
    pin_x, pin_y = v.cpu().pin_memory(), torch.zeros(n, dtype=torch.float64).pin_memory()
    both = torch.zeros(n + 8, dtype=torch.float64, device="cuda")
    both[:n] = v
    torch.cuda.synchronize()
    pairs = [(xo.data_ptr() + 4, y.data_ptr(), lambda: y),
             (v.data_ptr(), yo.data_ptr() + 4, lambda: yo[1:].clone().view(torch.float64)),
             (xo.data_ptr() + 4, yo.data_ptr() + 4, lambda: yo[1:].clone().view(torch.float64)),
             (both.data_ptr(), both.data_ptr() + 64, lambda: both[8:])]
    for xp, yp, got in pairs:
        y.zero_()
        yo.zero_()
        torch.cuda.synchronize()
        ctx.sigma_device(xp, yp)
        torch.cuda.synchronize()
        assert np.abs(got().cpu().numpy() - ref).max() <= tol
    ctx.sigma_timing(2, xo.data_ptr() + 4, yo.data_ptr() + 4)
    assert np.abs(yo[1:].clone().view(torch.float64).cpu().numpy() - ref).max() <= tol
    try:
        ctx.sigma_device(pin_x.data_ptr(), pin_y.data_ptr())
    except G.GbdmrgError as e:
        assert "ECUDA" in str(e)
    else:
        assert np.abs(pin_y.numpy() - ref).max() <= tol
    ctx.close()
