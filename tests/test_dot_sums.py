"""The sum of a warp's FP32 dot-product partials (Sum3): compiled for the host and run over the
steps a warp takes, against the exact sum.  The result is one FP64 number, so half a unit of its
last place (2^-53) is rounding; the rest of the three-part sum is below 2^-68.
"""
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2403_19854_gb300")

SOURCE = r"""
#include <cstdio>
#include "rk_common.cuh"
int main() {
  float v[32][4];
  for (;;) {
    for (auto& l : v)
      for (float& x : l)
        if (fread(&x, 4, 1, stdin) != 1) return 0;
    rk::Sum3 d[32];
    for (int l = 0; l < 32; ++l) {
      d[l] = rk::Sum3{v[l][0], v[l][1], 0.0f};
      d[l].merge(rk::Sum3{v[l][2], v[l][3], 0.0f});
    }
    for (int o = 16; o > 0; o >>= 1)
      for (int l = 0; l < o; ++l) d[l].merge(d[l + o]);
    const double s = d[0].value();
    fwrite(&s, 8, 1, stdout);
  }
}
"""


def test_warp_sum_is_no_less_accurate_than_fp64(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "sums.cu", tmp_path / "sums"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)], check=True)
    rng = np.random.default_rng(3)
    n = 2000
    s = rng.random((n, 32, 2)).astype(np.float32)
    s[n // 2:] *= np.float32(10.0) ** rng.uniform(-6, 6, (n - n // 2, 32, 2)).astype(np.float32)
    s[n - 200:] *= rng.choice(np.array([-1.0, 1.0], np.float32), (200, 32, 2))
    c = (s * rng.uniform(-3e-7, 3e-7, s.shape)).astype(np.float32)
    v = np.stack([s[..., 0], c[..., 0], s[..., 1], c[..., 1]], axis=-1).astype(np.float32)
    out = subprocess.run([str(exe)], input=v.tobytes(), stdout=subprocess.PIPE, check=True).stdout
    got = np.frombuffer(out, dtype=np.float64)
    assert got.size == n
    for k in range(n):
        exact = sum(Fraction(float(x)) for x in v[k].reshape(-1))
        scale = math.fsum(abs(float(x)) for x in v[k].reshape(-1))
        err = abs(Fraction(float(got[k])) - exact)
        assert err <= Fraction(2) ** -53 * abs(exact) * Fraction(1001, 1000) + Fraction(2) ** -68 * Fraction(scale), k
