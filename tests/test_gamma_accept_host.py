"""The FP32 short cut of the Gamma draws' acceptance test decides as FP64 does (host code, no GPU)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_19723_gb300", "csrc")

PROGRAM = r"""
#include "gamma_accept.cuh"
#include <cstdio>
int main() {
    double q[3];
    while (std::fread(q, sizeof(double), 3, stdin) == 3) {
        const double d = q[0] - 1.0 / 3.0, c = 1.0 / sqrt(9.0 * d), t = 1.0 + c * q[1];
        std::putchar(bp::gamma_accept(q[1], t, c, d, q[2]) ? 1 : 0);
    }
}
"""


@pytest.mark.parametrize("shape", [1.0, 1.2, 1.5, 2.0, 6.0, 30.0, 100.0, 1e4, 1e8])
def test_the_fp32_decision_is_the_fp64_one(shape, tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "accept.cpp", tmp_path / "accept"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O2", "-D__host__=", "-D__device__=", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    rng = np.random.default_rng(5)
    d = shape - 1.0 / 3.0
    c = 1.0 / np.sqrt(9.0 * d)
    # normal draws, and draws close to t = 0 (where they reach it: |g| < 6.8 for 32-bit uniforms)
    g = np.concatenate([rng.normal(size=60000), -(1.0 - 10.0 ** rng.uniform(-8, 0, 60000)) / c])
    g = g[(np.abs(g) < 6.8) & (1.0 + c * g > 0.0)]
    t = 1.0 + c * g
    side = 0.5 * g * g + d - d * t ** 3 + 3.0 * d * np.log(t)
    # uniforms at the boundary, further off than 64 bits can err
    off = 10.0 ** rng.uniform(-9, 0, g.size) * (1.0 + d) * rng.choice([-1.0, 1.0], g.size)
    keep = (side + off > -32 * np.log(2.0)) & (side + off < 0.0)
    g, want, u = g[keep], off[keep] < 0.0, np.exp(side[keep] + off[keep])
    out = subprocess.run([str(exe)], input=np.stack([np.full(g.size, shape), g, u], axis=1).tobytes(), capture_output=True,
                         check=True).stdout
    got = np.frombuffer(out, np.uint8).astype(bool)
    assert got.size == g.size > 1000
    assert np.array_equal(got, want)
