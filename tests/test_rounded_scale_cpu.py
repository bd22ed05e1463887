"""The FP32 scale of a new basis vector, 1/sqrt(h + l) (csrc/rotations.cuh), compiled for
the host, against extended precision."""
import subprocess

import numpy as np
import pytest

from paper_1507_05925_gb300 import build

SRC = r"""
#include <stdio.h>
#include "rotations.cuh"
int main() {
  float x[2];
  while (fread(x, 4, 2, stdin) == 2) {
    const float r = bie::rsqrt_rounded(x[0], x[1]);
    fwrite(&r, 4, 1, stdout);
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("scale")
    (d / "scale.cu").write_text(SRC)
    exe = d / "scale"
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, str(d / "scale.cu"), "-o", str(exe)],
                   check=True)

    def run(h, low):
        data = np.stack([h, low], 1).astype(np.float32).tobytes()
        return np.frombuffer(subprocess.run([str(exe)], input=data, capture_output=True, check=True).stdout, np.float32)

    return run


def test_scale_is_rounded_once(program):
    rng = np.random.default_rng(9)
    n = 400_000
    h = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-100, 100, n)).astype(np.float32)
    low = (rng.uniform(-0.5, 0.5, n) * np.spacing(h)).astype(np.float32)
    low[: n // 2] = 0.0
    got = program(h, low)
    exact = 1.0 / np.sqrt(h.astype(np.longdouble) + low.astype(np.longdouble))
    err = np.abs(got.astype(np.longdouble) - exact) / np.spacing(exact.astype(np.float32))
    # the Newton step's own error: 3/8 e^2 with |e| <= 2^-22, and the rounding of its last
    # product, 2^-24 |e|/2, both below 2^-15 of an ulp
    assert float(err.max()) <= 0.5 + 2.0 ** -15


def test_scale_at_the_ends_of_the_range(program):
    h = np.array([2.0 ** -140, 2.0 ** -126, 2.0 ** 127, np.finfo(np.float32).max], dtype=np.float32)
    got = program(h, np.zeros_like(h))
    exact = 1.0 / np.sqrt(h.astype(np.float64))
    assert np.all(np.abs(got - exact) <= 2.0 ** -22 * exact)
