"""The mixed-radix passes of the 3-D box transforms (csrc/fft_mixed.h) against numpy's FFT, on the CPU.

Lengths cover every radix as first, middle and last pass, two to four passes, and the largest sizes.
Bars: 8 rounding errors a pass, relative to the largest output (float64: 1e-14, float: 2e-6)."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_03608_gb300", "csrc")


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    exe = tmp_path_factory.mktemp("fftm") / "fft_mixed_check"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "fft_mixed_check.cpp"),
                           "-o", str(exe)])
    return str(exe)


@pytest.mark.parametrize("n", [4, 16, 20, 28, 36, 60, 160, 168, 216, 252, 256, 288, 432, 490, 500, 512, 686, 800, 864,
                               882, 896, 972, 1000, 1024, 1372, 2048])
def test_mixed_radix_transform(prog, n):
    rng = np.random.default_rng(n)
    z = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    inp = "%d\n" % n + "\n".join("%.17g" % v for v in np.column_stack([z.real, z.imag]).ravel())
    out = subprocess.run([prog], input=inp, capture_output=True, text=True, check=True).stdout.split()
    passes, lanes = int(out[0]), int(out[1])
    assert 2 <= passes <= 4 and lanes * 10 >= n
    v = np.array([float(x) for x in out[2:]]).reshape(3, n, 2)
    got = v[..., 0] + 1j * v[..., 1]
    fwd, inv = np.fft.fft(z), np.fft.ifft(z) * n
    assert np.max(np.abs(got[0] - fwd)) <= 1e-14 * np.max(np.abs(fwd))
    assert np.max(np.abs(got[1] - inv)) <= 1e-14 * np.max(np.abs(inv))
    assert np.max(np.abs(got[2] - fwd)) <= 2e-6 * np.max(np.abs(fwd))


@pytest.mark.parametrize("n", [11, 22, 13 * 16, 2])
def test_other_lengths_are_refused(prog, n):
    inp = "%d\n" % n + "\n".join(["0"] * (2 * n))
    assert subprocess.run([prog], input=inp, capture_output=True, text=True, check=True).stdout.split()[0] == "0"
