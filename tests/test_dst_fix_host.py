"""The fixed-point DST-I phases of the float64 transform kernels, run on the
host one simulated thread at a time, against an 80-bit sine sum: index
decomposition, exchange, split pairing and scan for every tile length, and an
error no larger than that of the float64 pre-fold / FFT / running-sum
transform, over dense, smooth, sparse and widely scaled lines (no GPU
needed)."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import scipy.fft

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2104_05024_gb300", "csrc")
SIZES = [32, 64, 128, 256, 384, 512]


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("dstfix") / "dst_fix_host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fno-strict-aliasing", "-w", "-I", CSRC,
                    os.path.join(HERE, "host", "dst_fix_host.cpp"), "-o", exe], check=True)
    return exe


def run(exe, x, RS=33):
    x = np.ascontiguousarray(x)
    inp = np.array([x.shape[1] + 1, RS], np.int32).tobytes() + x.tobytes()
    return np.frombuffer(subprocess.run([exe], input=inp, capture_output=True, check=True).stdout).reshape(x.shape)


def reference(x):
    """sum_j x_j sin(pi j k / N) in 80-bit arithmetic."""
    N = x.shape[1] + 1
    j = np.arange(1, N)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    return x.astype(np.longdouble) @ np.sin(pi * (np.outer(j, j) % (2 * N)).astype(np.longdouble) / N)


def float64_transform(x):
    """The same algorithm (pre-fold, real FFT, running sum) in float64."""
    N = x.shape[1] + 1
    j = np.arange(1, N)
    y = np.zeros((x.shape[0], N))
    y[:, 1:] = np.sin(np.pi * j / N) * (x + x[:, ::-1]) + 0.5 * (x - x[:, ::-1])
    Y = np.conj(scipy.fft.rfft(y, axis=1))[:, :N // 2]
    R = Y.real.copy()
    R[:, 0] *= 0.5
    out = np.empty((x.shape[0], N))
    out[:, 0::2], out[:, 1::2] = Y.imag, np.cumsum(R, axis=1)
    return out[:, 1:]


def lines(kind, N):
    rng = np.random.default_rng(N)
    t = np.linspace(-1.0, 1.0, N + 1)[1:-1]
    if kind == "dense":
        return rng.standard_normal((32, N - 1))
    if kind == "smooth":
        c, w = rng.uniform(-0.6, 0.6, (32, 1)), rng.uniform(0.05, 0.2, (32, 1))
        return np.exp(-(t - c) ** 2 / (2 * w ** 2))
    if kind == "sparse":
        return (rng.random((32, N - 1)) < 0.03) * rng.standard_normal((32, N - 1)) * 1e5
    if kind == "spectrum":
        return rng.standard_normal((32, N - 1)) / np.arange(1, N) ** 3
    return rng.standard_normal((32, N - 1)) * 10.0 ** rng.uniform(-12, 0, (32, N - 1))


@pytest.mark.parametrize("N", SIZES)
@pytest.mark.parametrize("kind", ["dense", "smooth", "sparse", "spectrum", "wide"])
def test_error_at_most_that_of_the_float64_transform(harness, N, kind):
    x = lines(kind, N)
    ref = reference(x)
    err = [float(np.linalg.norm((y - ref).astype(float)) / np.linalg.norm(ref.astype(float)))
           for y in (run(harness, x), float64_transform(x))]
    assert err[0] <= err[1], err


@pytest.mark.parametrize("N", SIZES)
def test_extreme_columns(harness, N):
    """Zero columns, single values, constant sign (the largest sums), powers
    of two across the exponent range, infinities and NaN."""
    x = lines("dense", N)
    x[0] = 0.0
    x[1] = 0.0
    x[1, N // 2 - 1] = 3.0
    x[2] = np.copysign(1.0 - 2.0 ** -53, x[2])
    x[3] = 1.0 - 2.0 ** -53
    x[4] *= 2.0 ** 1000
    x[5] *= 2.0 ** -900
    x[6, 0] = np.inf
    x[7, N - 2] = np.nan
    x[8, 1::2] = 0.0
    y = run(harness, x, 32)
    assert np.all(y[0] == 0.0)
    assert np.all(np.isnan(y[6])) and np.all(np.isnan(y[7]))
    fine = [r for r in range(32) if r not in (0, 6, 7)]
    ref = reference(x[fine])
    err = np.abs((y[fine] - ref) / np.abs(ref).max(axis=1, keepdims=True)).max(axis=1)
    # one eps of the largest output per rounding level of the transform
    assert np.all(err < 2e-16 * np.log2(N) * 2), err
