"""The fixed-point DST-I on the lines hardest for it, run on the host: a low
background with few values far above it (the largest value sets the unit of
the whole line, and the running sum collects what the roundings share), and
lines that drive the first level's sums to their bound (no GPU needed)."""
import numpy as np
import pytest
import scipy.fft

from test_dst_fix_host import SIZES, harness, reference, run  # noqa: F401

PI = np.longdouble("3.14159265358979323846264338327950288")


def float64_transform(x):
    """Pre-fold, real FFT, running sum in segments (8, or 16 of the longest
    lines) in float64, sines rounded from 80 bits."""
    N = x.shape[1] + 1
    L, G = N // 2, 16 if N >= 384 else 8
    s = np.sin(PI * np.arange(1, N).astype(np.longdouble) / N).astype(np.float64)
    y = np.zeros((x.shape[0], N))
    y[:, 1:] = s * (x + x[:, ::-1]) + 0.5 * (x - x[:, ::-1])
    Y = np.conj(scipy.fft.rfft(y, axis=1))[:, :L]
    R = Y.real.copy()
    R[:, 0] *= 0.5
    F, off = np.empty_like(R), np.zeros(x.shape[0])
    for g in range(G):
        c = np.cumsum(R[:, g * L // G:(g + 1) * L // G], axis=1)
        F[:, g * L // G:(g + 1) * L // G] = c + off[:, None]
        off = off + c[:, -1]
    out = np.empty((x.shape[0], N))
    out[:, 0::2], out[:, 1::2] = Y.imag, F
    return out[:, 1:]


def rms_error(y, ref):
    e = np.linalg.norm((y - ref).astype(float), axis=1) / np.linalg.norm(ref.astype(float), axis=1)
    return float(np.sqrt((e ** 2).mean()))


@pytest.mark.parametrize("N", SIZES)
@pytest.mark.parametrize("spikes", [1, 2, 4])
@pytest.mark.parametrize("sign", ["positive", "alternating", "random"])
def test_background_with_larger_values(harness, N, spikes, sign):  # noqa: F811
    rng = np.random.default_rng(N + spikes)
    n = N - 1
    for b in (0.02, 0.04, 0.06, 0.08, 0.1, 0.14, 0.18, 0.25, 0.4):
        x = b * rng.uniform(0.9, 1.1, (32, n))
        if sign == "alternating":
            x *= (-1.0) ** np.arange(n)
        elif sign == "random":
            x *= rng.choice([-1.0, 1.0], (32, n))
        for _ in range(spikes):
            x[np.arange(32), rng.integers(0, n, 32)] = rng.uniform(1.0, 1.05, 32)
        ref = reference(x)
        # float64's own error, and a quarter for the spread over 32 lines
        assert rms_error(run(harness, x), ref) <= 1.25 * rms_error(float64_transform(x), ref), b


@pytest.mark.parametrize("N", SIZES)
def test_first_level_sums_at_their_bound(harness, N):  # noqa: F811
    """Full-size lines with the signs of one output of the first level, and a
    bound on that level over all its outputs."""
    P, m = N // 16, 1.0 - 2.0 ** -53
    j = np.arange(N)
    big = np.maximum(np.sin(np.pi * j / N), 0.5)                 # |y_j| <= 2 m big_j
    big[0] = 0.0
    q = np.arange(P)
    worst, lines = 0.0, []
    for a in range(8):
        for k1 in range(P):
            e, o = 2 * (a + 8 * q), 2 * (a + 8 * q) + 1
            ang = 2.0 * np.pi * q * k1 / P
            for we, wo in ((np.cos(ang), -np.sin(ang)), (np.sin(ang), np.cos(ang))):
                worst = max(worst, 2.0 * (big[e] * np.abs(we) + big[o] * np.abs(wo)).sum())
                y = np.zeros(N)                                  # the signs of y wanted, 0 where free
                y[e], y[o] = np.sign(we), np.sign(wo)
                x = np.zeros(N)
                for i in range(1, N // 2):
                    s, t = y[i], y[N - i]
                    if np.sin(np.pi * i / N) >= 0.5 and s * t >= 0 and s + t:
                        x[i] = x[N - i] = np.sign(s + t) * m     # y_i = y_{N-i} = 2 m sin
                    else:
                        x[i] = m * np.sign(s if s else -t if t else 1.0)
                        x[N - i] = -x[i]                         # y_i = m, y_{N-i} = -m
                x[N // 2] = m * (y[N // 2] if y[N // 2] else 1.0)
                lines.append(x[1:])
    assert worst <= 1.83 * P
    late = {32: 55, 64: 54, 128: 53, 256: 52, 384: 51, 512: 51}[N]
    assert worst * 2.0 ** (late + 4) < 2.0 ** 61 - 2.0 ** 32
    pick = np.random.default_rng(N).permutation(len(lines))[:32]
    x = np.array([lines[i] for i in np.resize(pick, 32)])
    ref = reference(x)
    assert rms_error(run(harness, x, 32), ref) <= 1.25 * rms_error(float64_transform(x), ref)
