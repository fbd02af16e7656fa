"""The z solve by elimination at the edge of its rule (the slowest mode
remembers just under 48 rows) and where the time steps use it, against a
tridiagonal solve in extended precision: sources of a single x and y mode, so
that the other four passes add only their roundings."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from kfbi_workloads import configs as C, geometry as G  # noqa: E402
from paper_2104_05024_gb300 import kfbi as K  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def tridiagonal(f, eps, h2):
    """(2 + eps) v_k - v_{k-1} - v_{k+1} = -h2 f_k along the last axis."""
    n = f.shape[-1]
    d, y = np.empty(n, LD), np.empty(f.shape, LD)
    R = -h2 * f.astype(LD)
    d[0], y[..., 0] = 2 + eps, R[..., 0]
    for k in range(1, n):
        d[k] = 2 + eps - 1 / d[k - 1]
        y[..., k] = R[..., k] + y[..., k - 1] / d[k - 1]
    v = np.empty(f.shape, LD)
    v[..., -1] = y[..., -1] / d[-1]
    for k in range(n - 2, -1, -1):
        v[..., k] = (y[..., k] + v[..., k + 1]) / d[k]
    return v


# lambda just inside the rule, and the time steps' 60 (64: always inside)
@pytest.mark.parametrize("N,lam", [(64, 0.0), (128, 0.0), (256, 2.2), (256, 5.0), (256, 60.0), (384, 11.1), (384, 60.0),
                                   (512, 23.6)])
def test_single_modes_against_extended_precision(N, lam):
    h = K.KFBI(G.sphere3(0.5, 8), C.Grid(3, N))
    rng = np.random.default_rng(N)
    t = np.arange(1, N) / N
    f = np.array([rng.standard_normal(N - 1), np.exp(-(t - 0.4) ** 2 / 0.02),
                  (rng.random(N - 1) < 0.05) * rng.standard_normal(N - 1) * 1e5, np.sin(np.pi * t)])
    h2 = (LD(2) / N) ** 2
    j = np.arange(1, N).astype(LD)
    # each mode's amplitude is read back on one column, at its crest
    for p, crest in ((1, N // 2), (2, N // 4)):
        s = np.sin(PI * p * j / N).astype(np.float64)
        mode = torch.tensor(s, device=DEV)
        mode = mode[:, None] * mode[None, :]
        s2 = np.sin(PI * p / (2 * LD(N))) ** 2
        eps = h2 * LD(lam) + 8 * s2
        if p == 1 and (N, lam) in ((256, 2.2), (384, 11.1), (512, 23.6)):
            assert 47.5 < float(1 / np.sqrt(eps)) < 48.0
        ref = tridiagonal(f, eps, h2)
        for prec, unit in ((K.FP64, 2.0 ** -53), (K.FP32, 2.0 ** -24)):
            # two roundings a row that add up over the rows remembered (48 at
            # most), and four transforms of log2 N levels each
            bound = unit * (2.0 * np.sqrt(48.0) + 4.0 * np.log2(N))
            for i in range(len(f)):
                r = (torch.tensor(f[i], device=DEV)[:, None, None] * mode[None]).contiguous()
                v = torch.empty_like(r)
                h.box_solve(r, v, lam, precision=prec)
                got = v[:, crest - 1, crest - 1].cpu().numpy()
                err = float(np.linalg.norm((got - ref[i]).astype(float)) / np.linalg.norm(ref[i].astype(float)))
                assert err < bound, (p, prec, i, err, bound)
    h.close()
