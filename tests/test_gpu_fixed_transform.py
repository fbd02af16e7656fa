"""The float64 box solve (fixed-point transform lines) against dense float64
sine products, over every grid size, for smooth, sparse and widely scaled
fields; infinities and NaN reach the result as in float64."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def dense_solve(r, N, lam):
    """The same solve as matrix products in float64."""
    import torch
    k = torch.arange(1, N, dtype=torch.float64, device=r.device)
    S = torch.sin(((k[:, None] * k[None, :]) % (2 * N)) * (math.pi / N))
    mu = -(float(N) ** 2) * torch.sin(k * (math.pi / (2 * N))) ** 2      # h = 2 / N

    def transform(v):
        v = v @ S
        v = torch.einsum("yk,...yx->...kx", S, v)
        return torch.einsum("zk,zyx->kyx", S, v) if v.dim() == 3 else v

    d = r.dim()
    m = mu[:, None] + mu[None, :] if d == 2 else mu[:, None, None] + mu[None, :, None] + mu[None, None, :]
    return transform(transform(r) / (m - lam)) * (2.0 / N) ** d


def field(kind, shape, seed, dev):
    import torch
    rng = np.random.default_rng(seed)
    if kind == "smooth":
        x = np.linspace(-1.0, 1.0, shape[0] + 2)[1:-1]
        e = [np.exp(-(x - c) ** 2 / 0.08) for c in rng.uniform(-0.5, 0.5, len(shape))]
        v = e[0][:, None] * e[1][None, :] if len(shape) == 2 else np.einsum("a,b,c->abc", *e)
    elif kind == "sparse":
        v = (rng.random(shape) < 0.01) * rng.standard_normal(shape) * 1e6
    else:
        v = rng.standard_normal(shape) * 10.0 ** rng.uniform(-14, 0, shape)
    return torch.tensor(v, device=dev)


@pytest.mark.parametrize("kind", ["smooth", "sparse", "wide"])
@pytest.mark.parametrize("dim,N", [(2, 16), (2, 32), (2, 64), (2, 128), (2, 256), (2, 384), (2, 512), (3, 8), (3, 16),
                                   (3, 32), (3, 64), (3, 128)])
def test_box_solve_matches_dense_products(dim, N, kind):
    import torch
    from kfbi_workloads import configs as C, geometry as G
    from paper_2104_05024_gb300 import kfbi as K
    geom = G.ellipse_config0(max(32, N)) if dim == 2 else G.sphere3(0.5, max(4, N // 4))
    grid = C.Grid(dim, N)
    h = K.KFBI(geom, grid)
    dev = torch.device("cuda:0")
    r = field(kind, grid.shape, N + dim, dev)
    v = torch.empty_like(r)
    for lam in (0.5, 60.0):
        h.box_solve(r, v, lam, precision=K.FP64)
        ref = dense_solve(r, N, lam)
        err = float((v - ref).norm() / ref.norm())
        # 2 d transforms of the float64 algorithm, each below 3e-15 at N = 512
        # (its error grows like sqrt(N)), and the products' own roundings
        assert err < 2 * dim * 3e-15 * math.sqrt(N / 512.0) + 1e-15, (lam, err)
    h.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,lams", [(32, (0.0, 1e5)), (64, (0.0, 60.0)), (256, (0.0, 2.0, 60.0, 1e5)), (384, (5.0, 60.0))])
def test_z_elimination_and_transforms_match_dense_products(N, lams, precision):
    """Both sides of the rule that picks the z solve: elimination (lambda
    large against the mode spacing), transforms (Poisson and nearly so on
    fine grids)."""
    import torch
    from kfbi_workloads import configs as C, geometry as G
    from paper_2104_05024_gb300 import kfbi as K
    grid = C.Grid(3, N)
    h = K.KFBI(G.sphere3(0.5, max(4, N // 4)), grid)
    dev = torch.device("cuda:0")
    for kind in ("smooth", "sparse"):
        r = field(kind, grid.shape, N, dev)
        v = torch.empty_like(r)
        for lam in lams:
            h.box_solve(r, v, lam, precision=K.FP64 if precision == "fp64" else K.FP32)
            ref = dense_solve(r, N, lam)
            err = float((v - ref).norm() / ref.norm())
            # float64: six transforms' bound as above; float32: the same
            # roundings at 2^-24 instead of 2^-53
            bound = 6 * 3e-15 * math.sqrt(N / 512.0) + 1e-15
            assert err < (bound if precision == "fp64" else bound * 2.0 ** 29), (kind, lam, err)
    h.close()


def test_non_finite_sources_reach_the_solution():
    import torch
    from kfbi_workloads import configs as C, geometry as G
    from paper_2104_05024_gb300 import kfbi as K
    h = K.KFBI(G.sphere3(0.5, 8), C.Grid(3, 32))
    dev = torch.device("cuda:0")
    for bad in (float("inf"), float("nan")):
        r = torch.ones((31, 31, 31), dtype=torch.float64, device=dev)
        r[3, 4, 5] = bad
        v = torch.zeros_like(r)
        h.box_solve(r, v, 60.0, precision=K.FP64)
        assert not torch.isfinite(v).any()
    # zeros stay zeros, and the scale of the field does not matter
    r = torch.zeros((31, 31, 31), dtype=torch.float64, device=dev)
    h.box_solve(r, v, 60.0, precision=K.FP64)
    assert torch.equal(v, torch.zeros_like(v))
    r = torch.tensor(np.random.default_rng(0).standard_normal((31, 31, 31)), device=dev)
    a, b = torch.empty_like(r), torch.empty_like(r)
    h.box_solve(r, a, 60.0, precision=K.FP64)
    for e in (900, -800):
        h.box_solve(r * 2.0 ** e, b, 60.0, precision=K.FP64)
        assert torch.equal(a * 2.0 ** e, b)
    h.close()
