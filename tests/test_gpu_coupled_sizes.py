"""The float64 coupled system on its long lines (384 and 512 points, where the
middle pass's tiles come close to a block's shared memory, or exceed it and
take the fields in turn): box solve against dense float64 sine products,
operator against the oracle, and a whole solve."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from kfbi_workloads import configs as C, geometry as G  # noqa: E402
from oracle import coupled as CP  # noqa: E402
from paper_2104_05024_gb300 import kfbi as K  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
DI, DE, KAPPA = (3.0, 0.5, 0.5), (2.0, 1.0, 1.0), 40.0


def dense_solve(ri, re, N):
    """[A_i - kappa, kappa; kappa, A_e - kappa]^{-1} in sine modes by matrix
    products; the array axes are ([z,] y, x)."""
    k = torch.arange(1, N, dtype=torch.float64, device=DEV)
    S = torch.sin(((k[:, None] * k[None, :]) % (2 * N)) * (math.pi / N))
    mu = -(float(N) ** 2) * torch.sin(k * (math.pi / (2 * N))) ** 2      # h = 2 / N
    d = ri.dim()

    def transform(v):
        for a in range(d):
            v = torch.tensordot(S, v, dims=([1], [d - 1]))               # the last axis to the front, d times
        return v

    def modes(D):
        m = 0.0
        for a in range(d):                                               # axis a of the conductivity: x first
            m = m + D[a] * mu.reshape([-1 if i == d - 1 - a else 1 for i in range(d)])
        return m - KAPPA

    ai, ae = modes(DI), modes(DE)
    det = ai * ae - KAPPA ** 2
    fi, fe = transform(ri), transform(re)
    s = (2.0 / N) ** d
    return s * transform((ae * fi - KAPPA * fe) / det), s * transform((ai * fe - KAPPA * fi) / det)


@pytest.mark.parametrize("dim,N", [(2, 256), (2, 384), (2, 512), (3, 64), (3, 384), (3, 512)])
def test_coupled_box_solve_long_lines(dim, N):
    geom = G.ellipse_config0(N) if dim == 2 else G.sphere3(0.5, max(4, N // 16))
    grid = C.Grid(dim, N)
    h = K.KFBI(geom, grid, D_i=DI[:dim], D_e=DE[:dim])
    gen = torch.Generator(device=DEV).manual_seed(N)
    ri, re = (torch.randn(grid.shape, dtype=torch.float64, device=DEV, generator=gen) for _ in range(2))
    vi, ve = torch.empty_like(ri), torch.empty_like(ri)
    h.box_solve_coupled(ri, re, vi, ve, KAPPA)
    h.close()
    for v, w in zip((vi, ve), dense_solve(ri, re, N)):
        assert float((v - w).abs().max() / w.abs().max()) < 1e-12


@pytest.mark.parametrize("N", [384, 512])
def test_coupled_operator_and_solve_2d(N):
    geom, grid = G.ellipse_config0(2 * N), C.Grid(2, N)
    h = K.KFBI(geom, grid, D_i=DI[:2], D_e=DE[:2], tol=1e-10)
    X = geom.nodes
    psi = np.concatenate([1.0 + 0.5 * X[:, 0] - 0.3 * X[:, 1] ** 2, 0.4 - 0.2 * X[:, 1] + 0.1 * X[:, 0] ** 2])
    out = torch.empty(2 * geom.M, dtype=torch.float64, device=DEV)
    h.apply_A_coupled(torch.tensor(psi, device=DEV), out, KAPPA)
    ref = CP.CoupledKFBI(geom, grid, DI[:2], DE[:2]).apply_A(psi, KAPPA)
    assert np.abs(out.cpu().numpy() - ref).max() / np.abs(ref).max() < 1e-10
    # a whole solve reaches its tolerance, by the operator itself
    x = torch.zeros_like(out)
    st = h.solve_bie(out, x, KAPPA)
    back = torch.empty_like(out)
    h.apply_A_coupled(x, back, KAPPA)
    h.close()
    assert st["rel_res"] <= 1e-10
    assert float((back - out).norm() / out.norm()) < 1e-9


def test_coupled_operator_3d_384_unaffected_by_whole_solves():
    """The operator covers only the lines and planes near the interface: what
    whole-field solves left in the work grids elsewhere must not matter."""
    geom, grid = G.shell_config2(C.surface_res(384)), C.Grid(3, 384)
    h = K.KFBI(geom, grid, D_i=DI, D_e=DE)
    rng = np.random.default_rng(1)
    psi = torch.tensor(rng.standard_normal(2 * geom.M), device=DEV)
    a, b = torch.empty_like(psi), torch.empty_like(psi)
    h.apply_A_coupled(psi, a, KAPPA)
    r = torch.ones(grid.shape, dtype=torch.float64, device=DEV)
    vi, ve = torch.empty_like(r), torch.empty_like(r)
    h.box_solve_coupled(r, r, vi, ve, KAPPA)
    h.apply_A_coupled(psi, b, KAPPA)
    h.close()
    assert torch.isfinite(a).all() and torch.equal(a, b)
