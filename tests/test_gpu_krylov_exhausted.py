"""GMRES past the dimension of the problem: with tolerance 0 the iteration goes
on when the Krylov space is exhausted, where the new vector is all rounding.
Its norm is still that of the vector, so the residual estimate keeps falling
by rounding factors and is never exactly 0 (which would stop the iteration as
converged), and the solution stays at the rounding of its residual."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from kfbi_workloads import configs as C, geometry as G  # noqa: E402
from paper_2104_05024_gb300 import kfbi as K  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def solve(geom, grid, lam, its, seed):
    h = K.KFBI(geom, grid, restart=64)
    g = torch.tensor(np.random.default_rng(seed).standard_normal(geom.M), device=DEV)
    psi = torch.zeros_like(g)
    st = h.solve_bie(g, psi, lam, tol=0.0, max_iter=its)
    out = torch.empty_like(psi)
    h.apply_A(psi, out, lam)
    h.close()
    return st, float((g - out).norm() / g.norm())


@pytest.mark.parametrize("M", [12, 16, 24, 32, 48, 60])
def test_exhausted_space(M):
    for seed in range(3):
        st, true = solve(G.ellipse_config0(M), C.Grid(2, 64), 60.0, M + 4, seed)
        assert st["iters"] == M + 4 and st["rel_res"] > 0.0
        # well conditioned (residual 5e-16 within a few iterations): rounding
        # of M-term sums
        assert true < 1e-13
