"""The refined float32 box solve against the float64 one over grid sizes, both
box conditions and one or two rounds: the residual kernel takes 1, 2, 4 or 8
rows per thread by the grid's size (with a last chunk shorter than the others),
the Neumann box's x passes take their values singly or batched."""
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from kfbi_workloads import configs as C, geometry as G  # noqa: E402
from paper_2104_05024_gb300 import kfbi as K  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
SIZES = [(2, 16), (2, 32), (2, 64), (2, 128), (2, 256), (2, 512), (3, 8), (3, 16), (3, 32), (3, 64), (3, 128)]


@pytest.mark.parametrize("bc", ["dirichlet", "neumann"])
@pytest.mark.parametrize("dim,N", SIZES)
def test_refined_solve_matches_float64(dim, N, bc):
    geom = G.ellipse_config0(max(24, N)) if dim == 2 else G.sphere3(0.45, 4)
    grid = C.Grid(dim, N, bc=bc)
    gen = torch.Generator(device=DEV).manual_seed(N)
    r = torch.randn(grid.shape, dtype=torch.float64, device=DEV, generator=gen)
    ref, v = torch.empty_like(r), torch.empty_like(r)
    # two rounds: float64-accurate, the box solves' parity bound; one round
    # (time steps): about 1e-10 at 512 lines, 1e-12 at 256, growing with the
    # condition number, so with lambda = 60 alone
    for tol, bound, lams in ((1e-10, 1e-12, (0.5, 60.0)), (1e-8, 1e-9, (60.0,))):
        h = K.KFBI(geom, grid, tol=tol)
        for lam in lams:
            h.box_solve(r, ref, lam, precision=K.FP64)
            h.box_solve(r, v, lam, precision=K.MIXED)
            assert float((v - ref).norm() / ref.norm()) < bound, (tol, lam)
        h.close()
