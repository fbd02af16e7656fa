"""The operator application transforms only the lines and planes near the
interface (its right-hand side is zero and its result unread elsewhere): the
result equals, bit for bit, the same three steps taken through whole fields
(corrections, box solve of the whole field, interface limit)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def geometry(name, N):
    from kfbi_workloads import configs as C, geometry as G
    n = C.surface_res(N)
    if name == "bean":                      # not symmetric about the box centre
        return G.bean_mesh(max(4, N // 16))
    return {"shell": G.shell_config2, "star": G.star_config1, "sphere": lambda m: G.sphere3(0.9, m),
            "small": lambda m: G.ellipsoid3(0.3, 0.12, 0.2, max(4, m // 2))}[name](n)


def density(geom, scale=1.0):
    k = np.array([3.0, -2.0, 1.5])[:geom.dim]
    return scale * np.cos(geom.nodes @ k + 0.3) + 0.1 * np.sin(5.0 * geom.nodes[:, 0])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name,N", [("shell", 32), ("shell", 128), ("star", 64), ("bean", 128), ("small", 128),
                                    ("sphere", 128), ("shell", 256), ("shell", 384)])
def test_apply_equals_whole_field_steps(name, N, precision):
    import torch
    from kfbi_workloads import configs as C
    from paper_2104_05024_gb300 import kfbi as K
    if precision == "fp32" and N <= 64:
        pytest.skip("float32 grids of N <= 64 run the fused x-y passes on the whole grid")
    geom, grid = geometry(name, N), C.Grid(3, N)
    h = K.KFBI(geom, grid)
    dev = torch.device("cuda:0")
    lam = 60.0
    psi = torch.tensor(density(geom), device=dev)
    out, ref = torch.empty_like(psi), torch.empty_like(psi)
    rhs = torch.empty(grid.shape, dtype=torch.float64, device=dev)
    v = torch.empty_like(rhs)
    # a whole-field solve first: what the work grid holds elsewhere must not matter
    h.box_solve(torch.ones_like(rhs), v, lam, precision=K.FP64)
    h.box_solve(torch.ones_like(rhs), v, lam, precision=K.FP32)
    h.apply_A(psi, out, lam, precision=K.FP64 if precision == "fp64" else K.MIXED)
    h.correction(psi, rhs)
    h.box_solve(rhs, v, lam, precision=K.FP64 if precision == "fp64" else K.FP32)
    h.interface_limit(v, psi, ref)
    torch.cuda.synchronize()
    assert torch.isfinite(out).all()
    assert torch.equal(out, ref)
    # and the whole-field solve after it is not disturbed
    w = torch.empty_like(v)
    h.box_solve(rhs, w, lam, precision=K.FP64 if precision == "fp64" else K.FP32)
    assert torch.equal(v, w)
    h.close()
