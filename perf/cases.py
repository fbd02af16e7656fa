"""Performance cases of the KFBI library: the calls its users make, over the
sizes, precisions and box conditions they make them with.

Kinds of calls (all through the Python binding of the C ABI):

* box      one fast box solve v = L_h^{-1} r on a whole field (sine or cosine
           transforms), in float64 or in the refined float32 form;
* apply    one application of the boundary integral operator A psi
           (corrections, box solve, interface limit), the unit of every
           Krylov iteration, in float64;
* coupled  the same for the anisotropic coupled system;
* neumann  a whole Neumann solve (right-hand side, GMRES, solution);
* strang   a short bidomain run from its initial state;
* mlp      loss and gradients of the warm-start network for one minibatch.

Fields are float64.  Inputs are smooth: sums of Gaussian bumps on the grid,
sums of plane waves at the interface nodes, a ball of excited tissue for the
bidomain state.
"""
import math

import numpy as np
import torch

from kfbi_workloads import configs as C
from kfbi_workloads import geometry as G
from paper_2104_05024_gb300 import kfbi as K

DEV = "cuda:0"
SIZES = (16, 32, 64, 128, 256, 384, 512)


def listed():
    return [
        # the smallest call: one operator application on the 2-D ellipse at
        # 128^2 (launch latency, a chain of short kernels)
        {"name": "apply_2d_ellipse128_fp64", "kind": "apply", "geom": "ellipse", "N": 128, "box": "dirichlet"},
        # the paper's 2-D setting from start to end: 20 Strang steps on the
        # ellipse at 128^2, tolerance 1e-10, float64, previous-density start
        {"name": "strang_2d_ellipse128_fp64", "kind": "strang", "geom": "ellipse", "N": 128, "box": "dirichlet",
         "precision": "fp64", "warm": "previous", "tol": 1e-10, "steps": 20},
        # coarse 3-D grids of a convergence study: the star body at 64^3
        {"name": "apply_star64_fp64", "kind": "apply", "geom": "star", "N": 64, "box": "dirichlet"},
        # the plain method's Krylov iteration on the production grid
        {"name": "apply_shell256_fp64", "kind": "apply", "geom": "shell", "N": 256, "box": "dirichlet"},
        # the plain method's volume solve on a whole field
        {"name": "box_shell256_fp64", "kind": "box", "geom": "shell", "N": 256, "box": "dirichlet",
         "precision": "fp64"},
        # the refined float32 volume solve of every production time step
        {"name": "box_shell256_mixed", "kind": "box", "geom": "shell", "N": 256, "box": "dirichlet",
         "precision": "mixed"},
        # the same on a grid that does not fit in L2 (large single solves)
        {"name": "box_shell512_mixed", "kind": "box", "geom": "shell", "N": 512, "box": "dirichlet",
         "precision": "mixed"},
        # the Neumann box: (N+1)^3 unknowns, odd and unaligned rows
        {"name": "box_neumann256_mixed", "kind": "box", "geom": "shell", "N": 256, "box": "neumann",
         "precision": "mixed"},
        # the anisotropic system's Krylov iteration on the paper's sphere
        {"name": "coupled_sphere128_fp64", "kind": "coupled", "geom": "sphere", "N": 128, "box": "dirichlet"},
        # a whole Neumann solve in the refined float32 form, tolerance 1e-10
        {"name": "neumann_star128_mixed", "kind": "neumann", "geom": "star", "N": 128, "box": "dirichlet",
         "precision": "mixed", "tol": 1e-10},
        # the production run's opening on the prolate shell at 256^3:
        # float32 transforms with refinement, history projection
        {"name": "strang_shell256_mixed", "kind": "strang", "geom": "shell", "N": 256, "box": "dirichlet",
         "precision": "mixed", "warm": "projection", "tol": 1e-9, "steps": 10},
        # one minibatch of the warm-start network's training
        {"name": "mlp_grad_4096", "kind": "mlp", "B": 4096},
    ]


def draw(rng):
    kind = rng.choice(("box", "box", "apply", "apply", "coupled", "neumann", "strang", "mlp"))
    if kind == "mlp":
        return {"kind": kind, "B": int(round(math.exp(rng.uniform(math.log(64), math.log(16384)))))}
    geom = rng.choice(("ellipse", "star", "shell", "sphere"))
    box = "neumann" if kind != "coupled" and rng.random() < 0.25 else "dirichlet"
    precision = rng.choice(("fp64", "mixed"))
    # the largest grids are left to the calls that a listed case makes there
    top = {"box": 512 if precision == "mixed" else 384, "apply": 384, "coupled": 256, "neumann": 128, "strang": 64}[kind]
    sizes = [n for n in SIZES if n <= (512 if geom == "ellipse" else top) and n >= (64 if geom == "ellipse" else 32)]
    c = {"kind": kind, "geom": geom, "N": rng.choice(sizes), "box": box}
    if kind in ("box", "neumann", "strang"):
        c["precision"] = precision
    if kind in ("neumann", "strang"):
        c["tol"] = rng.choice((1e-10, 1e-11))
    if kind == "strang":
        c["warm"] = rng.choice(("previous", "projection"))
        c["steps"] = rng.randint(1, 6)
    if kind in ("box", "apply") and rng.random() < 0.5:
        c["lam"] = round(math.exp(rng.uniform(math.log(5.0), math.log(5000.0))), 3)
    return c


# ------------------------------------------------------------------ inputs

_GEOMETRY = {}


def _geometry(case):
    key = (case["geom"], case["N"])
    if key not in _GEOMETRY:
        n = C.surface_res(case["N"])
        _GEOMETRY[key] = {"ellipse": lambda: G.ellipse_config0(2 * case["N"]), "star": lambda: G.star_config1(n),
                          "shell": lambda: G.shell_config2(n), "sphere": lambda: G.sphere3(0.9, n)}[case["geom"]]()
    return _GEOMETRY[key]


def _dim(case):
    return 2 if case["geom"] == "ellipse" else 3


def _points(case):
    n = case["N"] + 1 if case["box"] == "neumann" else case["N"] - 1
    return n, n ** _dim(case)


def _lam(case):
    return float(case.get("lam", 60.0))


def _axis(case):
    N = case["N"]
    k = torch.arange(0, N + 1, dtype=torch.float64, device=DEV)
    x = -1.0 + 2.0 / N * k
    return x if case["box"] == "neumann" else x[1:-1]


def _bumps(case, seed, count=24):
    """Sum of Gaussian bumps on the whole field, [z][y][x]."""
    rng = np.random.default_rng(seed)
    d = _dim(case)
    amp, width = rng.uniform(-1.0, 1.0, count), rng.uniform(0.05, 0.2, count)
    cen = rng.uniform(-0.6, 0.6, (count, d))
    x = _axis(case)
    t = lambda a: torch.tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
    e = [torch.exp(-((x[None, :] - t(cen[:, a])[:, None]) ** 2) / (2.0 * t(width)[:, None] ** 2)) for a in range(d)]
    n = x.numel()
    if d == 2:
        return ((t(amp)[:, None] * e[1]).T @ e[0]).contiguous()
    out = torch.empty((n, n, n), dtype=torch.float64, device=DEV)
    for z in range(n):
        out[z] = ((t(amp) * e[2][:, z])[:, None] * e[1]).T @ e[0]
    return out


def _waves(case, seed, count=8):
    """Smooth values at the interface nodes: a sum of plane waves."""
    rng = np.random.default_rng(seed + 7919)
    nodes = _geometry(case).nodes
    v = np.zeros(len(nodes))
    for _ in range(count):
        k, p = rng.uniform(-6.0, 6.0, nodes.shape[1]), rng.uniform(0.0, 2.0 * np.pi)
        v += rng.uniform(-1.0, 1.0) * np.cos(nodes @ k + p)
    return torch.tensor(v, device=DEV)


def _ball(case, seed):
    """Excited tissue: V = 1 in a ball of radius 0.1 around a point of the domain."""
    rng = np.random.default_rng(seed)
    x = _axis(case)
    if _dim(case) == 2:
        c = (-0.4 + rng.uniform(-0.1, 0.1), rng.uniform(-0.1, 0.1))
        r2 = (x[None, :] - c[0]) ** 2 + (x[:, None] - c[1]) ** 2
    else:
        ct, ph = rng.uniform(-1.0, 1.0), rng.uniform(0.0, 2.0 * math.pi)
        st = math.sqrt(1.0 - ct * ct)
        s = {"shell": (0.8, 0.5, 0.5), "star": (0.35, 0.35, 0.35), "sphere": (0.6, 0.6, 0.6)}[case["geom"]]
        c = (s[0] * st * math.cos(ph), s[1] * st * math.sin(ph), s[2] * ct)
        r2 = (x[None, None, :] - c[0]) ** 2 + (x[None, :, None] - c[1]) ** 2 + (x[:, None, None] - c[2]) ** 2
    return (r2 < 0.01).to(torch.float64).contiguous()


MLP_DIMS = (9, 128, 128, 128, 128, 1)


def _mlp_inputs(case, seed):
    rng = np.random.default_rng(seed)
    parts = []
    for fan_in, fan_out in zip(MLP_DIMS[:-1], MLP_DIMS[1:]):
        lim = math.sqrt(6.0 / fan_in) if fan_out > 1 else math.sqrt(1.0 / fan_in)
        parts += [rng.uniform(-lim, lim, fan_out * fan_in), rng.uniform(-0.1, 0.1, fan_out)]
    params = np.concatenate(parts).astype(np.float32)
    norm = np.concatenate([rng.uniform(-0.2, 0.2, 9), rng.uniform(0.5, 1.5, 9), [0.05, 0.8]]).astype(np.float32)
    F = rng.standard_normal((case["B"], 9)).astype(np.float32)
    T = (np.tanh(F[:, 0] - F[:, 1]) + 0.1 * rng.standard_normal(case["B"])).astype(np.float32)
    return params, norm, F, T


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        params, norm, F, T = _mlp_inputs(case, seed)
        return {"case": case, "mlp": K.MLP(params, norm, case["B"]), "F": torch.tensor(F, device=DEV),
                "T": torch.tensor(T, device=DEV)}
    geom, grid = _geometry(case), C.Grid(_dim(case), case["N"], bc=case["box"])
    prec = K.MIXED if case.get("precision") == "mixed" else K.FP64
    warm = K.WARM_PROJECTION if case.get("warm") == "projection" else K.WARM_PREVIOUS
    kw = {"precision": prec, "warm": warm, "tol": case.get("tol", 1e-10), "dt": 0.05}
    if kind == "coupled":
        d = _dim(case)
        kw.update(D_i=(30.0, 5.0, 5.0)[:d], D_e=(20.0, 10.0, 10.0)[:d])
    h = K.KFBI(geom, grid, **kw)
    s = {"case": case, "h": h, "prec": prec, "lam": _lam(case)}
    M = geom.M
    if kind == "box":
        s["r"] = _bumps(case, seed)
        s["v"] = torch.empty_like(s["r"])
    elif kind in ("apply", "coupled"):
        s["psi"] = _waves(case, seed)
        if kind == "coupled":
            s["psi"] = torch.cat([s["psi"], _waves(case, seed + 1)])
        s["out"] = torch.empty_like(s["psi"])
    elif kind == "neumann":
        s["f"], s["gN"] = _bumps(case, seed), _waves(case, seed)
        s["u"] = torch.empty_like(s["f"])
        s["psi"] = torch.empty(M, dtype=torch.float64, device=DEV)
    else:
        s["V0"] = _ball(case, seed)
        s["V"], s["w"], s["ue"] = (torch.empty_like(s["V0"]) for _ in range(3))
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "mlp":
        loss, grad = s["mlp"].grad(s["F"], s["T"])
        return [float(loss), grad]
    h = s["h"]
    if kind == "box":
        h.box_solve(s["r"], s["v"], s["lam"], precision=s["prec"])
        return s["v"]
    if kind == "apply":
        h.apply_A(s["psi"], s["out"], s["lam"], precision=K.FP64)
        return s["out"]
    if kind == "coupled":
        h.apply_A_coupled(s["psi"], s["out"], 40.0)
        return s["out"]
    if kind == "neumann":
        s["psi"].zero_()
        h.solve_neumann(s["f"], s["gN"], s["u"], s["psi"], s["lam"])
        return [s["u"], s["psi"]]
    # a run from its initial state: no densities of an earlier run
    s["V"].copy_(s["V0"])
    s["w"].zero_()
    h.set_densities(None, None, None, 0)
    h.bidomain_step(C.FHN_CONFIG, s["V"], s["w"], s["ue"], nsteps=case["steps"])
    return [s["V"], s["w"], s["ue"]]


# -------------------------------------------------------------------- work

def work(case):
    """Each input and output once; the transforms' 2.5 N log2 N operations a
    line, for one box solve per operator application and for two per whole
    solve or time step (the volume and the boundary part)."""
    kind = case["kind"]
    if kind == "mlp":
        p = sum(a * b + b for a, b in zip(MLP_DIMS[:-1], MLP_DIMS[1:]))
        mac = sum(a * b for a, b in zip(MLP_DIMS[:-1], MLP_DIMS[1:]))
        return {"bytes": 4.0 * (case["B"] * 10 + 2 * p), "flops": 6.0 * mac * case["B"]}
    d, (n, pts) = _dim(case), _points(case)
    solve = 2 * d * pts * 2.5 * math.log2(case["N"])
    M = _geometry(case).M
    if kind == "box":
        return {"bytes": 16.0 * pts, "flops": solve}
    if kind == "apply":
        return {"bytes": 16.0 * M, "flops": solve}
    if kind == "coupled":
        return {"bytes": 32.0 * M, "flops": 2 * solve}
    if kind == "neumann":
        return {"bytes": 16.0 * pts + 24.0 * M, "flops": 2 * solve}
    return {"bytes": 40.0 * pts, "flops": case["steps"] * 2 * solve}


# ------------------------------------------------------------------- exact

def _sine(N):
    k = torch.arange(1, N, dtype=torch.float64, device=DEV)
    kp = (k[:, None] * k[None, :]) % (2 * N)
    return torch.sin(kp * (math.pi / N))


def _cosine(N):
    """Forward cosine matrix over the nodes 0..N: cos(pi k p / N) c_k, c_0 = c_N = 1/2."""
    k = torch.arange(0, N + 1, dtype=torch.float64, device=DEV)
    m = torch.cos(((k[:, None] * k[None, :]) % (2 * N)) * (math.pi / N))
    m[:, 0] *= 0.5
    m[:, N] *= 0.5
    return m


def _exact_box(case, r):
    N, d = case["N"], _dim(case)
    neumann = case["box"] == "neumann"
    S = _cosine(N) if neumann else _sine(N)
    p = torch.arange(0, N + 1, dtype=torch.float64, device=DEV) if neumann else \
        torch.arange(1, N, dtype=torch.float64, device=DEV)
    h = 2.0 / N
    mu = -(4.0 / (h * h)) * torch.sin(p * (math.pi / (2 * N))) ** 2
    n = S.shape[0]

    def transform(v):
        v = v @ S.T                                    # along x
        if d == 2:
            return S @ v
        for z in range(n):                             # along y, plane by plane
            v[z] = S @ v[z]
        return (S @ v.reshape(n, n * n)).reshape(n, n, n)

    v = transform(r)
    if d == 2:
        v = v / (mu[:, None] + mu[None, :] - _lam(case))
    else:
        for z in range(n):
            v[z] /= mu[z] + mu[:, None] + mu[None, :] - _lam(case)
    return transform(v) * (2.0 / N) ** d


def _exact_mlp(case, seed):
    params, norm, F, T = _mlp_inputs(case, seed)
    t = lambda a: torch.tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
    p, nv = t(params), t(norm)
    a = (t(F) - nv[:9]) / nv[9:18]
    y = (t(T) - nv[18]) / nv[19]
    at, Ws, bs = 0, [], []
    for fan_in, fan_out in zip(MLP_DIMS[:-1], MLP_DIMS[1:]):
        Ws.append(p[at:at + fan_in * fan_out].reshape(fan_out, fan_in).clone().requires_grad_())
        at += fan_in * fan_out
        bs.append(p[at:at + fan_out].clone().requires_grad_())
        at += fan_out
    for k, (W, b) in enumerate(zip(Ws, bs)):
        a = a @ W.T + b
        if k < len(Ws) - 1:
            a = a * torch.sigmoid(a)
    loss = 0.5 * ((a[:, 0] - y) ** 2).mean()
    loss.backward()
    grad = torch.cat([g.grad.reshape(-1) for pair in zip(Ws, bs) for g in pair])
    return [float(loss), grad.cpu().numpy()]


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "box":
        return _exact_box(case, _bumps(case, seed))
    # the integral operator needs the whole discretisation of the interface
    return None
