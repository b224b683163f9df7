"""Workloads of the cell solver, one dict each, as a user's program runs them.

A case is a dict of plain values.  ``listed()`` gives the named ones, ``draw``
more of the same ranges; ``prepare`` makes what a program has in hand before
the call (inputs from the seed, the solver handle), ``run`` makes one pass
through the public entry points and returns its outputs, ``work`` counts the
bytes and operations that the pass cannot do without, ``exact`` evaluates the
same outputs in 64 bits with plain torch where that is feasible.

Kinds:

* ``step``   one step of a design loop on a kept handle: map the new design in,
  solve the cell problems, homogenise, d_h and its gradient, element or nodal
  sensitivities;
* ``batch``  the same solves for several uneven designs in one batched call;
* ``apply``  the coupled operator on a block of vectors;
* ``blocks`` the two preconditioner blocks on a block of vectors;
* ``evolve`` the level-set update: regularised velocity, one upwind step.
"""
import math

import numpy as np
import torch

from paper_2410_03148_gb300 import Cell, figure, hj_step, solve_batch

RHO_VOID = 1e-3


def _material():
    """z-poled PZT-5H-class constants (SI, Voigt order 11, 22, 33, 23, 13, 12)."""
    C = np.zeros((6, 6))
    C[0, 0] = C[1, 1] = 127.205e9
    C[0, 1] = C[1, 0] = 80.212e9
    C[0, 2] = C[2, 0] = C[1, 2] = C[2, 1] = 84.670e9
    C[2, 2] = 117.436e9
    C[3, 3] = C[4, 4] = 22.988e9
    C[5, 5] = 23.474e9
    e = np.zeros((3, 6))
    e[2, 0] = e[2, 1] = -6.62
    e[2, 2] = 23.24
    e[0, 4] = e[1, 3] = 17.03
    return C, e, np.diag([1.503e-8, 1.503e-8, 1.300e-8])


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest cell anyone solves (smoke test, unit tests): launch latency
        {"name": "step_8", "kind": "step", "nx": 8, "ny": 8, "nz": 8, "input": "phi", "dtype": "f64",
         "precision": 1, "loads": 511, "tol": 1e-10},
        # a small ragged cell: one coarsening, then a dense coarsest level
        {"name": "step_14x10x12", "kind": "step", "nx": 14, "ny": 10, "nz": 12, "input": "phi", "dtype": "f32",
         "precision": 1, "loads": 511, "tol": 1e-10},
        # odd sizes (an imported voxel geometry), density input
        {"name": "step_33x31x35_rho", "kind": "step", "nx": 33, "ny": 31, "nz": 35, "input": "rho",
         "dtype": "f32", "precision": 1, "loads": 511, "tol": 1e-10},
        # the ordinary design step
        {"name": "step_64", "kind": "step", "nx": 64, "ny": 64, "nz": 64, "input": "phi", "dtype": "f32",
         "precision": 1, "loads": 511, "tol": 1e-10},
        # the largest design step (the benchmark's cell)
        {"name": "step_128", "kind": "step", "nx": 128, "ny": 128, "nz": 128, "input": "phi", "dtype": "f64",
         "precision": 1, "loads": 511, "tol": 1e-10},
        # the full-FP64 solver, as used to check a mixed-precision result
        {"name": "step_32_fp64", "kind": "step", "nx": 32, "ny": 32, "nz": 32, "input": "phi", "dtype": "f64",
         "precision": 0, "loads": 511, "tol": 1e-10},
        # one load at a loose tolerance on the weak-scaling study's geometry
        {"name": "e1_96", "kind": "step", "nx": 96, "ny": 96, "nz": 96, "input": "e1", "dtype": "f64",
         "precision": 1, "loads": 1, "tol": 1e-8},
        # a set of uneven designs solved together
        {"name": "batch_uneven", "kind": "batch", "sizes": "32,32,48,48,64,64", "tol": 1e-10},
        # the coupled operator by itself: a user's own Krylov method, large and FP32
        {"name": "apply_f32_128", "kind": "apply", "nx": 128, "ny": 128, "nz": 128, "nrhs": 9, "dtype": "f32"},
        # the same in FP64, ragged and odd sizes, a few vectors
        {"name": "apply_f64_50x37x41", "kind": "apply", "nx": 50, "ny": 37, "nz": 41, "nrhs": 5, "dtype": "f64"},
        # the preconditioner's blocks by themselves
        {"name": "blocks_64x48x80", "kind": "blocks", "nx": 64, "ny": 48, "nz": 80, "nrhs": 9, "dtype": "f32"},
        # the level-set update between two solves, two constraints
        {"name": "evolve_64", "kind": "evolve", "nx": 64, "ny": 64, "nz": 64, "ncons": 2, "dtype": "f64"},
    ]


def _coarsest(n, nc):
    """Unknowns of the coarsest multigrid level of a block with nc components:
    halved while every size is even (and at least 4) and the level has more
    than 200 unknowns."""
    n = list(n)
    while all(v % 2 == 0 and v >= 4 for v in n) and nc * n[0] * n[1] * n[2] > 200:
        n = [v // 2 for v in n]
    return nc * n[0] * n[1] * n[2]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _quick(n):
    """Grids whose coarsest level is a dense system of 650 to 3000 unknowns are
    left out: mapping a design into them takes many seconds."""
    return all(not 650 < _coarsest(n, nc) <= 3000 for nc in (1, 3))


def _grid(rng, lo, hi, spread):
    """Any size per direction about a common one, odd ones among them."""
    while True:
        base = _log(rng, lo, hi)
        n = [min(hi, max(5, int(round(base * math.exp(rng.uniform(-spread, spread)))))) for _ in range(3)]
        if _quick(n):
            return n


def _step_size(rng, hi):
    """Grid of a design step: even sizes that coarsen, or odd ones up to 35."""
    while True:
        base = _log(rng, 8, hi)
        if base <= 35 and rng.random() < 0.25:
            n = [max(5, base + rng.randint(-3, 3)) for _ in range(3)]
        else:
            m = 2 if base < 24 else (8 if base < 64 else 16)
            n = [min(hi, max(m, m * int(round(base * rng.uniform(0.8, 1.25) / m)))) for _ in range(3)]
            n = [max(8, v) for v in n]
        if _quick(n) and (_coarsest(n, 3) <= 650 or n[0] * n[1] * n[2] <= 40000):
            return n


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "fp64", "e1", "batch", "apply", "apply", "blocks", "evolve"])
    if kind == "step":
        nx, ny, nz = _step_size(rng, 128)
        return {"kind": "step", "nx": nx, "ny": ny, "nz": nz, "input": rng.choice(["phi", "phi", "rho"]),
                "dtype": rng.choice(["f32", "f64"]), "precision": 1, "loads": 511, "tol": 1e-10}
    if kind == "fp64":
        n = [rng.choice([8, 12, 16, 20, 24, 32]) for _ in range(3)]
        while _coarsest(n, 3) > 650:
            n = [rng.choice([8, 12, 16, 20, 24, 32]) for _ in range(3)]
        return {"kind": "step", "nx": n[0], "ny": n[1], "nz": n[2], "input": "phi", "dtype": "f64",
                "precision": 0, "loads": 511, "tol": 1e-10}
    if kind == "e1":
        n = 16 * rng.randint(1, 8)
        return {"kind": "step", "nx": n, "ny": n, "nz": n, "input": "e1", "dtype": "f64", "precision": 1,
                "loads": 1, "tol": 1e-8}
    if kind == "batch":
        k = rng.randint(2, 8)
        return {"kind": "batch", "sizes": ",".join(str(rng.choice([16, 24, 32, 48, 64])) for _ in range(k)),
                "tol": 1e-10}
    if kind == "evolve":
        n = _grid(rng, 12, 96, 0.35)
        return {"kind": "evolve", "nx": n[0], "ny": n[1], "nz": n[2], "ncons": rng.randint(0, 3), "dtype": "f64"}
    f64 = kind == "apply" and rng.random() < 0.4
    n = _grid(rng, 8, 80 if f64 else 128, 0.35)
    return {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "nrhs": rng.randint(1, 9),
            "dtype": "f64" if f64 else "f32"}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

_DT = {"f32": torch.float32, "f64": torch.float64}


def _coords(shape):
    nz, ny, nx = shape
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") / n for n in (nz, ny, nx)]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    return x, y, z


def _unit_gradient(phi):
    """phi divided by its mean gradient length on the elements that it cuts."""
    nz, ny, nx = phi.shape
    c = [torch.roll(phi, (-dz, -dy, -dx), (0, 1, 2)) for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)]
    gx = sum(c[i + 1] - c[i] for i in (0, 2, 4, 6)) * (nx / 4.0)
    gy = sum(c[i + 2] - c[i] for i in (0, 1, 4, 5)) * (ny / 4.0)
    gz = sum(c[i + 4] - c[i] for i in (0, 1, 2, 3)) * (nz / 4.0)
    s = torch.stack(c)
    cut = ((s.amin(0) < 0) & (s.amax(0) > 0)).double()
    n = float(cut.sum())
    return phi if n == 0 else phi / (float(((gx * gx + gy * gy + gz * gz).sqrt() * cut).sum()) / n)


def _levelset(shape, rng):
    """Level set of a seeded design: median minus a sum of 8 periodic Gaussians."""
    c, a, s = rng.uniform(0, 1, (8, 3)), rng.uniform(0.5, 1, 8), rng.uniform(0.08, 0.2, 8)
    xyz = _coords(shape)
    tot = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for k in range(8):
        d2 = 0.0
        for v, ck in zip(xyz, c[k]):
            d = v - float(ck)
            d = d - torch.round(d)
            d2 = d2 + d * d
        tot = tot + float(a[k]) * torch.exp(-d2 / (2.0 * float(s[k]) ** 2))
    return _unit_gradient(tot.reshape(-1).median() - tot)


def _e1(shape, rng):
    """-prod cos(2 pi x_i) - t, with t about the study's 0.2."""
    x, y, z = _coords(shape)
    p = 2.0 * math.pi
    return _unit_gradient(-torch.cos(p * x) * torch.cos(p * y) * torch.cos(p * z) - float(rng.uniform(0.15, 0.25)))


def _design(case, rng, shape=None):
    shape = shape or (case["nz"], case["ny"], case["nx"])
    if case.get("input") == "e1":
        d = _e1(shape, rng)
    else:
        d = _levelset(shape, rng)
        if case.get("input") == "rho":   # densities in (1e-3, 1) across a smooth boundary
            d = RHO_VOID + (1.0 - RHO_VOID) * torch.sigmoid(-d * min(shape) * 1.5)
    return d.to(_DT[case.get("dtype", "f64")])


def _options(case):
    o = {"precision": case["precision"], "load_mask": case["loads"], "tol": case["tol"]}
    if case["precision"] == 0:
        o["max_iter"] = 4000
    return o


def _vectors(case, rng, ncomp):
    g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    return torch.randn((case["nrhs"], ncomp, case["nz"], case["ny"], case["nx"]), generator=g, device="cuda",
                       dtype=torch.float64).to(_DT[case["dtype"]])


def _densities(case, rng):
    """Log-uniform element scales in [1e-3, 1]."""
    g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    u = torch.rand((case["nz"], case["ny"], case["nx"]), generator=g, device="cuda", dtype=torch.float64)
    return torch.exp(math.log(RHO_VOID) * u)


def _inputs(case, seed):
    """Everything random of a case, in a fixed order."""
    rng = np.random.default_rng(seed)
    k = case["kind"]
    if k == "step":
        return {"first": _design(case, rng), "new": _design(case, rng)}
    if k == "batch":
        sizes = [int(v) for v in case["sizes"].split(",")]
        return {"first": [_design(case, rng, (n, n, n)) for n in sizes],
                "new": [_design(case, rng, (n, n, n)) for n in sizes]}
    if k == "evolve":
        shape = (case["nz"], case["ny"], case["nx"])
        phi = _levelset(shape, rng)
        # sensitivities live on the interface: smooth weights times a regularised delta
        near = torch.exp(-(phi * min(shape) / 2.0) ** 2) / phi.numel()
        w = [_levelset(shape, rng) for _ in range(1 + case["ncons"])]
        return {"phi": phi, "d": [near * v for v in w], "c": [float(v) for v in rng.uniform(-0.2, 0.2, case["ncons"])]}
    rho = _densities(case, rng)
    if k == "apply":
        return {"rho": rho, "x": _vectors(case, rng, 4)}
    return {"rho": rho, "u": _vectors(case, rng, 3), "p": _vectors(case, rng, 1)}


def prepare(case, seed):
    inp = _inputs(case, seed)
    mat, k = _material(), case["kind"]
    st = {"case": case, **inp}
    if k == "step":
        # the handle of a design loop: set up on an earlier design
        st["cell"] = Cell(st.pop("first"), mat, kind="rho" if case["input"] == "rho" else "phi", **_options(case))
    elif k == "batch":
        torch.cuda.synchronize()   # the designs are ready before other streams read them
        st["cells"], st["streams"] = [], []
        for d in st.pop("first"):
            st["streams"].append(torch.cuda.Stream())
            with torch.cuda.stream(st["streams"][-1]):
                st["cells"].append(Cell(d, mat, kind="phi", tol=case["tol"], graphs=3))
    elif k == "evolve":
        st["cell"] = Cell(inp["phi"], mat, kind="phi")
    else:
        st["cell"] = Cell(inp["rho"], mat, kind="rho", precision=0 if case["dtype"] == "f64" else 1)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

_E11 = np.zeros((6, 6))
_E11[0, 0] = 1.0


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "step":
        cell = st["cell"]
        cell.update(st["new"])
        cell.solve()
        sens = cell.sensitivity if case["input"] == "rho" else cell.sensitivity_phi
        if case["loads"] != 511:   # one strain load: the gradient of C_11
            return {"g": sens(dC=_E11, dtype=torch.float32)}
        C, e, kap = cell.homogenise()
        dh, dC, de = figure("d_h", C, e)
        return {"C": C, "e": e, "kappa": kap, "d_h": dh, "g": sens(dC=dC, de=de, dtype=torch.float32)}
    if k == "batch":
        for c, d in zip(st["cells"], st["new"]):
            c.update(d)
        solve_batch(st["cells"])
        out = []
        for c in st["cells"]:
            C, e, kap = c.homogenise()
            _, dC, de = figure("d_h", C, e)
            out.append([C, e, kap, c.sensitivity_phi(dC=dC, de=de, dtype=torch.float32)])
        for s in st["streams"]:   # the gradients were written on the handles' streams
            torch.cuda.current_stream().wait_stream(s)
        return out
    if k == "apply":
        return {"y": st["cell"].apply(st["x"])}
    if k == "blocks":
        return {"u": st["cell"].apply_block("A", st["u"]), "p": st["cell"].apply_block("Sbar", st["p"])}
    v, norm, _, mu = st["cell"].hilbert_velocity(st["d"][0], st["d"][1:], st["c"])
    return {"v": v, "norm": norm, "mu": mu, "phi": hj_step(st["phi"], v, 1e-3)}


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: inputs read once, outputs written once (for solves: the design,
    the FP64 solution fields and the sensitivities).  Operations: one
    application of the assembled operators that the pass evaluates (1024
    multiply-adds per element and vector for the coupled one), once per load
    for a solve: any solver checks its residual."""
    k = case["kind"]
    if k == "batch":
        nn = sum(int(v) ** 3 for v in case["sizes"].split(","))
        return {"bytes": nn * (8 + 9 * 32), "flops": 9 * 2048 * nn}
    nn = case["nx"] * case["ny"] * case["nz"]
    size = 8 if case["dtype"] == "f64" else 4
    if k == "step":
        loads = bin(case["loads"]).count("1")
        return {"bytes": nn * (size + loads * 32 + 4), "flops": loads * 2048 * nn}
    if k == "apply":
        return {"bytes": nn * (size + case["nrhs"] * 8 * size), "flops": case["nrhs"] * 2048 * nn}
    if k == "blocks":
        return {"bytes": nn * size * (2 + case["nrhs"] * 8), "flops": case["nrhs"] * 2 * (576 + 64) * nn}
    nv = 1 + case["ncons"]
    return {"bytes": nn * 8 * (nv + 3), "flops": nn * (nv * 54 + 60)}


# ---------------------------------------------------------------------------
# 64-bit values of the outputs
# ---------------------------------------------------------------------------

def _element(nx, ny, nz):
    """Nondimensional element matrix [[A, B^T], [B, -C]] (32 x 32, local dof
    4 node + component, node = x + 2y + 4z), the affine loads at the local
    nodes (32 x 9) and the scales (C0, k0): 2x2x2 Gauss integration."""
    C, e, kap = _material()
    C0, k0 = np.abs(C).max(), np.abs(kap).max()
    C, e, kap = C / C0, e / math.sqrt(C0 * k0), kap / k0
    D = np.block([[C, e.T], [e, -kap]])
    h = np.array([1.0 / nx, 1.0 / ny, 1.0 / nz])
    gp = (0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0))
    K = np.zeros((32, 32))
    for q in range(8):
        xi = [gp[(q >> d) & 1] for d in range(3)]
        B = np.zeros((9, 32))
        for n in range(8):
            bit = [(n >> d) & 1 for d in range(3)]
            f = [xi[d] if bit[d] else 1.0 - xi[d] for d in range(3)]
            s = [1.0 if b else -1.0 for b in bit]
            g = [s[0] * f[1] * f[2] / h[0], f[0] * s[1] * f[2] / h[1], f[0] * f[1] * s[2] / h[2]]
            o = 4 * n
            B[0, o], B[1, o + 1], B[2, o + 2] = g
            B[3, o + 1], B[3, o + 2] = g[2], g[1]
            B[4, o], B[4, o + 2] = g[2], g[0]
            B[5, o], B[5, o + 1] = g[1], g[0]
            B[6, o + 3], B[7, o + 3], B[8, o + 3] = g
        K += B.T @ D @ B * (h.prod() / 8.0)
    Z = np.zeros((32, 9))
    for n in range(8):
        x = np.array([(n >> d) & 1 for d in range(3)]) * h
        o = 4 * n
        Z[o, 0], Z[o + 1, 1], Z[o + 2, 2] = x
        Z[o + 1, 3], Z[o + 2, 3] = x[2] / 2, x[1] / 2
        Z[o, 4], Z[o + 2, 4] = x[2] / 2, x[0] / 2
        Z[o, 5], Z[o + 1, 5] = x[1] / 2, x[0] / 2
        Z[o + 3, 6:9] = -x
    return 0.5 * (K + K.T), Z, C0, k0


def _corners(t):
    """(..., nz, ny, nx) nodal values -> the 8 corner values of every element."""
    return torch.stack([torch.roll(t, (-(a >> 2), -((a >> 1) & 1), -(a & 1)), (-3, -2, -1)) for a in range(8)])


def _to_nodes(f):
    """Adjoint of _corners: sum the 8 corner contributions at the nodes."""
    return sum(torch.roll(f[a], (a >> 2, (a >> 1) & 1, a & 1), (-3, -2, -1)) for a in range(8))


def _multiply(K, rho, x):
    """sum_e rho_e P_e^T K P_e x for one vector x (nc, nz, ny, nx)."""
    nc = x.shape[0]
    u = _corners(x).reshape(8 * nc, -1)
    f = (torch.as_tensor(K, device=x.device) @ u) * rho.reshape(1, -1)
    return _to_nodes(f.reshape((8, nc) + tuple(rho.shape)))


def _exact_step(case, inp):
    """Dense solve of the nine cell problems, for small grids."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    N = nx * ny * nz
    d = inp["new"].double()
    drho = None
    if case["input"] == "rho":
        rho = d
    else:
        eta = 2.0 * max(1.0 / nx, 1.0 / ny, 1.0 / nz)
        t = (_corners(d).sum(0) * 0.125 / eta).clamp(-1.0, 1.0)
        rho = 1.0 - (1.0 - RHO_VOID) * 0.5 * (1.0 + t + torch.sin(math.pi * t) / math.pi)
        drho = -(1.0 - RHO_VOID) * 0.5 * (1.0 + torch.cos(math.pi * t)) / eta * (t.abs() < 1.0)
    K, Z, C0, k0 = _element(nx, ny, nz)
    K, Z = torch.as_tensor(K, device="cuda"), torch.as_tensor(Z, device="cuda")
    node = _corners(torch.arange(N, device="cuda").reshape(nz, ny, nx)).reshape(8, N)
    dof = (4 * node[:, None, :] + torch.arange(4, device="cuda")[None, :, None]).reshape(32, N)
    A = torch.zeros(16 * N * N, dtype=torch.float64, device="cuda")
    r = rho.reshape(-1)
    for a in range(32):
        for b in range(32):
            A.index_add_(0, dof[a] * (4 * N) + dof[b], r * K[a, b])
    A = A.reshape(4 * N, 4 * N)
    for c in range(4):   # fix the mean of every component
        A[c::4, c::4] += (1.0 if c < 3 else -1.0) / N
    rhs = torch.zeros((4 * N, 9), dtype=torch.float64, device="cuda")
    F = K @ Z
    for a in range(32):
        rhs.index_add_(0, dof[a], -r[:, None] * F[a][None, :])
    y = torch.linalg.solve(A, rhs)
    for _ in range(2):   # refine the solve
        y = y + torch.linalg.solve(A, rhs - A @ y)
    W = y[dof] + Z[:, None, :]                       # 32 x N x 9
    KW = torch.einsum("ab,bnj->anj", K, W)
    H = torch.einsum("n,ani,anj->ij", r, W, KW).cpu().numpy()
    se = math.sqrt(C0 * k0)
    C, e, kap = C0 * H[:6, :6], -se * H[6:, :6], -k0 * H[6:, 6:]
    # d_h = e_3 . S m with S = C^-1, m = (1,1,1,0,0,0)
    S = np.linalg.inv(C)
    m = np.array([1.0, 1, 1, 0, 0, 0])
    w, se3 = S @ m, S.T @ e[2]
    dC, de = -np.outer(se3, w), np.zeros((3, 6))
    de[2] = w
    G = np.zeros((9, 9))
    G[:6, :6] = C0 * dC
    G[6:, :6] = -0.5 * se * de
    G[:6, 6:] = G[6:, :6].T
    g = torch.einsum("ani,ij,anj->n", W, torch.as_tensor(G, device="cuda"), KW).reshape(nz, ny, nx)
    if drho is not None:
        g = _to_nodes((g * drho * 0.125).expand(8, nz, ny, nx))
    return {"C": C, "e": e, "kappa": kap, "d_h": float(e[2] @ w), "g": g}


def _exact_evolve(case, inp):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    alpha = 4.0 / min(nx, ny, nz)
    sm = []
    for n in (nx, ny, nz):
        c = torch.cos(2.0 * math.pi * torch.arange(n, dtype=torch.float64, device="cuda") / n)
        sm.append(((2.0 - 2.0 * c) * n, (4.0 + 2.0 * c) / (6.0 * n)))
    (sx, mx), (sy, my), (sz, mz) = sm
    prod = lambda a, b, c: c[:, None, None] * b[None, :, None] * a[None, None, :]
    lam = alpha ** 2 * (prod(sx, my, mz) + prod(mx, sy, mz) + prod(mx, my, sz)) + prod(mx, my, mz)
    d = inp["d"]
    g = [torch.fft.ifftn(torch.fft.fftn(v) / lam).real for v in d]
    gram = np.array([[float((a * b).sum()) for b in d] for a in g])
    gram = 0.5 * (gram + gram.T)
    n = case["ncons"]
    v, norm2, mu = g[0], gram[0, 0], np.zeros(0)
    coef = np.zeros(n)
    if n:
        R = np.linalg.cholesky(gram[1:, 1:]).T
        p = np.linalg.solve(R.T, gram[1:, 0])
        norm2 = norm2 - p @ p
        mu = np.linalg.solve(R.T, np.array(inp["c"]))
    norm = math.sqrt(norm2)
    v = g[0] / norm
    if n:
        coef = np.linalg.solve(R, mu - p / norm)
        for c, gi in zip(coef, g[1:]):
            v = v + float(c) * gi
    phi = inp["phi"]
    gp = gm = 0.0
    for dim, m in ((2, nx), (1, ny), (0, nz)):
        lo, hi = (phi - torch.roll(phi, 1, dim)) * m, (torch.roll(phi, -1, dim) - phi) * m
        gp = gp + lo.clamp(min=0) ** 2 + hi.clamp(max=0) ** 2
        gm = gm + lo.clamp(max=0) ** 2 + hi.clamp(min=0) ** 2
    new = phi - 1e-3 * (v.clamp(min=0) * gp.sqrt() + v.clamp(max=0) * gm.sqrt())
    return {"v": v, "norm": norm, "mu": mu, "phi": new}


def exact(case, seed):
    k = case["kind"]
    if k == "batch":
        return None
    if k == "step":
        # a dense solve of 4 N unknowns
        if case["loads"] != 511 or case["nx"] * case["ny"] * case["nz"] > 2400:
            return None
        return _exact_step(case, _inputs(case, seed))
    inp = _inputs(case, seed)
    if k == "evolve":
        return _exact_evolve(case, inp)
    K, _, _, _ = _element(case["nx"], case["ny"], case["nz"])
    rho = inp["rho"]
    if k == "apply":
        sign = torch.tensor([1.0, 1.0, 1.0, -1.0], dtype=torch.float64, device="cuda").reshape(4, 1, 1, 1)
        return {"y": torch.stack([sign * _multiply(K, rho, x.double()) for x in inp["x"]])}
    iu = [4 * n + c for n in range(8) for c in range(3)]
    ip = [4 * n + 3 for n in range(8)]
    Au, Bu, Cp = K[np.ix_(iu, iu)], K[np.ix_(ip, iu)], -K[np.ix_(ip, ip)]
    S = Cp + Bu @ np.linalg.solve(Au + 1e-10 * np.eye(24), Bu.T)
    return {"u": torch.stack([_multiply(Au, rho, x.double()) for x in inp["u"]]),
            "p": torch.stack([_multiply(S, rho, x.double()) for x in inp["p"]])}
