"""GPU parity of the modal element operators (mm2 materials) and of the corner
form that serves other materials, against the FP64 oracle, at the edges of the
modal kernels' work split: blocks own 30 columns of a sequence with nx + 2
positions per strip of 3, 7, 11 or 15 node rows (the four warps exchange the row
between them) and march through chunks of z planes.  Shapes (nz, ny, nx) cover
rows that end a window or start one (nx = 28 .. 31, 58 .. 61), rows shorter than
a strip (ny = 2, 3), whole and ragged last strips (ny = 7, 11, 15, 16, 33), the
smallest periodic sizes, several strips per window (small nx) and several
chunks.  Tolerances: those of the oracle parity tests (FP64 1e-12, FP32 2e-6 of
max|K| max|x| x 8; the FP32-pair residual 2e-14 of 8 x 32 terms), and for
materials without the mirror planes the same.
"""
import numpy as np
import pytest
import torch

import cellgen
from oracle import fem, material, precond

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_03148_gb300 import load
    return load()


def general_material():
    """The mm2 constants with a small normal-shear and shear-shear coupling, an
    e11 and an off-diagonal permittivity (still positive definite)."""
    C, e, k = (np.array(v, dtype=float) for v in cellgen.pzt5h_class())
    C[0, 3] = C[3, 0] = 2.0e9
    C[4, 5] = C[5, 4] = 1.5e9
    e[0, 0] = 1.0
    k[0, 1] = k[1, 0] = 1.0e-9
    return C, e, k


SHAPES = [(2, 2, 2), (3, 2, 28), (2, 3, 29), (3, 5, 30), (5, 4, 31), (2, 7, 58), (3, 6, 61), (9, 8, 3), (33, 9, 16),
          (6, 33, 5), (3, 11, 9), (5, 15, 8), (4, 16, 30), (4, 64, 64), (40, 45, 50)]


@pytest.mark.parametrize("shape,mat", [(s, "mm2") for s in SHAPES] + [(s, "general") for s in SHAPES[:3]])
def test_operators_match_oracle(shape, mat):
    from paper_2410_03148_gb300 import Cell
    from paper_2410_03148_gb300 import _binding as B
    M = cellgen.pzt5h_class() if mat == "mm2" else general_material()
    dev = torch.device("cuda:0")
    rho = cellgen.random_rho(shape, seed=21)
    cell = Cell(torch.as_tensor(rho, device=dev), M, kind="rho", autotune=0, restart=4)
    N = rho.size
    rng = np.random.default_rng(22)
    P = fem.CellProblem(rho, *M)
    Cn, en, kn, _ = material.nondimensionalise(*M)
    K0 = fem.element_matrix(Cn, en, kn, fem.cell_h(shape))
    full = P.Kg.tocsr().astype(float)
    sign = np.tile([1.0, 1.0, 1.0, -1.0], N)[:, None]
    ops = [("full", 4, lambda v: sign * (full @ v), np.abs(K0).max())]
    for blk, nc in (("A", 3), ("Sbar", 1)):
        Ke = precond.block_matrix(K0, blk)
        A = precond.assemble_block(rho, Ke, nc, shape)
        ops.append((blk, nc, lambda v, A=A: A @ v, np.abs(Ke).max()))
    for name, nc, mul, kmax in ops:
        for nrhs in (1, 9):
            x = rng.standard_normal((nrhs, nc) + shape)
            for dt, tol in ((torch.float64, 1e-12), (torch.float32, 2e-6)):
                xt = torch.as_tensor(x, device=dev, dtype=dt)
                y = cell.apply(xt) if name == "full" else cell.apply_block(name, xt)
                xd = xt.double().cpu().numpy().reshape(nrhs, nc, N).transpose(2, 1, 0).reshape(-1, nrhs)
                want = mul(xd).reshape(N, nc, nrhs).transpose(2, 1, 0).reshape(x.shape)
                err = np.abs(y.double().cpu().numpy() - want).max()
                assert err < tol * 8 * kmax * np.abs(x).max(), (name, nrhs, dt, err)
            if name == "full":
                xt = torch.as_tensor(x, device=dev)
                y = torch.empty_like(xt)
                B.cell_apply(cell._h, xt.data_ptr(), y.data_ptr(), nrhs, B.CELL_F64_DF)
                xd = x.reshape(nrhs, nc, N).transpose(2, 1, 0).reshape(-1, nrhs)
                want = mul(xd).reshape(N, nc, nrhs).transpose(2, 1, 0).reshape(x.shape)
                err = np.abs(y.cpu().numpy() - want).max()
                assert err < 2e-14 * 8 * 32 * kmax * np.abs(x).max(), (nrhs, err)


def test_large_grid_sbar_matches_fp64():
    """Sbar in FP32 above the size from which a warp takes six element rows (23
    node rows per strip, ragged here), against the FP64 kernel (FP32 bound
    2e-6 of max|S0| max|x| x 8)."""
    from paper_2410_03148_gb300 import Cell
    from paper_2410_03148_gb300 import _binding as B
    M = cellgen.pzt5h_class()
    shape = (77, 85, 91)
    cell = Cell(torch.as_tensor(cellgen.random_rho(shape, seed=5), device="cuda:0"), M, kind="rho", autotune=0, restart=1)
    x = torch.randn((9, 1) + shape, device="cuda:0", dtype=torch.float32, generator=torch.Generator("cuda:0").manual_seed(1))
    y = cell.apply_block("Sbar", x).double()
    want = cell.apply_block("Sbar", x.double())
    S0 = B.cell_element_matrices(cell._desc)[1]
    assert float((y - want).abs().max()) < 2e-6 * 8 * np.abs(S0).max() * float(x.abs().max())


@pytest.mark.parametrize("shape", [(6, 7, 5), (8, 8, 8)])
@pytest.mark.parametrize("precision", [0, 1])
def test_general_material_solve_matches_oracle(shape, precision):
    """A material without the mirror planes takes the corner-form operators and
    the Galerkin hierarchy through the whole solve."""
    from paper_2410_03148_gb300 import Cell
    from oracle import ersatz
    M = general_material()
    phi = cellgen.gaussian_levelset(shape, seed=2)
    ref = fem.solve_cell(ersatz.rho_from_levelset(phi), *M)
    cell = Cell(torch.as_tensor(phi, device="cuda:0"), M, kind="phi", precision=precision)
    cell.solve()
    for got, key in zip(cell.homogenise(), ("C", "e", "kappa")):
        assert np.abs(got - ref[key]).max() < 1e-8 * np.abs(ref[key]).max(), key


@pytest.mark.parametrize("shape", [(9, 7, 10), (3, 12, 5), (2, 5, 24), (11, 10, 9)])
@pytest.mark.parametrize("opt", [{}, {"cheb_degree": 1}, {"cheb_degree": 2}, {"cheb_degree": 4}, {"vcycles_u": 2, "vcycles_phi": 2},
                                 {"coarse_dofs": 1}, {"coarse_dofs": 600, "precond": 1}, {"precision": 0},
                                 {"precision": 0, "cheb_degree": 5}])
def test_rediscretised_hierarchy_options(shape, opt):
    """Odd, elongated and 3-node axes (coarse grids of any ratio up to 2, axes
    coarsened one after another), every parity of the smoothing degree (which
    buffer holds the iterate), repeated V-cycles, the coarsest sizes: the solve
    meets its residual tolerance and C^H, e^H, kappa^H the oracle's (1e-8, the
    energy form's error at tol 1e-10)."""
    from paper_2410_03148_gb300 import Cell
    from oracle import ersatz
    M = cellgen.pzt5h_class()
    phi = cellgen.gaussian_levelset(shape, seed=4)
    ref = fem.solve_cell(ersatz.rho_from_levelset(phi), *M)
    cell = Cell(torch.as_tensor(phi, device="cuda:0"), M, kind="phi", max_iter=2000, **opt)
    st = cell.solve()
    assert max(st["rel_residual"]) <= 1e-10
    for got, key in zip(cell.homogenise(), ("C", "e", "kappa")):
        assert np.abs(got - ref[key]).max() < 1e-8 * np.abs(ref[key]).max(), key


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("opt", [{"restart": 3}, {"restart": 17, "inner_tol": 1e-7}, {"restart": 40, "inner_tol": 1e-12, "max_refine": 4},
                                 {"restart": 63, "inner_tol": 1e-12, "max_refine": 3, "cheb_degree": 1, "vcycles_phi": 1}])
def test_arnoldi_step_lengths(precision, opt):
    """Every form of the Gram-Schmidt kernels: up to 4, 8 and 16 basis vectors in
    registers, more read twice (an inner tolerance below FP32 rounding keeps a
    cycle going to its restart length), short restarts, one and two entries
    per lane of the forward substitution (up to 63 vectors)."""
    from paper_2410_03148_gb300 import Cell
    from oracle import ersatz
    shape = (7, 10, 9)
    M = cellgen.pzt5h_class()
    phi = cellgen.gaussian_levelset(shape, seed=6)
    ref = fem.solve_cell(ersatz.rho_from_levelset(phi), *M)
    cell = Cell(torch.as_tensor(phi, device="cuda:0"), M, kind="phi", **{"precision": precision, "max_iter": 2000, **opt})
    st = cell.solve()
    assert max(st["rel_residual"]) <= 1e-10
    for got, key in zip(cell.homogenise(), ("C", "e", "kappa")):
        assert np.abs(got - ref[key]).max() < 1e-8 * np.abs(ref[key]).max(), key
