"""Solver path of materials without the mm2 mirror planes: corner-form
operators, tensor-core smoothers on the finest grid, Galerkin levels with
assembled 27-point stencils, constant-bank slots.  (mm2 materials take the
modal operators on rediscretised levels through the whole solve and launch
none of these.)

Grids, as nz x ny x nx: 16^3 has an elastic level of 8^3 nodes with a stencil
(small: the four-lane kernel) above the dense 4^3 one; 24 x 20 x 32 halves to 12
x 10 x 16 and 6 x 5 x 8 (stencils, a dense coarsest level of 720 unknowns); 17 x
16 x 12 does not coarsen (Chebyshev on the finest level); 40 x 36 x 48 has 8640
nodes on level 1 (the one-thread-per-node stencil kernel, whose loads per thread
are tuned) and 1080 on the coarsest, which for the elastic block is too large
for a dense inverse.

Bounds: equal tensors where only launch geometry differs (bitwise); C^H, e^H,
kappa^H to 1e-8 of the block's largest entry otherwise (tol 1e-10: the energy
form's error is quadratic in the solve's), 1e-10 between two mixed solves of
the same arithmetic.
"""
import functools

import numpy as np
import pytest
import torch

import cellgen
from oracle import ersatz, fem, laminate, precond, sensitivity
from oracle.material import nondimensionalise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_03148_gb300 import load
    return load()


def material():
    """PZT-5H constants with a small normal-shear and shear-shear coupling, an
    e11 and an off-diagonal permittivity (positive definite)."""
    C, e, k = (np.array(v, dtype=float) for v in cellgen.pzt5h_class())
    C[0, 3] = C[3, 0] = 2.0e9
    C[4, 5] = C[5, 4] = 1.5e9
    e[0, 0] = 1.0
    k[0, 1] = k[1, 0] = 1.0e-9
    return C, e, k


def make_cell(phi, **opt):
    from paper_2410_03148_gb300 import Cell
    return Cell(torch.as_tensor(phi, device="cuda:0"), material(), kind="phi", **opt)


def solved(phi, **opt):
    c = make_cell(phi, **opt)
    st = c.solve()
    assert max(st["rel_residual"]) <= 1e-10
    out = c.homogenise()
    c.close()
    return st, out


def close(a, b, tol):
    return all(np.abs(x - y).max() <= tol * np.abs(y).max() for x, y in zip(a, b))


@functools.lru_cache(maxsize=None)
def oracle_16():
    phi = cellgen.gaussian_levelset(16, seed=1)
    return phi, fem.solve_cell(ersatz.rho_from_levelset(phi), *material())


def tensors(ref):
    return tuple(ref[k] for k in ("C", "e", "kappa"))


@pytest.mark.parametrize("opt", [{"tensor_cores": 0}, {"tensor_cores": 1}, {"tensor_cores": 2}, {"graphs": 0},
                                 {"precision": 0}, {"cheb_degree": 2, "vcycles_u": 2, "vcycles_phi": 2},
                                 {"precond": 1, "max_iter": 2000}])
def test_solve_with_a_stencil_level_matches_oracle(opt):
    phi, ref = oracle_16()
    st, out = solved(phi, **opt)
    assert st["nlevels_u"] == 3
    assert close(out, tensors(ref), 1e-8), st


@pytest.mark.parametrize("shape", [(16, 16, 16), (3, 17, 23), (7, 31, 24), (40, 16, 32)])
def test_operators_match_oracle(shape):
    """Corner-form operators over several blocks of a plane (the last one
    ragged), FP64, FP32 and FP32 pairs, nine loads; tolerances of the oracle
    parity tests."""
    from paper_2410_03148_gb300 import Cell
    from paper_2410_03148_gb300 import _binding as B
    M = material()
    rho = cellgen.random_rho(shape, seed=21)
    cell = Cell(torch.as_tensor(rho, device="cuda:0"), M, kind="rho", autotune=0, restart=2)
    N = rho.size
    P = fem.CellProblem(rho, *M)
    Cn, en, kn, _ = nondimensionalise(*M)
    K0 = fem.element_matrix(Cn, en, kn, fem.cell_h(shape))
    full, sign = P.Kg.tocsr().astype(float), np.tile([1.0, 1.0, 1.0, -1.0], N)[:, None]
    ops = [("full", 4, lambda v: sign * (full @ v), np.abs(K0).max())]
    for blk, nc in (("A", 3), ("Sbar", 1)):
        Ke = precond.block_matrix(K0, blk)
        A = precond.assemble_block(rho, Ke, nc, shape)
        ops.append((blk, nc, lambda v, A=A: A @ v, np.abs(Ke).max()))
    x = np.random.default_rng(22).standard_normal((9, 4) + shape)
    for name, nc, mul, kmax in ops:
        v = x[:, :nc]
        for dt, tol in ((torch.float64, 1e-12), (torch.float32, 2e-6), ("pairs", 32 * 2e-14)):
            if dt == "pairs" and name != "full":
                continue
            xt = torch.as_tensor(np.ascontiguousarray(v), device="cuda:0", dtype=torch.float64 if dt == "pairs" else dt)
            if dt == "pairs":
                y = torch.empty_like(xt)
                B.cell_apply(cell._h, xt.data_ptr(), y.data_ptr(), 9, B.CELL_F64_DF)
            else:
                y = cell.apply(xt) if name == "full" else cell.apply_block(name, xt)
            xd = xt.double().cpu().numpy().reshape(9, nc, N).transpose(2, 1, 0).reshape(-1, 9)
            want = mul(xd).reshape(N, nc, 9).transpose(2, 1, 0).reshape(v.shape)
            err = np.abs(y.double().cpu().numpy() - want).max()
            assert err < tol * 8 * kmax * np.abs(v).max(), (name, dt, err)


@pytest.mark.parametrize("gdtype,tol", [(torch.float64, 1e-8), (torch.float32, 1e-5)])
@pytest.mark.parametrize("precision", [0, 1])
def test_sensitivities_match_oracle(precision, gdtype, tol):
    """Element and nodal sensitivities with full upstream gradients."""
    phi, ref = oracle_16()
    rng = np.random.default_rng(5)
    dC, de, dk = rng.standard_normal((6, 6)), rng.standard_normal((3, 6)), rng.standard_normal((3, 3))
    cell = make_cell(phi, precision=precision)
    cell.solve()
    P = ref["problem"]
    g_rho = sensitivity.grad_rho(P, ref["y"], sensitivity.G_from_si(dC, de, dk, P.sc))
    g_phi = ersatz.grad_phi(phi, g_rho)
    for got, want in ((cell.sensitivity(dC, de, dk, dtype=gdtype), g_rho),
                      (cell.sensitivity_phi(dC, de, dk, dtype=gdtype), g_phi)):
        assert np.abs(got.double().cpu().numpy() - want).max() < tol * np.abs(want).max()


@pytest.mark.parametrize("tc", [0, 1, 2])
@pytest.mark.parametrize("n,axis", [(32, 0), (64, 2)])
def test_laminate_closed_form(n, axis, tc):
    from paper_2410_03148_gb300 import Cell
    rho = cellgen.laminate_rho((n, n, n), axis, seed=7 + axis)
    layers = {0: rho[0, 0, :], 1: rho[0, :, 0], 2: rho[:, 0, 0]}[axis]
    cell = Cell(torch.as_tensor(np.ascontiguousarray(rho), device="cuda:0"), material(), kind="rho", tensor_cores=tc)
    cell.solve()
    assert close(cell.homogenise(), laminate.laminate_tensors(*material(), layers, axis)[:3], 1e-8)


@pytest.mark.parametrize("precision", [0, 1])
def test_graphs_and_updates(precision):
    """Direct launches, per-iteration graphs and the whole-solve graph, on a
    fresh handle and on one that held another design, give the same bits."""
    first, second = (cellgen.gaussian_levelset(16, seed=s) for s in (21, 22))
    want = solved(second, precision=precision, graphs=0)
    for graphs in (0, 1, 2):
        c = make_cell(first, precision=precision, graphs=graphs)
        c.solve()
        c.update(torch.as_tensor(second, device="cuda:0"))
        st = c.solve()
        assert st["iters"] == want[0]["iters"] and st["rel_residual"] == want[0]["rel_residual"]
        assert all(np.array_equal(x, y) for x, y in zip(c.homogenise(), want[1]))
        c.close()


@pytest.mark.parametrize("shape", [(24, 20, 32), (17, 16, 12)])
def test_smoother_tiles(shape):
    """Forced CTA tiles of the tensor-core smoothers (ragged x tiles, y tiles and
    z chunks, one or two M tiles per warp) in every mode of the V-cycle."""
    phi = cellgen.gaussian_levelset(shape, seed=8)
    outs = []
    for xt, L in ((16, 5), (8, 3), (32 if shape[2] >= 32 else 16, 64)):
        c = make_cell(phi, autotune=0, graphs=0, max_iter=2000)
        for blk in ("A", "Sbar"):
            c.set_tile(blk, xt, L)
        st = c.solve()
        assert st["tc_tiles"][0]["xt"] == xt
        outs.append((st["iters"], c.homogenise()))
        c.close()
    for its, H in outs[1:]:
        assert its == outs[0][0]
        assert all(np.array_equal(x, y) for x, y in zip(H, outs[0][1]))
    _, smoothed_in_fp32 = solved(phi, tensor_cores=0, max_iter=2000)
    assert close(outs[0][1], smoothed_in_fp32, 1e-8)


def test_tuned_tiles():
    phi = cellgen.gaussian_levelset(24, seed=31)
    sa, a = solved(phi, autotune=0)
    sb, b = solved(phi, autotune=1)
    assert sa["iters"] == sb["iters"] and all(np.array_equal(x, y) for x, y in zip(a, b))
    assert all(t["xt"] in (8, 16, 32) and t["us"] > 0 for t in sb["tc_tiles"])


def test_constant_bank_and_parameter_kernels():
    """Element matrices from a constant-bank slot or from the kernel parameter:
    the same arithmetic in a possibly different order."""
    phi = cellgen.gaussian_levelset(16, seed=13)
    _, a = solved(phi, const_bank=0, tensor_cores=0)
    _, b = solved(phi, const_bank=1, tensor_cores=0)
    assert close(a, b, 1e-10)


def test_stencil_loads_per_thread():
    phi = cellgen.gaussian_levelset((40, 36, 48), seed=5)
    st, ref = solved(phi)
    for blk in range(2):
        assert st["stencil_rg"][blk][0] == 0 and st["stencil_rg"][blk][1] in (1, 3, 9)
    for rg in (1, 3, 9):
        c = make_cell(phi, autotune=0, graphs=0)
        for blk, n in (("A", st["nlevels_u"]), ("Sbar", st["nlevels_phi"])):
            for lev in range(1, n):
                c.set_stencil_rg(blk, lev, rg)
        s = c.solve()
        assert s["iters"] == st["iters"]
        assert all(np.array_equal(x, y) for x, y in zip(c.homogenise(), ref))
        c.close()


@pytest.mark.parametrize("graphs", [2, 3])
def test_batch(graphs):
    """Uneven designs solved in one call equal their single solves bitwise."""
    from paper_2410_03148_gb300 import solve_batch
    phis = [cellgen.gaussian_levelset(n, seed=40 + n) for n in (16, 8, 24)]
    cells = [make_cell(p, graphs=graphs) for p in phis]
    solve_batch(cells)
    got = [c.homogenise() for c in cells]
    for c in cells:
        c.close()
    for p, g in zip(phis, got):
        _, one = solved(p, autotune=0)
        assert all(np.array_equal(x, y) for x, y in zip(g, one))
