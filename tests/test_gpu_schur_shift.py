"""The shift of the local Schur complement on every level of the hierarchy.

The finest grid decides which shifts are accepted: S0 = C_e + B_e (A_e + shift
I)^-1 B_e^T exists where the factorisation of A_e + shift I does (A_e is singular:
rigid modes), which rounding decides for shifts near 1e-17.  A handle whose
finest element matrices exist sets up and solves, whatever its coarse levels'
element matrices do; C^H, e^H, kappa^H do not depend on the shift (1e-8, the energy
form's error at tol 1e-10).
"""
import numpy as np
import pytest
import torch

import cellgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_03148_gb300 import load
    return load()


@pytest.mark.parametrize("shape", [(32, 32, 32), (20, 34, 17), (9, 10, 33)])
def test_shifts_at_the_rounding_limit(shape):
    from paper_2410_03148_gb300 import Cell
    from paper_2410_03148_gb300 import _binding as B
    phi = torch.as_tensor(cellgen.gaussian_levelset(shape, seed=3), device="cuda:0")
    mat = cellgen.pzt5h_class()
    ref = Cell(phi, mat)
    ref.solve()
    want = ref.homogenise()
    accepted = 0
    for shift in (1e-19, 3e-19, 1e-18, 2e-18, 4e-18, 8e-18, 2e-17, 1e-16, 1e-3, 1.0):
        desc = B.make_desc(tuple(reversed(shape)), *mat, phi.data_ptr(), B.CELL_INPUT_PHI, B.CELL_F64,
                           B.cell_default_options(schur_shift=shift), 0, 1e-3, 0.0)
        try:
            B.cell_element_matrices(desc)
        except B.CellError:
            continue
        accepted += 1
        cell = Cell(phi, mat, schur_shift=shift)
        cell.solve()
        for x, y in zip(cell.homogenise(), want):
            assert np.abs(x - y).max() <= 1e-8 * np.abs(y).max(), shift
        cell.close()
    assert accepted >= 3
