"""The gain common to every value of a single-precision transform (its rounded
constants) is divided out: what is left of E_x is rounding, which averages out
over the grid points."""
import gen
import numpy as np
import oracle
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(32, 32, 32), (72, 72, 72), (96, 96, 96), (45, 27, 32)])
def test_energy_has_no_common_gain_error(grid):
    """Rounded constants alone would leave 3.3e-7 to 4e-7 of E_x at 32, 72 and
    96 (18 axis transforms of 1.8e-8 to 2.2e-8 each).  Single rounding errors
    are below 2^-22 of a value after ~50 operations and independent: over the
    products of thousands of grid points less than 1e-8, over the few pair
    sums of E_x at most 2^-24 each; 1e-7 bounds their sum."""
    import torch

    import paper_2110_07670_gb300 as ace
    cell, ecut, no = np.diag([0.3 * n for n in grid]), 30.0, 6
    psi = gen.random_orbitals(cell, ecut, no, seed=grid[0])
    ref = oracle.ace_build(psi, cell, grid, ecut, 0.25)
    plan = ace.Plan(grid, cell, ecut, no, "mixed")
    d = torch.from_numpy(psi.astype(np.complex64)).cuda()
    _, E = ace.ace_build(plan, d, 0.25)
    assert abs(E - ref["E_x"]) <= 1e-7 * abs(ref["E_x"])
    plan.close()
