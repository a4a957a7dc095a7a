"""The runtime-size tile passes (csrc/pass_kernel.cuh) in single precision, on the
boxes that the plane and pencil kernels leave to them: planes beyond a block's
shared memory (separate x, y and z passes; with and without bulk copies and
four-wide vectors), pencils beyond it, extents of one.  Against the oracle, with
the tolerances of the other single-precision boxes."""
import gen
import numpy as np
import oracle
import pytest

pytestmark = pytest.mark.gpu

TOL_E, TOL_W = 1e-6, 2e-6


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("grid,cut", [((6, 180, 180), False), ((6, 180, 180), True), ((5, 135, 225), False),
                                      ((4, 162, 180), True), ((1800, 4, 6), False), ((1, 12, 10), False),
                                      ((12, 1, 10), False), ((10, 12, 1), False)])
def test_tile_passes_match_oracle(grid, cut):
    import torch

    import paper_2110_07670_gb300 as ace
    # a spacing of 0.55 bohr: at 20 Ry every axis of five points or more holds the sphere
    cell = np.diag([0.55 * n for n in grid])
    ecut, n = 20.0, 3
    psi = gen.random_orbitals(cell, ecut, n, seed=sum(grid))
    rc = ace.sphere_radius(cell) if cut else 0.0
    if cut:
        with oracle.coulomb_cutoff(rc):
            ref = oracle.ace_build(psi, cell, grid, ecut, 0.25)
    else:
        ref = oracle.ace_build(psi, cell, grid, ecut, 0.25)
    plan = ace.Plan(grid, cell, ecut, n, "mixed", coulomb_rc=rc)
    d = torch.from_numpy(psi.astype(np.complex64)).cuda()
    _, E = ace.ace_build(plan, d, 0.25)
    W, _ = ace.ace_last_intermediates(plan, n)
    assert abs(E - ref["E_x"]) <= TOL_E * 3 * n / 4
    assert rel(W.cpu().numpy(), ref["W_G"]) <= TOL_W
    if not cut:
        tr = gen.random_trials(cell, ecut, 3, seed=1)
        V = ace.hfx_apply_exact(plan, d, 0.25, torch.from_numpy(tr.astype(np.complex64)).cuda())
        assert rel(V.cpu().numpy(), oracle.vx_apply(psi, tr, cell, grid, ecut, 0.25)) <= TOL_W
    plan.close()
