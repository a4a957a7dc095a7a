"""The runtime-size plane and pencil kernels (csrc/generic.cuh) against the
oracle, on boxes at their edges: odd planes (single pencils, odd rows), rows
that are and are not a multiple of four, axes of one, two and three FFT stages,
lines shorter than a warp, pencil groups with a remainder.  An odd number of
orbitals leaves a half-empty transform in every pass."""
import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu

# an FP32 3D FFT of these sizes has about 1e-7 relative rms error and W sums
# at most 5 of them: the parity tolerances of the library
TOL_E, TOL_W = 1e-6, 2e-6


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("grid", [(15, 9, 25), (27, 45, 15), (20, 16, 18), (9, 8, 250), (250, 10, 12), (5, 162, 6),
                                  (12, 75, 54), (6, 5, 4 * 27), (10, 12, 15)])
@pytest.mark.parametrize("cut", [False, True])
def test_generic_boxes_match_oracle(grid, cut):
    import torch

    import paper_2110_07670_gb300 as ace
    # a spacing of 0.55 bohr: at 20 Ry every axis of five points or more holds the sphere
    cell = np.diag([0.55 * n for n in grid])
    ecut, n = 20.0, 5
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
