"""The compile-time cubes beyond the requestable pair variants (automatic choice
and tile passes) against the oracle; what was refused on them stays refused."""
import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [36, 40, 48, 50, 54, 64, 72, 128, 144])
def test_cube_matches_oracle(n):
    import torch

    import paper_2110_07670_gb300 as ace
    cell, ecut, no = gen.cubic_cell(10.0), 30.0, 3
    psi = gen.random_orbitals(cell, ecut, no, seed=n)
    ref = oracle.ace_build(psi, cell, (n, n, n), ecut, 0.25)
    d = torch.from_numpy(psi.astype(np.complex64)).cuda()
    for kw in ({}, {"pair_variant": 1}, {"kernels": 2}):
        plan = ace.Plan((n, n, n), cell, ecut, no, "mixed", **kw)
        _, E = ace.ace_build(plan, d, 0.25)
        W, _ = ace.ace_last_intermediates(plan, no)
        assert abs(E - ref["E_x"]) <= 1e-6 * 3 * no / 4
        assert np.abs(W.cpu().numpy() - ref["W_G"]).max() <= 2e-6 * np.abs(ref["W_G"]).max()
        plan.close()
    for v in (2, 3, 4, 5):
        with pytest.raises(ace.AceError):
            ace.Plan((n, n, n), cell, ecut, no, "mixed", pair_variant=v)
