"""The counters and phases of the fast energy: its Gram, and the sum over it."""
import gen
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,kernels", [("mixed", 0), ("mixed", 1), ("fp64", 0)])
def test_fast_energy_has_its_phase_and_its_launches(prec, kernels):
    import torch

    import paper_2110_07670_gb300 as ace
    cell, ecut, n = gen.cubic_cell(8.0), 20.0, 8
    plan = ace.Plan((32, 32, 32), cell, ecut, n, prec, kernels=kernels)
    xi = torch.from_numpy(gen.random_orbitals(cell, ecut, n, seed=1)).to(plan.cdtype).cuda()
    ace.ace_apply_energy(plan, xi, xi)
    ace.ace_set_timing(plan, True)
    ace.ace_get_stats(plan)
    ace.ace_apply_energy(plan, xi, xi)
    st = ace.ace_get_stats(plan)
    assert st["launches"] == 3  # the Gram, its finish, the sum
    assert st["gram_ms"] > 0 and st["energy_ms"] > 0
    plan.close()
