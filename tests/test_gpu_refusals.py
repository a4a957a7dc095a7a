"""Calls refused at the Gamma point after work has been enqueued: the caller's
output and the last build's intermediates stay as they were, and the plan goes
on working."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_gamma_refusal_leaves_results_alone(prec):
    import torch

    import paper_2110_07670_gb300 as ace
    s = gen.config_small()
    n = len(s["psi"])
    plan = ace.Plan(s["grid"], s["cell"], s["ecut"], n, prec)
    psi = torch.from_numpy(s["psi"].astype(np.complex64 if prec == "mixed" else np.complex128)).cuda()
    xi, E = ace.ace_build(plan, psi, 0.25)
    W, M = ace.ace_last_intermediates(plan, n)
    bad = psi.clone()
    bad[n - 1, 0] = 0.5j
    keep = xi.clone()
    for call in (lambda: ace.ace_build(plan, bad, 0.25, xi=xi), lambda: ace.ace_build_pairs(plan, bad, 0.25),
                 lambda: ace.hfx_apply_exact(plan, psi, 0.25, bad), lambda: ace.ace_overlap_screen(plan, bad, 0.01)):
        with pytest.raises(ace.AceError):
            call()
    W2, M2 = ace.ace_last_intermediates(plan, n)
    assert torch.equal(xi, keep) and torch.equal(W, W2) and np.array_equal(M, M2)
    _, E2 = ace.ace_build(plan, psi, 0.25)
    assert abs(E2 - E) <= 1e-6 * abs(E)
    plan.close()
