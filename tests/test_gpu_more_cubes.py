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


@pytest.mark.parametrize("n,rows", [(50, 4), (54, 0), (96, 3), (120, 3), (120, 1), (144, 4)])
def test_natural_planes_match_oracle(n, rows, tmp_path, monkeypatch):
    """The hybrid passes on padded natural planes: float4 vectors that cross a
    row (n % 4 == 2), two rows per half-warp (n % 32 == 0), pads on every second
    row (120, at even and odd radices), one block per SM (144); five orbitals
    give 15 pairs, the last transform half empty; two streams, batches of two.
    Same tolerances as the other variants."""
    import torch

    import paper_2110_07670_gb300 as ace
    cell, ecut, no = gen.cubic_cell(10.0), 30.0, 5
    psi = gen.random_orbitals(cell, ecut, no, seed=n)
    ref = oracle.ace_build(psi, cell, (n, n, n), ecut, 0.25)
    d = torch.from_numpy(psi.astype(np.complex64)).cuda()
    # boxes whose variant cannot be asked for take it from a saved choice
    # (variant, streams, row block), keyed as the plan's own line is
    cache = tmp_path / "tune"
    monkeypatch.setenv("ACE_TUNE_CACHE", str(cache))
    if n == 120:
        monkeypatch.setenv("ACE_PAIR_RADIX", {3: "12", 1: "8"}[rows])
    ace.Plan((n, n, n), cell, ecut, no, "mixed", pair_batch=4).close()
    key = cache.read_text().splitlines()[-1].split(" = ")[0]
    r0 = 8 if (n, rows) == (120, 1) else 0
    cache.write_text(f"{key} = 4 2 {rows} {r0}\n")
    plan = ace.Plan((n, n, n), cell, ecut, no, "mixed", pair_batch=4)
    assert plan.config()["pair_variant"] == 4
    _, E = ace.ace_build(plan, d, 0.25)
    W, _ = ace.ace_last_intermediates(plan, no)
    assert abs(E - ref["E_x"]) <= 1e-6 * 3 * no / 4
    assert np.abs(W.cpu().numpy() - ref["W_G"]).max() <= 2e-6 * np.abs(ref["W_G"]).max()
    plan.close()
