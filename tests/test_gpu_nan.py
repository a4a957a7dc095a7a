"""NaN and infinity in the operands of the tensor-core products come out as NaN.
The NaN that device arithmetic makes has every bit set, with either sign; a NaN
written by the host does not, so both are tried."""
import gen
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BITS = {"device": 0x7fffffff, "negated": -1, "host": 0x7fc00000, "infinity": 0x7f800000}


def put(c, row, bits):
    """Set the imaginary part of a G != 0 coefficient of c[row] (complex64) to bits."""
    import torch
    torch.view_as_real(c).view(torch.int32)[row, c.shape[1] // 2, 1] = bits


@pytest.mark.parametrize("bits", list(BITS.values()), ids=list(BITS))
@pytest.mark.parametrize("n,trials", [(8, 5), (40, 130)])
def test_apply_keeps_nan(n, trials, bits):
    import torch

    import paper_2110_07670_gb300 as ace
    cell, ecut = gen.cubic_cell(8.0), 20.0
    plan = ace.Plan((32, 32, 32), cell, ecut, n, "mixed")
    xi = torch.from_numpy(gen.random_orbitals(cell, ecut, n, seed=1).astype(np.complex64)).cuda()
    psi = torch.from_numpy(gen.random_trials(cell, ecut, trials, seed=2).astype(np.complex64)).cuda()
    good = ace.ace_apply(plan, xi, psi)
    bad = psi.clone()
    put(bad, 3, bits)
    out = ace.ace_apply(plan, xi, bad)
    rest = [t for t in range(trials) if t != 3]
    assert torch.isnan(torch.view_as_real(out[3])).all()
    assert torch.equal(out[rest], good[rest])
    assert np.isnan(ace.ace_apply_energy(plan, xi, bad))
    # a NaN in xi enters every overlap with that ACE vector
    put(xi, n - 1, bits)
    for prepared in (False, True):
        if prepared:
            ace.ace_apply_prepare(plan, xi)
        assert torch.isnan(torch.view_as_real(ace.ace_apply(plan, xi, psi))).all()
        assert np.isnan(ace.ace_apply_energy(plan, xi, psi))
    plan.close()


@pytest.mark.parametrize("bits", list(BITS.values()), ids=list(BITS))
def test_screen_keeps_nan(bits):
    import torch

    import paper_2110_07670_gb300 as ace
    cell, ecut, n = gen.cubic_cell(8.0), 20.0, 8
    plan = ace.Plan((32, 32, 32), cell, ecut, n, "mixed")
    psi = torch.from_numpy(gen.random_orbitals(cell, ecut, n, seed=1).astype(np.complex64)).cuda()
    _, S = ace.ace_overlap_screen(plan, psi, 0.01)
    put(psi, 2, bits)
    _, S2 = ace.ace_overlap_screen(plan, psi, 0.01)
    # orbitals 2 and 3 share a transform, which mixes them
    assert np.isnan(S2[2:4]).all() and np.isnan(S2[:, 2:4]).all()
    rest = np.array([i for i in range(n) if i not in (2, 3)])
    assert np.array_equal(S2[np.ix_(rest, rest)], S[np.ix_(rest, rest)])
    plan.close()
