"""A build refused for its pair list: the call's stream has read the orbitals by
then, also behind other work on it, and later calls on other streams judge their
own orbitals.  Orbitals refused at the Gamma point are named first, as before the
list is looked at."""
import gen
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BAD = [(np.array([0, 1, 1, 1, 1, 1, 1, 1, 1], np.int32), np.array([8], np.int32)),  # column out of range
       (np.array([0, 2, 1, 1, 1, 1, 1, 1, 1], np.int32), np.array([0, 1], np.int32)),  # rows not monotone
       (np.array([1, 1, 1, 1, 1, 1, 1, 1, 1], np.int32), np.array([0], np.int32))]  # not from 0


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("pairs", BAD)
def test_refused_pair_list_leaves_the_stream_idle(pairs, prec):
    import torch

    import paper_2110_07670_gb300 as ace
    s = gen.config_small()
    n = len(s["psi"])
    assert n == 8
    plan = ace.Plan(s["grid"], s["cell"], s["ecut"], n, prec)
    psi = torch.from_numpy(s["psi"].astype(np.complex64 if prec == "mixed" else np.complex128)).cuda()
    odd = psi.clone()
    odd[3, 0] = 0.5j
    _, E = ace.ace_build(plan, psi, 0.25)
    side = torch.cuda.Stream()
    for call in (ace.ace_build, ace.ace_build_pairs):
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(200_000_000)  # a tenth of a second
        with pytest.raises(ace.AceError, match="pair"):
            call(plan, psi, 0.25, pairs=pairs, stream=side)
        assert side.query()
        with pytest.raises(ace.AceError, match="vector 3"):
            call(plan, odd, 0.25)
        with pytest.raises(ace.AceError, match="vector 3"):
            call(plan, odd, 0.25, pairs=pairs)
        assert abs(call(plan, psi, 0.25)[1] - E) <= 1e-6 * abs(E)
    plan.close()
