"""The CUDA-core Gram multiplies only the 16 x 16 register tiles that hold rows
and columns: sizes on both sides of every tile count."""
import gen
import numpy as np
import oracle
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,trials", [(1, 1), (15, 17), (16, 33), (17, 16), (32, 49), (33, 15), (5, 65)])
def test_apply_on_cuda_core_gram(n, trials, prec):
    """K psi of given xi against NumPy in double, within the worst case of the
    rounding: a Gram entry sums slices of 32 products in the plan's precision
    (33 eps of the sum of their magnitudes) and rounds once, the product adds n
    terms (n + 1 eps); real and imaginary parts of xi are at most |xi|."""
    import torch

    import paper_2110_07670_gb300 as ace
    cell, ecut, grid = gen.cubic_cell(8.0), 20.0, (32, 32, 32)
    rng = np.random.default_rng(n * 100 + trials)
    plan = ace.Plan(grid, cell, ecut, max(n, 1), prec, kernels=1)
    ct = np.complex128 if prec == "fp64" else np.complex64
    npw = gen.random_orbitals(cell, ecut, 1, seed=0).shape[1]

    def rand(k):
        a = rng.standard_normal((k, npw)) + 1j * rng.standard_normal((k, npw))
        a[:, 0] = a[:, 0].real
        return a.astype(ct)

    xi, psi = rand(n), rand(trials)
    out = ace.ace_apply(plan, torch.from_numpy(xi).cuda(), torch.from_numpy(psi).cuda()).cpu().numpy()
    x, p = xi.astype(np.complex128), psi.astype(np.complex128)
    c = 2.0 * (p @ x.conj().T).real - np.outer(p[:, 0].real, x[:, 0].real)
    ref = -c @ x
    eps = 2.0 ** -52 if prec == "fp64" else 2.0 ** -23
    ab = 2.0 * np.abs(p.view(np.float64)) @ np.abs(x.view(np.float64)).T  # sums of the products' magnitudes
    bound = (33 + 1 + n + 1) * eps * (ab @ np.abs(x))
    assert (np.abs(out - ref) <= np.sqrt(2.0) * bound).all()
    plan.close()
