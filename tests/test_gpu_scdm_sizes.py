"""SCDM's pivot and column kernels at the edges of their sizes: one and a few
orbitals, rows that are and are not a multiple of a warp, the largest set of the
one-block pivot kernel (160) and one beyond it, sets well beyond, nearly dependent
orbitals (the second Gram-Schmidt pass runs), both precisions where the kernels
differ."""
import numpy as np
import pytest

import gen
from test_gpu_scdm import _check_scdm, _lib  # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec", [(1, "mixed"), (2, "mixed"), (31, "mixed"), (33, "mixed"), (100, "mixed"),
                                    (160, "mixed"), (161, "mixed"), (256, "mixed"), (257, "mixed"),
                                    (33, "fp64")])
def test_scdm_sizes_match_oracle(n, prec):
    cell, ecut = gen.cubic_cell(8.0), 25.0
    psi = gen.random_orbitals(cell, ecut, n, seed=600 + n)
    _check_scdm(dict(cell=cell, ecut=ecut, grid=(16, 16, 16), psi=psi), prec, False)


def test_scdm_cancelling_residuals():
    """Orbitals concentrated around one point: the columns there are nearly
    parallel, so residuals fall far below half the column's length."""
    cell, ecut, n = gen.cubic_cell(8.0), 25.0, 12
    miller = gen.half_sphere(cell, ecut)
    rng = np.random.default_rng(5)
    c = np.stack([gen.gaussian_sum_coefficients(cell, miller, 4.0 + 0.5 * rng.standard_normal((3, 3)),
                                                rng.uniform(0.9, 1.2, 3), rng.standard_normal(3)) for _ in range(n)])
    c[:, 0] = c[:, 0].real
    _check_scdm(dict(cell=cell, ecut=ecut, grid=(16, 16, 16), psi=gen.lowdin(c)), "mixed", False)
