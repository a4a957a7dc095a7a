"""The sums of a Gram's float slices in three floats (la.cu sum_add3): no
further from the exact sum than a sum in double.  On the host with numpy's
float32 rounding, on the GPU where the sums leave the range of a float."""
from fractions import Fraction

import numpy as np
import pytest

f32 = np.float32


def two_sum(s, x):
    t = f32(s + x)
    b = f32(t - s)
    return t, f32(f32(s - f32(t - b)) + f32(x - b))


def sum_add3(acc, x):
    s, e1 = two_sum(acc[0], x)
    e, e2 = two_sum(acc[1], e1)
    return s, e, f32(acc[2] + e2)


@pytest.mark.parametrize("n,spread,seed", [(18, 0, 1), (18, 8, 2), (300, 4, 3), (1000, 12, 4)])
def test_three_float_sum_is_as_good_as_double(n, spread, seed):
    """Four interleaved sums combined, as the kernel does; each rounding to double
    at the end is within 2^-53 of the sum, what the float sums lose far below
    2^-53 of the sum of magnitudes (a pair of floats alone loses 2^-47 of it)."""
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal(n) * 10.0 ** rng.uniform(-spread, 0, n)).astype(f32)
    if seed == 2:  # cancelling to a few small terms
        x = np.concatenate([x, -x[:-3]])
    exact, scale = sum(Fraction(float(v)) for v in x), float(np.abs(x.astype(np.float64)).sum())
    part = [(f32(0), f32(0), f32(0))] * 4
    for i, v in enumerate(x):
        part[i % 4] = sum_add3(part[i % 4], v)
    s = part[0]
    for o in part[1:]:
        s = sum_add3(s, o[0])
        e, err = two_sum(s[1], o[1])
        s = (s[0], e, f32(s[2] + f32(err + o[2])))
    got = float(s[0]) + (float(s[1]) + float(s[2]))
    assert abs(Fraction(got) - exact) <= abs(exact) * Fraction(2) ** -53 + Fraction(scale) * Fraction(2) ** -60


@pytest.mark.gpu
def test_sums_beyond_the_range_of_a_float():
    """Slices of 1.5e38 each, 142 of them: the overlaps are finite in double, and
    so is the energy.  Slices that overflow themselves give infinity, no NaN."""
    import gen
    import torch

    import paper_2110_07670_gb300 as ace
    cell, ecut, n = gen.cubic_cell(12.0), 60.0, 4
    plan = ace.Plan((32, 32, 32), cell, ecut, n, "mixed")
    for a in (1.25e18, 1e20):
        c = torch.full((n, plan.n_pw_half), complex(a, a), dtype=torch.complex64, device="cuda")
        c[:, 0] = a
        v = torch.view_as_real(c).double().reshape(n, -1)
        ref = -float(((2 * v @ v.T - torch.outer(v[:, 0], v[:, 0])) ** 2).sum())
        E = ace.ace_apply_energy(plan, c, c)
        if a < 1e19:
            assert abs(E - ref) <= 1e-6 * abs(ref)  # (a float's range, and its precision)
        else:
            assert E == -np.inf
    plan.close()
