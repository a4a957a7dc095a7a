"""The pivoted QR of single-precision columns against sums in extended precision:
its vectors are orthonormal to double, its rows of R are float-float dot products.
Sizes on both sides of the one-block pivot kernel's largest set; smooth columns,
whose residuals cancel, and random ones."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PTRS = "part nu R Q r c nu0 rdiag piv status"


class _Work(ctypes.Structure):
    _fields_ = [(k, ctypes.c_void_p) for k in PTRS.split()] + [("blocks", ctypes.c_int)]


def _columns(smooth, n, m):
    import torch
    g = torch.Generator("cuda").manual_seed(n)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    if not smooth:
        return rnd(n, m).float()
    x, c = (18 * torch.rand(k, 3, generator=g, device="cuda", dtype=torch.float64) for k in (m, n))
    f = sum(rnd(n, 1) * torch.exp(-torch.cdist(c + 0.8 * rnd(n, 3), x) ** 2 / 2) for _ in range(3))
    return (torch.linalg.qr(rnd(n, n))[0] @ f).float().contiguous()


@pytest.mark.parametrize("n,m", [(8, 3000), (33, 6001), (128, 22000), (160, 22000), (161, 22000)])
@pytest.mark.parametrize("smooth", [False, True])
def test_qr_is_orthonormal_to_double(n, m, smooth):
    import torch

    import paper_2110_07670_gb300 as ace
    lib = ctypes.CDLL(ace.library_path())
    vp, ll = ctypes.c_void_p, ctypes.c_longlong
    blocks = lib._ZN3ace14scdm_qr_blocksExii
    blocks.argtypes = [ll, ctypes.c_int, ctypes.c_int]
    init = lib._ZN3ace14launch_qr_initIfEE9cudaErrorPKT_ixPdPviP11CUstream_st
    init.argtypes = [vp, ctypes.c_int, ll, vp, vp, ctypes.c_int, vp]
    step = lib._ZN3ace14launch_qr_stepIfEE9cudaErrorPKT_ixiNS_6QrWorkEP11CUstream_st
    step.argtypes = [vp, ctypes.c_int, ll, ctypes.c_int, _Work, vp]
    A = _columns(smooth, n, m)
    qb = blocks(m, n, 4)
    size = dict(part=2 * qb, nu=m, R=n * m, Q=n * n, r=n, c=n, nu0=1, rdiag=n, piv=n, status=1)
    buf = {k: torch.zeros(s, dtype=torch.int32 if k in ("piv", "status") else torch.float64, device="cuda")
           for k, s in size.items()}
    w = _Work(*[buf[k].data_ptr() for k in PTRS.split()], qb)
    torch.cuda.synchronize()
    assert init(A.data_ptr(), n, m, w.nu, w.part, qb, None) == 0
    for k in range(n):
        assert step(A.data_ptr(), n, m, k, w, None) == 0
    torch.cuda.synchronize()
    assert int(buf["status"]) == 0
    piv = buf["piv"].cpu().numpy()
    assert len(set(piv.tolist())) == n
    # one unit of rounding per projection and what it cancels, 16 in all; with
    # float-float coefficients it is 2^-48, some 32
    Q = buf["Q"].view(n, n).cpu().numpy().astype(np.longdouble)
    assert np.abs(Q @ Q.T - np.eye(n)).max() <= 16 * 2.0 ** -53
    # R = Q A where a column was not yet chosen: float-float products, 2^-47, and
    # 2^-149 for each of a term's roundings below a float's normal range
    a = A[:, ::97].cpu().numpy().astype(np.longdouble)
    R, alive = buf["R"].view(n, m)[:, ::97].cpu().numpy(), np.ones(a.shape, bool)
    for k, p in enumerate(piv):
        if p % 97 == 0:
            alive[k:, p // 97] = False
    assert (np.abs(R - Q @ a)[alive] <= (2.0 ** -47 * (np.abs(Q) @ np.abs(a)))[alive] + n * 2.0 ** -147).all()
    # the pivots' residual lengths
    ap = A[:, torch.from_numpy(piv).long().cuda()].cpu().numpy().astype(np.longdouble)
    d = np.einsum("ki,ik->k", Q, ap)
    assert np.abs(buf["rdiag"].cpu().numpy() - d).max() <= 1e-14 * np.abs(ap).sum(0).max()
