"""The calls whose speed counts: ACE builds, the inner-step apply, exact
exchange, the s-MTACE screen and SCDM, through the Python binding, over the
range of boxes, occupied sets, precisions and pair lists that the library takes.

A case is one call on one system.  Its inputs are orthonormal Gaussian-sum
orbitals (three sites per molecule, four orbitals per molecule, molecules on a
jittered lattice; the shape of the paper's water boxes) or random orbitals,
made on the GPU in double precision from the seed alone.  A program that runs
these calls keeps the plan of its box and cutoff, so prepare() creates it.

exact() evaluates the same operators in double precision with torch's FFTs and
dense products: Eq. 2-5 of arXiv:2110.07670 and, for SCDM, its Section 2.4-2.5.
"""
import math

import numpy as np
import torch

import paper_2110_07670_gb300 as ace

ALPHA = 0.25  # PBE0
# Grid spacing of the paper-shaped boxes at 80 Ry: points per bohr.
DENSITY = 5.16

# kind: "build" ace_build, "apply" ace_apply, "exact" hfx_apply_exact, "screen"
#   ace_overlap_screen, "scdm" ace_scdm
# grid: points along each lattice vector; length: cell edge in bohr along the
#   first axis (the others in the ratio of the grid); skew: off-diagonal part of
#   the cell, in edges; n: occupied orbitals; trials: vectors of an apply
# pairs: "all", or the fraction of pairs a distance screen keeps ("near")
# rc: the Coulomb interaction cut off at the sphere radius instead of G = 0 dropped


def _case(name, kind, grid, n, **more):
    c = {"name": name, "kind": kind, "n0": grid[0], "n1": grid[1], "n2": grid[2], "n": n,
         "length": grid[0] / DENSITY, "ecut": 80.0, "skew": 0.0, "fp64": False, "orbitals": "gauss",
         "near": 0.0, "rc": False, "trials": 0, "prepared": False, "energy": False, "preselect": True, "rho_cut": 0.025}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: launches and latency (the repository's small configuration)
        _case("build_8_32", "build", (32, 32, 32), 8, length=10.0, ecut=30.0, orbitals="random"),
        # an odd occupied set in a triclinic cell with three different axes
        _case("build_27_40x48x45", "build", (40, 48, 45), 27, skew=0.08),
        # a mid-sized cell of the batched range, 14 bohr
        _case("build_64_72", "build", (72, 72, 72), 64),
        # 32 water molecules: an outer MTS step, the benchmark's workload
        _case("build_128_96", "build", (96, 96, 96), 128, length=18.6),
        # 64 water molecules: the largest full pair list
        _case("build_256_120", "build", (120, 120, 120), 256, length=23.5),
        # 512 localised orbitals, pairs within 8 bohr: s-MTACE's screened build
        _case("build_512_160_near", "build", (160, 160, 160), 512, length=29.6, orbitals="local", near=8.0),
        # the double-precision form
        _case("build_16_48_fp64", "build", (48, 48, 48), 16, fp64=True),
        # an inner MTS step: K psi and the fast energy on the drifted occupied set
        _case("inner_128x128_96", "apply", (96, 96, 96), 128, length=18.6, trials=128, energy=True),
        # the inner steps of the larger box with xi prepared once per outer step
        _case("apply_256x256_120", "apply", (120, 120, 120), 256, length=23.5, trials=256, prepared=True),
        # the uncompressed operator on a few trial vectors
        _case("exact_48x12_80", "exact", (80, 80, 80), 48, trials=12),
        # the s-MTACE screen of 32 water molecules
        _case("screen_128_96", "screen", (96, 96, 96), 128, length=18.6),
        # s'-MTACE localisation of delocalised orbitals, with the pre-selection
        _case("scdm_128_96", "scdm", (96, 96, 96), 128, length=18.6, orbitals="rotated"),
    ]


def _smooth(lo, hi):
    """Axis lengths 2^a 3^b 5^c."""
    out = []
    for n in range(lo, hi + 1):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def draw(rng):
    kind = rng.choice(["build"] * 5 + ["apply"] * 3 + ["exact", "screen", "scdm"])
    log = lambda a, b: math.exp(rng.uniform(math.log(a), math.log(b)))  # noqa: E731
    sizes = _smooth(30, 160 if kind in ("build", "apply") else 108)
    near = lambda x: min(sizes, key=lambda s: abs(s - x))  # noqa: E731
    n0 = near(log(sizes[0], sizes[-1]))
    grid = (n0, n0, n0) if rng.random() < 0.7 else (n0, near(n0 * rng.uniform(0.8, 1.2)), near(n0 * rng.uniform(0.8, 1.2)))
    N = grid[0] * grid[1] * grid[2]
    fp64 = kind in ("build", "apply", "exact") and rng.random() < 0.2
    density = rng.uniform(5.16, 5.4)
    room = max(2.0, N / density ** 3 / 25.0)  # orbitals of a dense cell
    n = max(1, int(log(2, min(512.0, room))))
    c = _case("", kind, grid, n, length=grid[0] / density, fp64=fp64, skew=rng.choice([0.0, 0.0, 0.1]))
    del c["name"]
    # pair solves times grid points: at most what the largest listed build does
    most = 4e8 if fp64 else 1.2e10
    if kind == "build":
        while c["n"] > 1 and c["n"] * (c["n"] + 1) / 2 * N > most:
            c["n"] = c["n"] * 9 // 10
        c["rc"] = rng.random() < 0.25
        if c["n"] >= 32 and c["skew"] == 0.0 and rng.random() < 0.4:
            c["orbitals"], c["near"] = "local", 8.0
    elif kind == "apply":
        c["trials"] = max(1, min(512, int(c["n"] * log(0.25, 4))))
        c["prepared"] = rng.random() < 0.5
        c["energy"] = rng.random() < 0.3
        while fp64 and c["n"] * c["trials"] * N / 60.0 > 4e8:
            c["trials"], c["n"] = (c["trials"] + 1) // 2, (c["n"] + 1) // 2
    elif kind == "exact":
        c["trials"] = max(1, int(log(1, 16)))
        while c["n"] > 1 and c["n"] * c["trials"] * N > most:
            c["n"] = c["n"] * 9 // 10
    elif kind == "screen":
        c["rho_cut"] = rng.choice([0.025, 0.01, 0.002])
    else:
        # enough orbitals that grid points pass the pre-selection
        c["n"], c["orbitals"] = min(max(24, c["n"]), 192), "rotated"
        if N < 60 ** 3:
            c["n0"] = c["n1"] = c["n2"] = 60
            c["length"] = 60 / density
        c["preselect"] = c["n"] * N > 2.5e7 or rng.random() < 0.5
    return c


# ------------------------------------------------------------------ geometry

def _cell(c):
    h = c["length"] / c["n0"]
    a = np.diag([c["n0"] * h, c["n1"] * h, c["n2"] * h])
    if c["skew"]:
        s = c["skew"] * c["length"]
        a[1, 0], a[2, 0], a[2, 1] = s, -0.5 * s, 0.7 * s
    return a


def _sphere(cell, ecut):
    """Half sphere {h>0} U {h=0,k>0} U {h=k=0,l>=0} of |G|^2 <= ecut, lexicographic."""
    b = 2 * np.pi * np.linalg.inv(cell).T
    lim = [int(math.sqrt(ecut) * np.linalg.norm(cell[i]) / (2 * np.pi)) + 1 for i in range(3)]
    ax = [torch.arange(0 if i == 0 else -lim[i], lim[i] + 1, device="cuda") for i in range(3)]
    H, K, L = (t.reshape(-1) for t in torch.meshgrid(*ax, indexing="ij"))
    m = torch.stack([H, K, L], 1)
    G = m.double() @ torch.from_numpy(b).cuda()
    keep = ((G * G).sum(1) <= ecut) & ((H > 0) | ((H == 0) & (K > 0)) | ((H == 0) & (K == 0) & (L >= 0)))
    return m[keep], G[keep]


def _overlap(a, b):
    """<a_i|b_j> of real functions stored on the half sphere, G = 0 first."""
    x, y = torch.view_as_real(a).reshape(len(a), -1), torch.view_as_real(b).reshape(len(b), -1)
    return 2 * (x @ y.T) - torch.outer(a[:, 0].real, b[:, 0].real)


def _lowdin(c):
    c[:, 0] = c[:, 0].real.to(c.dtype)
    w, v = torch.linalg.eigh(_overlap(c, c))
    return ((v * w.clamp_min(1e-12) ** -0.5) @ v.T).to(c.dtype) @ c


def _random(n, npw, gen):
    c = torch.view_as_complex(torch.randn(n, npw, 2, generator=gen, device="cuda", dtype=torch.float64))
    c[:, 0] = c[:, 0].real.to(c.dtype)
    return c


def _orbitals(c, cell, G, n, gen):
    """n orthonormal orbitals on the half sphere (complex128) and their centres."""
    if c["orbitals"] == "random":
        return _lowdin(_random(n, len(G), gen)), None
    uni = lambda *s: torch.rand(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    A = torch.from_numpy(cell).cuda()
    per = 4 if c["orbitals"] == "gauss" else 1  # orbitals of one molecule
    mol = -(-n // per)
    side = max(1, math.ceil(mol ** (1 / 3) - 1e-9))
    spots = torch.randperm(side ** 3, generator=gen, device="cuda")[:mol]
    frac = torch.stack([spots // side ** 2, spots // side % side, spots % side], 1)
    centres = ((frac.double() + 0.2 + 0.6 * uni(mol, 3)) / side) @ A
    d = torch.randn(mol, 3, 3, generator=gen, device="cuda", dtype=torch.float64)
    sites = centres[:, None] + d / d.norm(dim=2, keepdim=True) * (0.4 + 1.2 * uni(mol, 3, 1))
    out = torch.zeros(n, len(G), device="cuda", dtype=torch.complex128)
    g2, omega = (G * G).sum(1), abs(np.linalg.det(cell))
    for s in range(3):
        sig, wgt = 0.6 + 0.6 * uni(n, 1), torch.randn(n, 1, generator=gen, device="cuda", dtype=torch.float64)
        at = sites[torch.arange(n, device="cuda") // per, s]
        amp = wgt * (4 * math.pi * sig * sig) ** 0.75 * torch.exp(-0.5 * sig * sig * g2) / math.sqrt(omega)
        out += torch.polar(amp.abs(), -(at @ G.T)) * amp.sign()
    out = _lowdin(out)
    if c["orbitals"] == "rotated":  # canonical orbitals spread over the cell
        q, _ = torch.linalg.qr(torch.randn(n, n, generator=gen, device="cuda", dtype=torch.float64))
        out = q.to(out.dtype) @ out
    return out, centres


def _near_pairs(centres, cell, cut):
    """CSR of the pairs i <= j with centres closer than cut (minimum image)."""
    f = centres @ torch.from_numpy(np.linalg.inv(cell)).cuda()
    d = f[:, None] - f[None]
    d = (d - d.round()) @ torch.from_numpy(cell).cuda()
    keep = (d.norm(dim=2) < cut) | torch.eye(len(f), dtype=torch.bool, device="cuda")
    keep = keep.triu().cpu().numpy()
    return np.concatenate([[0], keep.sum(1).cumsum()]).astype(np.int32), np.nonzero(keep)[1].astype(np.int32)


def _inputs(c, seed):
    """What the caller has, in double precision: orbitals, pair list, trials, xi."""
    gen = torch.Generator("cuda").manual_seed(seed)
    cell = _cell(c)
    m, G = _sphere(cell, c["ecut"])
    psi, centres = _orbitals(c, cell, G, c["n"], gen)
    d = {"cell": cell, "m": m, "G": G, "pairs": _near_pairs(centres, cell, c["near"]) if c["near"] else None}
    if c["kind"] == "apply":
        # ACE vectors: the smooth span of the occupied set, lengths of its exchange eigenvalues
        mix = torch.randn(c["n"], c["n"], generator=gen, device="cuda", dtype=torch.float64)
        q, _ = torch.linalg.qr(mix)
        lam = 0.05 + 0.6 * torch.rand(c["n"], 1, generator=gen, device="cuda", dtype=torch.float64)
        d["xi"] = (lam.sqrt() * q).to(psi.dtype) @ (psi + 0.02 * _random(c["n"], len(G), gen) / (1 + (G * G).sum(1)))
    if c["trials"]:
        # trial vectors: the occupied set drifted by inner steps, random ones beyond it
        t = _random(c["trials"], len(G), gen) / (1 + (G * G).sum(1))
        t /= t.norm(dim=1, keepdim=True)
        k = min(c["trials"], c["n"])
        t[:k] = psi[:k] + 0.05 * t[:k]
        d["trials"] = t
    d["psi"] = psi
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    rc = ace.sphere_radius(d["cell"]) if case["rc"] else 0.0
    plan = ace.Plan((case["n0"], case["n1"], case["n2"]), d["cell"], case["ecut"], case["n"],
                    "fp64" if case["fp64"] else "mixed", coulomb_rc=rc)
    s = {"case": case, "plan": plan, "pairs": d["pairs"]}
    for k in ("psi", "xi", "trials"):
        if k in d:
            s[k] = d[k].to(plan.cdtype).contiguous()
    if case["prepared"]:
        ace.ace_apply_prepare(plan, s["xi"])
    if case["kind"] == "screen":
        s["rows"] = np.arange(case["n"]) * case["n"]
    return s


def run(state):
    case, plan = state["case"], state["plan"]
    kind = case["kind"]
    if kind == "build":
        xi, E = ace.ace_build(plan, state["psi"], ALPHA, pairs=state["pairs"])
        return {"xi": xi, "E_x": E}
    if kind == "apply":
        out = {"K": ace.ace_apply(plan, state["xi"], state["trials"])}
        if case["energy"]:
            out["E"] = ace.ace_apply_energy(plan, state["xi"], state["trials"])
        return out
    if kind == "exact":
        return {"V": ace.hfx_apply_exact(plan, state["psi"], ALPHA, state["trials"])}
    if kind == "screen":
        (row_ptr, col), S = ace.ace_overlap_screen(plan, state["psi"], case["rho_cut"])
        # the kept pairs as a map: lists of different inputs have different lengths
        keep = np.zeros(S.shape, np.int8)
        keep.reshape(-1)[col + np.repeat(state["rows"], np.diff(row_ptr))] = 1
        return {"keep": keep, "S": S}
    phi, pivots, O, count = ace.ace_scdm(plan, state["psi"], preselect=case["preselect"])
    # a float: grid points within rounding of an average may fall either way
    return {"phi": phi, "pivots": pivots, "O": O, "candidates": float(count)}


def work(case):
    N = case["n0"] * case["n1"] * case["n2"]
    n, T = case["n"], case["trials"]
    npw = 0.5 * abs(np.linalg.det(_cell(case))) * case["ecut"] ** 1.5 / (6 * math.pi ** 2)
    e = 16 if case["fp64"] else 8
    fft = 5.0 * N * math.log2(N)
    if case["kind"] == "build":
        pairs = n * (n + 1) / 2
        if case["near"]:  # pairs within a sphere of the cell
            pairs = min(pairs, n / 2 * (1 + n * 4.19 * case["near"] ** 3 / abs(np.linalg.det(_cell(case)))))
        # two pair densities per complex transform; forward, Coulomb, inverse, accumulate
        flops = pairs / 2 * (2 * fft + 20 * N) + n * fft + 6.0 * n * n * npw
        return {"bytes": 2 * e * n * npw, "flops": flops}
    if case["kind"] == "apply":
        return {"bytes": e * npw * (n + 2 * T), "flops": 8.0 * n * T * npw}
    if case["kind"] == "exact":
        return {"bytes": e * npw * (n + 2 * T), "flops": n * T / 2 * (2 * fft + 12 * N) + (n / 2 + T) * fft}
    if case["kind"] == "screen":
        return {"bytes": e * n * npw + 8.0 * n * n, "flops": n / 2 * fft + 2.0 * n * n * N}
    m = 0.08 * N if case["preselect"] else N  # candidate points
    return {"bytes": 2 * e * n * npw, "flops": 2 * n * fft + 8.0 * n * N + 2.0 * n * n * m}


def tolerance(case):
    # about four times the largest error against exact() seen over the listed
    # and some thirty drawn cases (1e-15 and 7e-7; single elements 2e-6), with
    # room for less well conditioned occupied sets in double precision
    if case["fp64"]:
        return {"rel": 1e-13, "max": 1e-11}
    return {"rel": 3e-6, "max": 3e-5, "differ": 0.01 if case["kind"] == "scdm" else 0.001}


# ------------------------------------------------------------- in 64 bits

def _box_index(m, grid):
    n0, n1, n2 = grid
    return (m[:, 0] % n0 * n1 + m[:, 1] % n1) * n2 + m[:, 2] % n2


def _to_real(c, m, grid, omega, out=None):
    """Real-space values [rows, N] of half-sphere coefficients."""
    N = grid[0] * grid[1] * grid[2]
    out = torch.empty(len(c), N, device="cuda", dtype=torch.float64) if out is None else out
    ip, im = _box_index(m, grid), _box_index(-m, grid)
    for i in range(0, len(c), 8):
        box = torch.zeros(len(c[i:i + 8]), N, device="cuda", dtype=torch.complex128)
        box[:, im] = c[i:i + 8].conj()
        box[:, ip] = c[i:i + 8]
        out[i:i + 8] = torch.fft.ifftn(box.view(-1, *grid), dim=(1, 2, 3)).real.reshape(-1, N) * (N / math.sqrt(omega))
    return out


def _to_sphere(f, m, grid, scale):
    ip = _box_index(m, grid)
    out = torch.empty(len(f), len(m), device="cuda", dtype=torch.complex128)
    for i in range(0, len(f), 8):
        z = torch.fft.fftn(f[i:i + 8].view(-1, *grid), dim=(1, 2, 3)).reshape(-1, f.shape[1])
        out[i:i + 8] = z[:, ip] * scale
    return out


def _kernel(case, cell):
    """K(G) on the half box of a real transform; folded frequencies."""
    grid = (case["n0"], case["n1"], case["n2"])
    b = torch.from_numpy(2 * np.pi * np.linalg.inv(cell).T).cuda()
    fold = [torch.tensor([i if i < n - n // 2 else i - n for i in range(n)], device="cuda", dtype=torch.float64) for n in grid]
    h, k, l = torch.meshgrid(fold[0], fold[1], fold[2][:grid[2] // 2 + 1], indexing="ij")
    g2 = ((h[..., None] * b[0] + k[..., None] * b[1] + l[..., None] * b[2]) ** 2).sum(-1)
    safe = torch.where(g2 > 0, g2, torch.ones_like(g2))
    if case["rc"]:
        rc = (3 * abs(np.linalg.det(cell)) / (4 * math.pi)) ** (1 / 3)
        return torch.where(g2 > 0, 4 * math.pi * (1 - torch.cos(safe.sqrt() * rc)) / safe, torch.full_like(g2, 2 * math.pi * rc * rc))
    return torch.where(g2 > 0, 4 * math.pi / safe, torch.zeros_like(g2))


def _potential(rho, K, grid):
    f = torch.fft.rfftn(rho.view(-1, *grid), dim=(1, 2, 3))
    return torch.fft.irfftn(f.mul_(K), s=grid, dim=(1, 2, 3)).reshape(rho.shape)


def exact(case, seed):
    d = _inputs(case, seed)
    cell, m, grid = d["cell"], d["m"], (case["n0"], case["n1"], case["n2"])
    N, omega, n = grid[0] * grid[1] * grid[2], abs(np.linalg.det(cell)), case["n"]
    # the values that the call is given, in its own precision
    as_given = (lambda t: t) if case["fp64"] else (lambda t: t.to(torch.complex64).to(torch.complex128))
    psi = as_given(d["psi"])
    if case["kind"] == "apply":
        xi, t = as_given(d["xi"]), as_given(d["trials"])
        C = _overlap(t, xi)
        out = {"K": -(C.to(xi.dtype) @ xi)}
        if case["energy"]:
            out["E"] = float(-(C * C).sum())
        return out
    phi = _to_real(psi, m, grid, omega)
    if case["kind"] == "screen":
        S = torch.zeros(n, n, device="cuda", dtype=torch.float64)
        for x in range(0, N, 1 << 16):
            a = phi[:, x:x + (1 << 16)].abs()
            S += a @ a.T
        S = (S * (omega / N)).cpu().numpy()
        keep = np.triu((S >= case["rho_cut"]) | np.eye(n, dtype=bool))
        return {"keep": keep.astype(np.int8), "S": S}
    if case["kind"] == "scdm":
        return _exact_scdm(psi, phi, m, d["G"], grid, omega, case["preselect"])
    K = _kernel(case, cell)
    step = max(1, int(3e9 // (8 * N)) // 8)
    scale = -ALPHA * math.sqrt(omega) / N
    if case["kind"] == "exact":
        t = _to_real(as_given(d["trials"]), m, grid, omega)
        acc = torch.zeros_like(t)
        for i in range(len(t)):
            for j in range(0, n, step):
                acc[i] += (_potential(phi[j:j + step] * t[i], K, grid) * phi[j:j + step]).sum(0)
        return {"V": _to_sphere(acc, m, grid, scale)}
    W = torch.zeros_like(phi)
    e = torch.zeros((), device="cuda", dtype=torch.float64)
    for i in range(n):
        js = np.arange(i, n) if d["pairs"] is None else d["pairs"][1][d["pairs"][0][i]:d["pairs"][0][i + 1]]
        for x in range(0, len(js), step):
            j = torch.from_numpy(js[x:x + step].astype(np.int64)).cuda()
            f = phi[j]
            v = _potential(f * phi[i], K, grid)
            off = (j != i).double()[:, None]
            e += ((1 + off[:, 0]) * torch.einsum("jr,jr->j", v, f * phi[i])).sum()
            W[i] += torch.einsum("jr,jr->r", v, f)
            W.index_add_(0, j, v.mul_(phi[i]).mul_(off))
    del phi
    W = _to_sphere(W, m, grid, scale)
    M = _overlap(psi, W)
    L = torch.linalg.cholesky(-(M + M.T) / 2)
    xi = torch.linalg.solve_triangular(L, torch.view_as_real(W).reshape(n, -1), upper=False)
    return {"xi": torch.view_as_complex(xi.reshape(n, -1, 2).contiguous()), "E_x": float(-ALPHA * omega / N * e)}


def _exact_scdm(psi, phi, m, G, grid, omega, preselect):
    n = len(psi)
    sel = torch.arange(phi.shape[1], device="cuda")
    if preselect:
        rho = (phi * phi).sum(0)
        g = torch.zeros_like(rho)
        for x in range(3):
            g += ((phi * _to_real(1j * G[:, x] * psi, m, grid, omega)).sum(0) * 2) ** 2
        g = g.sqrt()
        sel = torch.nonzero((rho > rho.mean()) & (g < g.mean()))[:, 0]
    A = phi[:, sel]
    R, nu = A.clone(), (A * A).sum(0)
    piv = []
    for k in range(n):
        p = int(nu.argmax())
        piv.append(p)
        q = R[:, p] / R[:, p].norm()
        R -= torch.outer(q, q @ R)
        nu = (R * R).sum(0)
        nu[torch.tensor(piv, device="cuda")] = -1
    V = A[:, torch.tensor(piv, device="cuda")].T
    U, _, Wh = torch.linalg.svd(V)
    O = U @ Wh
    return {"phi": O.to(psi.dtype) @ psi, "pivots": sel[torch.tensor(piv, device="cuda")].to(torch.int32).cpu().numpy(),
            "O": O.cpu().numpy(), "candidates": float(len(sel))}
