"""Performance cases of the LTMP2 library: what a program that uses it calls, with inputs of
the kind it meets, the least work of each pass, and the same results in plain 64-bit torch.

Every case builds a mean field first: seeded Gaussian wells in a cubic cell, a plane-wave
sphere, orbitals and energies from a dense diagonalisation, all other orbitals virtual.  The
sizes are those of the repository's own workloads and tests: the 8^3 and 12^3 test systems,
the systems of the batching workload (r = 0.375 n, 6 bohr per well, two occupied orbitals
per well, 6 to 10 Laplace points) and the 24^3 benchmark system.
"""
import math

import numpy as np
import torch

import paper_1611_06797_gb300 as L

FP = {"fp64": L.FP64, "fp32": L.FP32}


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # one small cell, the shortest call: launches and latency
        dict(name="energy_f64_8", kind="energy", prec="fp64", real=True, grid=8, a=5.5, r2=9, wells=2, n_occ=2,
             n_tau=6, levels=0),
        # small cell with a handful of occupied orbitals
        dict(name="energy_f64_12", kind="energy", prec="fp64", real=True, grid=12, a=6.0, r2=25, wells=2, n_occ=4,
             n_tau=6, levels=0),
        # orbitals with arbitrary phases (no time-reversal pairing)
        dict(name="energy_f64_complex_16", kind="energy", prec="fp64", real=False, grid=16, a=9.524406, r2=36,
             wells=4, n_occ=8, n_tau=6, levels=0),
        # an ordinary whole energy in double precision
        dict(name="energy_f64_20", kind="energy", prec="fp64", real=True, grid=20, a=13.736571, r2=56, wells=12,
             n_occ=24, n_tau=7, levels=0),
        # one share (of eight) of the outer G' loop of the benchmark system: a rank of a
        # sharded run, or a chunk of a checkpointed one
        dict(name="share_f64_24", kind="share", prec="fp64", real=True, grid=24, a=12.0, r2=81, wells=16, n_occ=32,
             n_tau=8, part=3, parts=8),
        # the benchmark system's whole energy in the precision form
        dict(name="energy_f32_24", kind="energy", prec="fp32", real=True, grid=24, a=12.0, r2=81, wells=16,
             n_occ=32, n_tau=8, levels=0),
        # an odd grid and a large system in the precision form, one share of its outer loop
        dict(name="share_f32_27", kind="share", prec="fp32", real=True, grid=27, a=19.048813, r2=102, wells=32,
             n_occ=64, n_tau=9, part=15, parts=32),
        # internal cutoff extrapolation: energies on eight nested auxiliary spheres
        dict(name="levels_f64_18", kind="energy", prec="fp64", real=True, grid=18, a=12.0, r2=45, wells=8, n_occ=16,
             n_tau=6, levels=8),
        # k-point sampling of the small cell, both precisions
        dict(name="kpoints_f64_12", kind="kpoints", prec="fp64", grid=12, a=6.0, r2=25, wells=2, n_occ=2, n_tau=6,
             mesh1=2, mesh2=2, mesh3=1),
        dict(name="kpoints_f32_12", kind="kpoints", prec="fp32", grid=12, a=6.0, r2=25, wells=2, n_occ=2, n_tau=6,
             mesh1=2, mesh2=2, mesh3=2),
        # an open shell: two spin channels of different occupation
        dict(name="uhf_f64_16", kind="uhf", prec="fp64", real=True, grid=16, a=9.524406, r2=36, wells=4, n_occ=9,
             n_occ_b=7, n_tau=6),
        # the double-precision product on its own, ragged sizes
        dict(name="dgemm_f64", kind="dgemm", m=4501, n=3071, k=3039),
    ]


# one system of each grid the batching workload and the tests use
_SIZES = [(8, 9), (10, 12), (12, 20), (16, 36), (18, 45), (20, 56), (24, 81), (25, 87), (27, 102)]


def draw(rng):
    kind = rng.choice(["energy", "energy", "energy", "share", "share", "kpoints", "uhf", "dgemm"])
    if kind == "dgemm":
        size = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return dict(kind=kind, m=size(65, 6000), n=size(33, 3200), k=size(17, 3200))
    prec = rng.choice(["fp64", "fp32"])
    if kind == "kpoints":
        grid, r2 = rng.choice([(8, 9), (10, 12), (12, 25)])
        mesh = rng.choice([(2, 1, 1), (1, 3, 1), (2, 2, 1), (1, 2, 2), (2, 2, 2)])
        wells = rng.choice([1, 2])   # one filled band per well keeps a gap
        return dict(kind=kind, prec=prec, grid=grid, a=round(rng.uniform(5.0, 6.5), 6), r2=r2, wells=wells,
                    n_occ=wells, n_tau=rng.choice([3, 4, 6]), mesh1=mesh[0], mesh2=mesh[1], mesh3=mesh[2])
    top = 7 if kind == "share" else 6 if prec == "fp32" else 5
    at = rng.randrange(3 if kind == "share" else 0, min(top, 4) if kind == "uhf" else top + (kind == "share"))
    grid, r2 = _SIZES[at]
    r2 -= rng.randrange(0, max(1, r2 // 8))
    # wells up to the batching workload's number at that grid (4 at 16^3 .. 32 at 27^3)
    most = max(1, int(round(4.0 * (grid / 16.0) ** 3)))
    wells = max(2, rng.randint(max(1, most // 3), most))   # one well alone has degenerate levels
    n_occ = max(1, min(2 * wells + rng.choice([-1, 0, 0, 1]), 64))
    case = dict(kind=kind, prec=prec, real=rng.random() < (0.75 if grid <= 16 else 1.0), grid=grid,
                a=round(6.0 * wells ** (1.0 / 3.0) + rng.uniform(-0.3, 0.3), 6), r2=r2, wells=wells, n_occ=n_occ,
                n_tau=rng.randint(4, 8))
    if kind == "share":
        case["parts"] = rng.randint(10, 40) if grid > 20 else rng.randint(3, 9)
        case["part"] = rng.randrange(case["parts"])
    elif kind == "uhf":
        case["n_occ_b"] = max(1, n_occ - rng.randint(0, 2))
    else:
        case["levels"] = rng.choice([0, 0, 0, 4, 8]) if grid <= 20 else 0
    return case


# ---------------------------------------------------------------- mean field
def _sphere(r2):
    R = int(math.isqrt(int(r2))) + 1
    x = np.arange(-R, R + 1)
    m = np.stack(np.meshgrid(x, x, x, indexing="ij"), -1).reshape(-1, 3)
    s = (m * m).sum(1)
    m, s = m[s <= r2], s[s <= r2]
    return m[np.lexsort((m[:, 2], m[:, 1], m[:, 0], s))]


def _factors(n):
    """n = n1 n2 n3, as nearly cubic as it goes."""
    best = (n, 1, 1)
    for x in range(1, n + 1):
        if n % x == 0:
            for y in range(1, n // x + 1):
                if (n // x) % y == 0:
                    f = (x, y, n // x // y)
                    if max(f) - min(f) < max(best) - min(best):
                        best = f
    return tuple(sorted(best, reverse=True))


def _positions(wells, a, rng):
    """Wells on a site lattice, displaced by 0.2 bohr."""
    f = _factors(wells)
    idx = np.stack(np.meshgrid(*[np.arange(k) for k in f], indexing="ij"), -1).reshape(-1, 3)
    return (idx + 0.5) * (a / np.array(f, dtype=float)) + rng.normal(0.0, 0.2, size=(wells, 3))


def _potential(a, pos, R, depth=2.0, width=0.8):
    """V(G) of Gaussian wells on the box |m| <= R of Miller indices, [2R+1]^3."""
    b = 2.0 * math.pi / a
    k = np.arange(-R, R + 1) * b
    ph = [np.exp(-1j * np.outer(pos[:, c], k)) * np.exp(-0.5 * (k * width) ** 2)[None, :] for c in range(3)]
    s = np.einsum("wx,wy,wz->xyz", ph[0], ph[1], ph[2], optimize=True)
    return s * (-(depth / a ** 3) * (2.0 * math.pi * width ** 2) ** 1.5)


class _Solid:
    pass


def _eigh(H):
    """Eigenvalues in ascending order (equal ones come back in either order) and vectors."""
    e, v = torch.linalg.eigh(H)
    e, order = torch.sort(e, stable=True)
    return e, v[:, order]


def _gather(V, m1, m2, sign):
    """V(m1 + sign m2) for all pairs, from the box table V."""
    R = (V.shape[0] - 1) // 2
    d = [m1[:, None, c] + sign * m2[None, :, c] + R for c in range(3)]
    return V[d[0], d[1], d[2]]


def _gamma_solid(case, seed, depth=2.0):
    """Orbitals of one closed-shell cell: dense diagonalisation in the cos/sin basis (real
    orbitals), each times its own phase when the case asks for general ones."""
    a, grid = case["a"], case["grid"]
    rng = np.random.default_rng([seed, 11])
    pos = _positions(case["wells"], a, rng)
    mil = _sphere(case["r2"])
    if 2 * np.abs(mil).max() >= grid:
        raise ValueError("the sphere does not fit the grid")
    R = 2 * int(np.abs(mil).max())
    V = torch.from_numpy(_potential(a, pos, R, depth)).cuda()
    first = np.where(mil[:, 0] != 0, mil[:, 0], np.where(mil[:, 1] != 0, mil[:, 1], mil[:, 2]))
    P = np.nonzero(first > 0)[0]
    key = {tuple(m): k for k, m in enumerate(mil.tolist())}
    Q = np.array([key[tuple(-x for x in m)] for m in mil[P].tolist()])
    zero = key[(0, 0, 0)]
    mp = torch.from_numpy(mil[P]).cuda()
    n = len(P)
    dif, add = _gather(V, mp, mp, -1), _gather(V, mp, mp, 1)
    H = torch.empty((2 * n + 1, 2 * n + 1), dtype=torch.float64, device="cuda")
    H[1:n + 1, 1:n + 1] = dif.real + add.real
    H[n + 1:, n + 1:] = dif.real - add.real
    H[1:n + 1, n + 1:] = dif.imag - add.imag
    H[n + 1:, 1:n + 1] = H[1:n + 1, n + 1:].T
    v0 = _gather(V, mp, torch.zeros((1, 3), dtype=mp.dtype, device="cuda"), 1)[:, 0] * math.sqrt(2.0)
    H[0, 0] = V[R, R, R].real
    H[0, 1:n + 1] = H[1:n + 1, 0] = v0.real
    H[0, n + 1:] = H[n + 1:, 0] = -v0.imag
    kin = 0.5 * (2.0 * math.pi / a) ** 2 * (mp.double() ** 2).sum(1)
    H.diagonal()[1:] += torch.cat([kin, kin])
    eps, vec = _eigh(H)
    vt = vec.T / math.sqrt(2.0)
    co = torch.zeros((2 * n + 1, 2 * n + 1), dtype=torch.complex128, device="cuda")
    co[:, zero] = vec[0, :].to(co.dtype)
    co[:, torch.from_numpy(P).cuda()] = torch.complex(vt[:, 1:n + 1], -vt[:, n + 1:])
    co[:, torch.from_numpy(Q).cuda()] = torch.complex(vt[:, 1:n + 1], vt[:, n + 1:].contiguous())
    if not case["real"]:
        ph = rng.random(2 * n + 1) * 2.0 * math.pi
        co *= torch.polar(torch.ones(2 * n + 1, dtype=torch.float64), torch.from_numpy(ph)).cuda()[:, None]
    s = _Solid()
    s.lattice = np.eye(3) * a
    s.grid = np.array([grid] * 3, dtype=np.int32)
    s.miller = mil.astype(np.int32)
    s.coeff = co.cpu().numpy()
    s.eps = eps.cpu().numpy()
    s.n_occ = case["n_occ"]
    s.ecut_aux = 2.0 / 3.0 * 0.5 * (case["r2"] + 1e-6) * (2.0 * math.pi / a) ** 2
    return s


def _kpoint_solid(case, seed):
    """Bloch orbitals on a Gamma-centred mesh, one plane-wave set for every k."""
    a, grid = case["a"], case["grid"]
    mesh = np.array([case["mesh1"], case["mesh2"], case["mesh3"]])
    rng = np.random.default_rng([seed, 13])
    pos = _positions(case["wells"], a, rng)
    if case["wells"] == 2:   # body-centred, which keeps a gap between the bands
        pos = np.array([[0.25] * 3, [0.75] * 3]) * a + rng.normal(0.0, 0.2, size=(2, 3))
    mil = _sphere(case["r2"])
    R = 2 * int(np.abs(mil).max())
    m = torch.from_numpy(mil).cuda()
    V = _gather(torch.from_numpy(_potential(a, pos, R)).cuda(), m, m, -1)
    kappa = np.stack(np.meshgrid(*[np.arange(x) for x in mesh], indexing="ij"), -1).reshape(-1, 3)
    co, ep = [], []
    for kap in kappa:
        G = (mil + kap / mesh) * (2.0 * math.pi / a)
        H = V.clone()
        H.diagonal().add_(torch.from_numpy(0.5 * (G * G).sum(1)).cuda())
        e, v = _eigh(H)
        co.append(v.T.contiguous().cpu().numpy())
        ep.append(e.cpu().numpy())
    s = _Solid()
    s.lattice, s.grid, s.mesh, s.kappa = np.eye(3) * a, np.array([grid] * 3, dtype=np.int32), mesh, kappa
    s.miller, s.coeff, s.eps, s.n_occ = mil.astype(np.int32), np.stack(co), np.stack(ep), case["n_occ"]
    s.ecut_aux = 2.0 / 3.0 * 0.5 * (case["r2"] + 1e-6) * (2.0 * math.pi / a) ** 2
    return s


def _gap_width(s):
    e = np.atleast_2d(s.eps)
    return float(e[:, s.n_occ].min() - e[:, s.n_occ - 1].max()), float(e.max() - e.min())


def _quadrature(solids, n_tau):
    """An exponential sum for 1/x on the range of the denominators: the trapezoid rule in ln tau,
    with the step that balances its own error and the two tails."""
    lo, hi = zip(*[_gap_width(s) for s in solids])
    xmin, xmax = 2.0 * min(lo), 2.0 * max(hi)
    h = 1.0
    for _ in range(200):
        C = math.pi ** 2 / h
        h = 0.5 * (h + (math.log(C * xmax / xmin) + C) / n_tau)
    t = -math.pi ** 2 / h - math.log(xmax) + h * (np.arange(n_tau) + 0.5)
    return np.exp(t), h * np.exp(t)


def _inputs(case, seed):
    kind = case["kind"]
    if kind == "kpoints":
        s = [_kpoint_solid(case, seed)]
    elif kind == "uhf":
        # the minority electrons see wells of 0.9 times the depth
        s = [_gamma_solid(case, seed), _gamma_solid(dict(case, n_occ=case["n_occ_b"]), seed, depth=1.8)]
    else:
        s = [_gamma_solid(case, seed)]
    tau, w = _quadrature(s, case["n_tau"])
    return s, tau, w


def _range(case, n_prim):
    """The part-th of `parts` balanced shares of the outer loop."""
    return case["part"] * n_prim // case["parts"], (case["part"] + 1) * n_prim // case["parts"]


# ---------------------------------------------------------------- what a program holds, and one pass
def prepare(case, seed):
    if case["kind"] == "dgemm":
        g = torch.Generator(device="cuda").manual_seed(seed)
        rnd = lambda r, c: torch.randn(r, c, generator=g, device="cuda", dtype=torch.float64)
        # rows of different magnitude, as products over orbitals have
        a = rnd(case["m"], case["k"]) * torch.exp(3.0 * rnd(case["m"], 1))
        b = rnd(case["n"], case["k"]) * torch.exp(3.0 * rnd(case["n"], 1))
        return dict(case=case, a=a, b=b)
    s, tau, w = _inputs(case, seed)
    prec = FP[case["prec"]]
    if case["kind"] == "kpoints":
        x = s[0]
        ctx = [L.ltmp2_setup_kpoints(x.lattice, x.grid, x.mesh, x.miller, x.coeff, x.eps, x.n_occ, x.ecut_aux, prec)]
    else:
        flags = L.FLAG_REAL_ORBITALS if case["real"] else 0
        ctx = [L.ltmp2_setup(x.lattice, x.grid, x.miller, x.coeff, x.eps, x.n_occ, x.ecut_aux, prec, flags) for x in s]
    if case.get("levels"):
        L.ltmp2_set_extrapolation(ctx[0], case["levels"])
    return dict(case=case, ctx=ctx, tau=tau, w=w)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "dgemm":
        return L.ltmp2_dgemm_nt(state["a"], state["b"])
    ctx, tau, w = state["ctx"], state["tau"], state["w"]
    if kind == "share":
        b, e = _range(case, L.ltmp2_num_primary_gprime(ctx[0]))
        ed, ex, pd, px = L.ltmp2_energy_partial(ctx[0], tau, w, b, e)
        return [np.array([ed, ex]), pd, px]
    if kind == "uhf":
        ed, ex, es = L.ltmp2_energy_uhf(ctx[0], ctx[1], tau, w)
        return [np.array([ed, ex]), es]
    ed, ex, pair = L.ltmp2_energy(ctx[0], tau, w)
    out = [np.array([ed, ex]), pair]
    if case.get("levels"):
        lev = L.ltmp2_level_energies(ctx[0])
        out += [lev["E_d"], lev["E_x"]]
    return out


# ---------------------------------------------------------------- the least work of one pass
def _columns(r2):
    """(points, columns, m1 range) of the sphere |m|^2 <= r2."""
    R = int(math.isqrt(int(r2)))
    pts = cols = 0
    for x in range(-R, R + 1):
        for y in range(-R, R + 1):
            rest = r2 - x * x - y * y
            if rest >= 0:
                cols += 1
                pts += 2 * int(math.floor(math.sqrt(rest))) + 1
    return pts, cols, 2 * R + 1


def work(case):
    """One E_MP2: per Laplace point the virtuals' Green's function and the transformed states (or
    both through the virtuals alone), the line transforms of the co-densities of every
    unordered pair, kept to the columns that the auxiliary sphere needs (5 n log2 n a line),
    and the two contractions; the orbitals read once and the pair energies written once."""
    if case["kind"] == "dgemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8 * (m * k + n * k + m * n), "flops": 2 * m * n * k}
    npw, dorb, xorb = _columns(case["r2"])
    naux, daux, xaux = _columns((case["r2"] + 1e-6) * 2.0 / 3.0)
    n, nt = case["grid"], case["n_tau"]
    line = 5.0 * n * math.log2(n)
    nk = case.get("mesh1", 1) * case.get("mesh2", 1) * case.get("mesh3", 1)
    prim = nk * naux // 2 if case["kind"] != "share" else naux // 2 / case["parts"]
    real = case.get("real", False)
    spins = [case["n_occ"]] + ([case["n_occ_b"]] if case["kind"] == "uhf" else [])
    flops = byts = 0.0
    for no in spins:
        NO = no * nk
        cols = prim * NO * (1 if real else 2)
        # a real Green's function where the orbitals are real: half and a quarter of the products
        # (its columns are complex); the last Laplace points hold few virtuals, counted as half
        flops += 0.5 * nt * ((2 if real else 8) * nk * npw * npw * (npw - no) + (4 if real else 8) * cols * npw * npw)
        flops += nt * cols * (dorb + n * (xorb + n)) * line                      # w to real space
        items = cols * (NO + 1) / 2
        flops += nt * items * (2 * n ** 3 + (n * (n + xaux) + daux) * line)      # products and co-densities
        flops += nt * prim * (NO * (NO + 1) / 2 * 2) * 8 * naux                   # exchange and direct sums
        byts += 16 * nk * npw * npw + 8 * NO * NO
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    """About four times the largest distance from exact() seen over the listed cases and a dozen drawn
    ones: 6e-15 in double precision (sums over all G, G' and Laplace points, of both signs for
    the exchange term), 1e-6 in the precision form, 2e-15 for the product."""
    if case["kind"] == "dgemm":
        return {"rel": 8e-15}
    return {"rel": 3e-14} if case["prec"] == "fp64" else {"rel": 5e-6}


# ---------------------------------------------------------------- 64 bits, plain torch
def _aux(s):
    """The auxiliary set without G = 0, |G|^2 / 2, v(G) and the positions of -G."""
    b = 2.0 * math.pi / s.lattice[0, 0]
    R = int(math.sqrt(2.0 * s.ecut_aux) / b) + 1
    x = np.arange(-R, R + 1)
    m = np.stack(np.meshgrid(x, x, x, indexing="ij"), -1).reshape(-1, 3)
    e = 0.5 * (m * m).sum(1) * b * b
    keep = (e <= s.ecut_aux) & (e > 0)
    m, e = m[keep], e[keep]
    key = {tuple(k): q for q, k in enumerate(m.tolist())}
    neg = np.array([key[(-k[0], -k[1], -k[2])] for k in m.tolist()])
    first = np.where(m[:, 0] != 0, m[:, 0], np.where(m[:, 1] != 0, m[:, 1], m[:, 2]))
    return m, e, 2.0 * math.pi / e, neg, np.nonzero(first > 0)[0]


def _flat(m, n):
    w = np.mod(m, n)
    return torch.from_numpy((w[..., 0] * n + w[..., 1]) * n + w[..., 2]).cuda()


def _codensities(s, tau, real, prim, m, neg):
    """Per Laplace point and block of primary G': M[slot, j, i, G] = <i| e^{-iGr} P_v(tau) e^{-iG'r} |j>
    e^{(e_j - mu) tau}, slot 0 for G' and, for general orbitals, slot 1 for -G'."""
    n, no = int(s.grid[0]), s.n_occ
    n3 = n ** 3
    co = torch.from_numpy(s.coeff).cuda()
    eps = torch.from_numpy(s.eps).cuda() - 0.5 * (s.eps[no - 1] + s.eps[no])
    pw = _flat(s.miller, n)
    cg = torch.zeros((no, n3), dtype=torch.complex128, device="cuda")
    cg[:, pw] = co[:no]
    u = torch.fft.ifftn(cg.reshape(no, n, n, n), dim=(1, 2, 3)) * n3
    ga = _flat(m, n)
    step = max(1, int(2.0e9 / (no * no * n3 * 16)))
    for k, t in enumerate(tau):
        d = torch.exp(-eps[no:] * t)
        P = (co[no:].T * d) @ co[no:].conj()
        f = torch.exp(eps[:no] * t)[:, None, None]
        for g0 in range(0, len(prim), step):
            gp = prim[g0:g0 + step]
            out = []
            for sign in ([1] if real else [1, -1]):
                idx = _flat(s.miller[None, :, :] + sign * m[gp][:, None, :], n)          # [g, q]
                S = cg[:, idx] * f                                                        # [j, g, q]
                W = (S.reshape(-1, S.shape[-1]) @ P.T).reshape(no, len(gp), -1)
                wg = torch.zeros((no, len(gp), n3), dtype=torch.complex128, device="cuda")
                wg[:, :, pw] = W
                wr = torch.fft.ifftn(wg.reshape(no, len(gp), n, n, n), dim=(2, 3, 4)) * n3
                M = torch.empty((len(gp), no, no, len(m)), dtype=torch.complex128, device="cuda")
                for i in range(no):
                    F = torch.fft.fftn(u[i].conj()[None, None] * wr, dim=(2, 3, 4)).reshape(no, len(gp), n3)
                    M[:, :, i, :] = F[:, :, ga].transpose(0, 1) / n3
                out.append(M)
            yield k, gp, out


def _pair_sums(s, tau, w, real, prim, levels=0):
    """Pair matrices e^d_ij, e^x_ij, and per nested sphere the energies."""
    m, e, v, neg, _ = _aux(s)
    vt = torch.from_numpy(v).cuda()
    ng = torch.from_numpy(neg).cuda()
    om, no = s.lattice[0, 0] ** 3, s.n_occ
    cuts = [s.ecut_aux / 1.05 ** q for q in range(max(1, levels))]
    masks = [e <= c if q else np.ones(len(e), bool) for q, c in enumerate(cuts)]
    ed = [torch.zeros((no, no), dtype=torch.float64, device="cuda") for _ in cuts]
    ex = [torch.zeros((no, no), dtype=torch.float64, device="cuda") for _ in cuts]
    for k, gp, out in _codensities(s, tau, real, prim, m, neg):
        A = out[0]
        B = A.conj() if real else out[1][..., ng]            # M_ij(-G; -G')
        dA, dB = A.diagonal(dim1=1, dim2=2), B.diagonal(dim1=1, dim2=2)      # [g, G, i]
        for q, mask in enumerate(masks):
            mt = torch.from_numpy(mask * v).cuda()
            c = torch.from_numpy(w[k] / om ** 2 * v[gp] * mask[gp]).cuda()
            X = torch.einsum("gjic,gijc->gij", A * mt, B)     # M_ij(G; G') M_ji(-G; -G')
            Y = torch.einsum("gci,gcj->gij", dA * mt[None, :, None], dB)
            ex[q] += torch.einsum("g,gij->ij", c, (X + X.transpose(1, 2)).real)
            ed[q] -= 2.0 * torch.einsum("g,gij->ij", c, (Y + Y.transpose(1, 2)).real)
    return ed, ex


def _cross(sa, sb, tau, w, real, prim):
    """Opposite-spin direct energy."""
    m, e, v, neg, _ = _aux(sa)
    vt, ng = torch.from_numpy(v).cuda(), torch.from_numpy(neg).cuda()
    om = sa.lattice[0, 0] ** 3
    total = 0.0
    keep = {}
    for x, s in enumerate((sa, sb)):
        for k, gp, out in _codensities(s, tau, real, prim, m, neg):
            A = out[0].diagonal(dim1=1, dim2=2)
            B = A.conj() if real else out[1][..., ng].diagonal(dim1=1, dim2=2)
            for r, g in enumerate(gp):
                keep[(x, k, int(g))] = (A[r].sum(1), B[r].sum(1))    # the sums over the orbitals
    for (x, k, g), (A, B) in keep.items():
        if x == 0:
            A1, B1 = keep[(1, k, g)]
            # <+G'| alpha, -G'| beta> and the other way round
            total -= w[k] / om ** 2 * v[g] * float((vt * (A * B1 + B * A1)).sum().real)
    return total


def _kpoint_pairs(s, tau, w):
    """Canonical sums over k1, k2, k3 and i, j, a, b with the exponential sum as denominator."""
    n, no, mesh, nk = int(s.grid[0]), s.n_occ, s.mesh, len(s.kappa)
    b = 2.0 * math.pi / s.lattice[0, 0]
    om = nk * s.lattice[0, 0] ** 3
    co = torch.from_numpy(s.coeff).cuda()
    eps = torch.from_numpy(s.eps).cuda()
    index = {tuple(k): q for q, k in enumerate(s.kappa.tolist())}
    pw = _flat(s.miller, n)
    cg = torch.zeros((nk, co.shape[1], n ** 3), dtype=torch.complex128, device="cuda")
    cg[:, :, pw] = co
    ur = torch.fft.ifftn(cg.reshape(nk, -1, n, n, n), dim=(2, 3, 4)) * n ** 3
    R = int(math.sqrt(2.0 * s.ecut_aux) / b) + 2
    x = np.arange(-R, R + 1)
    box = np.stack(np.meshgrid(x, x, x, indexing="ij"), -1).reshape(-1, 3)
    rho = {}
    for k in range(nk):
        for q in range(nk):
            d = s.kappa[q] - s.kappa[k]
            Q = (box + d / mesh) * b
            q2 = (Q * Q).sum(1)
            keep = (0.5 * q2 <= s.ecut_aux) & (q2 > 1e-20)
            g = box[keep]
            f = torch.fft.fftn(ur[k, :no, None].conj() * ur[q, None, no:], dim=(2, 3, 4)).reshape(no, -1, n ** 3) / n ** 3
            sup = g * mesh + d
            rho[(k, q)] = (f[:, :, _flat(g, n)], sup, torch.from_numpy(4.0 * math.pi / q2[keep]).cuda() / om,
                           {tuple(y): z for z, y in enumerate(sup.tolist())})
    out_d = torch.zeros((nk * no, nk * no), dtype=torch.float64, device="cuda")
    out_x = torch.zeros_like(out_d)
    for k1 in range(nk):
        for k2 in range(nk):
            for k3 in range(nk):
                k4 = index[tuple(np.mod(s.kappa[k1] + s.kappa[k2] - s.kappa[k3], mesh).tolist())]
                rA, sA, vA, _ = rho[(k1, k3)]
                rB, _, _, pB = rho[(k2, k4)]
                rC, sC, vC, _ = rho[(k1, k4)]
                rD, _, _, pD = rho[(k2, k3)]
                nb = torch.tensor([pB[tuple(y)] for y in (-sA).tolist()], device="cuda")
                nd = torch.tensor([pD[tuple(y)] for y in (-sC).tolist()], device="cuda")
                rBn, rDn = rB[:, :, nb], rD[:, :, nd]
                for i in range(no):
                    for j in range(no):
                        K = (rA[i] * vA) @ rBn[j].T
                        Kx = (rC[i] * vC) @ rDn[j].T
                        D = torch.zeros_like(K, dtype=torch.float64)
                        for t, c in zip(tau, w):
                            D -= c * torch.exp(t * (eps[k1, i] + eps[k2, j])) * torch.outer(
                                torch.exp(-t * eps[k3, no:]), torch.exp(-t * eps[k4, no:]))
                        out_d[k1 * no + i, k2 * no + j] += 2.0 * ((K.real ** 2 + K.imag ** 2) * D).sum() / nk
                        out_x[k1 * no + i, k2 * no + j] -= ((K * Kx.T.conj()).real * D).sum() / nk
    return out_d, out_x


def _seconds(case):
    """About what exact() takes: the complex transforms of every ordered pair, and the products."""
    if case["kind"] in ("kpoints", "dgemm"):
        return 1.0
    naux = _columns((case["r2"] + 1e-6) * 2.0 / 3.0)[0]
    npw = _columns(case["r2"])[0]
    prim = naux / 2 / case.get("parts", 1) * (1 if case["real"] else 2)
    occ = [case["n_occ"]] + ([case["n_occ_b"]] * 2 + [case["n_occ"]] if case["kind"] == "uhf" else [])
    return sum(case["n_tau"] * (prim * no * no * case["grid"] ** 3 * 1.3e-10 * 1.6 + 8 * npw * npw * (npw + prim * no) / 9e11)
               for no in occ)


def exact(case, seed):
    if case["kind"] == "dgemm":
        st = prepare(case, seed)
        return st["a"] @ st["b"].T
    if _seconds(case) > 18.0:
        return None
    s, tau, w = _inputs(case, seed)
    if case["kind"] == "kpoints":
        d, x = _kpoint_pairs(s[0], tau, w)
        return [np.array([float(d.sum()), float(x.sum())]), (d + x).cpu().numpy()]
    prim = _aux(s[0])[4]
    real = case["real"]
    if case["kind"] == "share":
        # the library walks the primary half column by column, (m1, m2) and then m3
        m = _aux(s[0])[0][prim]
        prim = prim[np.lexsort((m[:, 2], m[:, 1], m[:, 0]))]
        b, e = _range(case, len(prim))
        d, x = _pair_sums(s[0], tau, w, real, prim[b:e])
        return [np.array([float(d[0].sum()), float(x[0].sum())]), d[0].cpu().numpy(), x[0].cpu().numpy()]
    if case["kind"] == "uhf":
        es = []
        da = [_pair_sums(y, tau, w, real, prim) for y in s]
        ed = [float(q[0][0].sum()) for q in da]
        ex = [float(q[1][0].sum()) for q in da]
        c = _cross(s[0], s[1], tau, w, real, prim)
        es = [0.25 * ed[0] + 0.5 * ex[0], 0.25 * ed[1] + 0.5 * ex[1], c]
        return [np.array([0.25 * (ed[0] + ed[1]) + c, 0.5 * (ex[0] + ex[1])]), np.array(es)]
    d, x = _pair_sums(s[0], tau, w, real, prim, case.get("levels", 0))
    out = [np.array([float(d[0].sum()), float(x[0].sum())]), (d[0] + x[0]).cpu().numpy()]
    if case.get("levels"):
        out += [np.array([float(q.sum()) for q in d]), np.array([float(q.sum()) for q in x])]
    return out
