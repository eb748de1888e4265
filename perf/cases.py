"""The work that users of this library have it do, as cases that can be timed and checked.

Each case is a plain dict: a system (its atoms, basis and grid), the precision of the context and the
public call that is made on it.  `prepare` builds what a program holds before the call (a planned
context, the potential on the grid, a density matrix or a gradient on the stored pattern), `run` makes
the call, `exact` computes the same outputs in 64 bits with torch alone.

The systems are synthetic and seeded, in atomic units, and follow the sizes of this repository's
configurations: a water molecule with Gaussian shells, silicon clusters with 6s3p2d shells (25 functions
an atom), C/H/N/O clusters and molecules with 5s3p1d (heavy) and 2s1p (H) shells, with one f shell more
on heavy atoms where `f_shell` says so.  The atoms, and so the pattern of H, are the same for every
seed up to a rotation of the whole system; the seed fixes that rotation, the radial functions, the
grid's angular rotations, the batches, the potential and the matrices.
"""
import math
import types

import numpy as np
import torch

import paper_2208_12335_gb300 as fgi

ANG = 1.0 / 0.529177210903                     # Bohr per Angstrom
F64 = torch.float64
SPECIES = {"O_water": 8.0, "H_water": 1.0, "Si": 14.0, "H": 1.0, "C": 6.0, "N": 7.0, "O": 8.0}
# shells (l) of each species and, per l, the ranges of their leading exponents
SI_ALPHA = {0: [(4.0, 8.0), (1.5, 3.0), (0.6, 1.2), (0.3, 0.6), (0.15, 0.3), (0.08, 0.15)],
            1: [(1.5, 3.0), (0.4, 1.0), (0.12, 0.3)], 2: [(0.5, 1.2), (0.15, 0.4)]}
HEAVY_ALPHA = {0: [(4.0, 8.0), (1.5, 3.0), (0.6, 1.2), (0.25, 0.5), (0.1, 0.2)],
               1: [(1.0, 2.0), (0.3, 0.7), (0.12, 0.25)], 2: [(0.4, 1.0)], 3: [(0.5, 1.2)]}
H_ALPHA = {0: [(0.8, 1.6), (0.15, 0.35)], 1: [(0.3, 0.8)]}


def _case(name, call, system, atoms, n_rad, n_ang, p_max, p_min, precision="split_bf16", molecules=1,
          uneven=False, mixed_sign=False, f_shell=False, l_max=4):
    return dict(name=name, call=call, system=system, atoms=atoms, molecules=molecules, n_rad=n_rad, n_ang=n_ang,
                p_max=p_max, p_min=p_min, uneven=uneven, precision=precision, mixed_sign=mixed_sign,
                f_shell=f_shell, l_max=l_max)


def listed():
    return [
        # one iteration of a self-consistency loop on a very small molecule (density, its Hartree potential,
        # H): all latency and launches
        _case("water_scf", "scf", "water", 3, 40, 110, 200, 50),
        # the FP64 context that a program checks the fast path with, on one molecule
        _case("molecule20_fp64", "step", "chno", 20, 36, 146, 300, 50, precision="fp64"),
        # differentiable H of one molecule, forward and backward, with a potential that changes sign
        # (v_ext + v_H + v_xc does)
        _case("molecule30_grad", "grad", "chno", 30, 45, 194, 300, 50, mixed_sign=True),
        # the silicon cluster, each call by itself: H of an effective potential of one sign,
        _case("si64_h", "h", "si", 64, 60, 302, 300, 100),
        # the density of an occupied-orbital matrix with the electron count,
        _case("si64_density", "density", "si", 64, 60, 302, 300, 100),
        # the gradients with respect to the potential and the atoms (forces, inverse problems),
        _case("si64_adjoint", "adjoint", "si", 64, 60, 302, 300, 100),
        # its Hartree potential,
        _case("si64_hartree", "hartree", "si", 64, 60, 302, 300, 100),
        # and H and density at plain BF16 (early iterations, screening)
        _case("si64_bf16", "step", "si", 64, 60, 302, 300, 100, precision="bf16"),
        # a cluster with f shells, odd grid sizes, small uneven batches and a potential of both signs
        _case("cluster75_f_h", "h", "chno", 75, 61, 387, 233, 31, uneven=True, mixed_sign=True, f_shell=True),
        # many independent small molecules in one plan (screening, data sets)
        _case("molecules64_step", "step", "chno", 22, 45, 194, 300, 50, molecules=64),
        # Hartree potential at high order on a larger cluster: every point sees every atom
        _case("cluster250_hartree", "hartree", "chno", 250, 70, 434, 400, 50, uneven=True, l_max=6),
        # the largest: H and density of the 1000-atom cluster with uneven batches
        _case("cluster1000_step", "step", "chno", 1000, 70, 590, 400, 50, uneven=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of these ranges: any call on any system, sizes from one small molecule to several
    hundred atoms (FP64 contexts: molecules, as they are used for)."""
    precision = rng.choice(["split_bf16"] * 5 + ["bf16", "fp64"])
    call = rng.choice(["h", "density", "step", "adjoint", "grad", "hartree", "scf"])
    system = rng.choice(["chno", "chno", "chno", "si", "si", "many"])
    molecules = 1
    if precision == "fp64":
        system, atoms = "chno", _log_int(rng, 3, 16 if call in ("grad", "adjoint") else 24)
    elif system == "many":
        system, atoms, molecules = "chno", rng.randint(5, 30), _log_int(rng, 2, 64)
    elif system == "si":
        atoms = _log_int(rng, 5, 64)
    else:
        atoms = _log_int(rng, 4, 300)
    p_max = _log_int(rng, 100, 1000)
    return dict(call=call, system=system, atoms=atoms, molecules=molecules, n_rad=rng.randint(30, 60),
                n_ang=_log_int(rng, 110, 434), p_max=p_max, p_min=min(rng.randint(30, 100), p_max // 3),
                uneven=rng.random() < 0.5, precision=precision, mixed_sign=rng.random() < 0.4,
                f_shell=system == "chno" and rng.random() < 0.25, l_max=rng.choice([4, 4, 6, 2]))


# ------------------------------------------------------------------ systems
def _geometry(case):
    """Per molecule (species names, positions in Bohr); the same for every seed."""
    if case["system"] == "water":
        r, half = 0.96 * ANG, math.radians(104.5) / 2.0
        xyz = np.array([[0.0, 0.0, 0.0], [r * math.sin(half), 0.0, r * math.cos(half)],
                        [-r * math.sin(half), 0.0, r * math.cos(half)]])
        return [(["O_water", "H_water", "H_water"], xyz)]
    rng = np.random.default_rng([7, case["atoms"], case["molecules"]])
    if case["system"] == "si":
        cell = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0],
                         [.25, .25, .25], [.25, .75, .75], [.75, .25, .75], [.75, .75, .25]])
        k = math.ceil((case["atoms"] / 8) ** (1 / 3))
        at = np.array([[i, j, m] for i in range(k) for j in range(k) for m in range(k)], dtype=np.float64)
        pos = (at[:, None, :] + cell[None]).reshape(-1, 3) * 5.43
        pos -= pos.mean(axis=0)
        near = np.argsort((pos ** 2).sum(axis=1), kind="stable")[:case["atoms"]]
        pos = pos[np.sort(near)]
        return [(["Si"] * len(pos), (pos + rng.normal(0.0, 0.05, pos.shape)) * ANG)]
    out = []
    for _ in range(case["molecules"]):
        # random packing in a sphere at 0.1 atoms per cubic Angstrom, no two atoms closer than 1 Angstrom
        n = case["atoms"] if case["molecules"] == 1 else max(3, case["atoms"] + int(rng.integers(-case["atoms"] // 2, case["atoms"] // 2 + 1)))
        radius = (3.0 * n / (0.4 * math.pi)) ** (1.0 / 3.0)
        pos, tries = np.zeros((n, 3)), 0
        k = 0
        while k < n:
            tries += 1
            if tries % (200 * n) == 0:
                radius *= 1.05
            p = rng.uniform(-radius, radius, 3)
            if p @ p > radius * radius or (k and ((pos[:k] - p) ** 2).sum(axis=1).min() < 1.0):
                continue
            pos[k] = p
            k += 1
        out.append(([("H" if rng.uniform() < 0.5 else "CNO"[int(rng.integers(0, 3))]) for _ in range(n)], pos * ANG))
    return out


def _shells(case, species, rng):
    """Radial functions of a species: (l, exponents, coefficients, cutoff, start of the switch, intervals)."""
    if species == "O_water":
        return [(l, [a * rng.uniform(0.9, 1.1)], [1.0], 5.0 * ANG, None, 4000) for l, a in ((0, 10.0), (0, 0.8), (1, 0.6))]
    if species == "H_water":
        return [(0, [0.5 * rng.uniform(0.9, 1.1)], [1.0], 5.0 * ANG, None, 4000)]
    table, cut, n = (SI_ALPHA, 6.0 * ANG, 2000) if species == "Si" else (H_ALPHA if species == "H" else HEAVY_ALPHA, 5.0 * ANG, 1500)
    out = []
    for l, ranges in table.items():
        if l == 3 and not case["f_shell"]:
            continue
        for lo, hi in ranges:
            a = math.exp(rng.uniform(math.log(lo), math.log(hi)))
            more = int(rng.integers(1, 3))
            out.append((l, [a] + [a * rng.uniform(1.5, 3.0) for _ in range(more)],
                        [1.0] + [rng.uniform(-0.5, 0.5) for _ in range(more)], cut, cut - ANG, n))
    return out


def _spline(shell):
    """(h, coef [n][4]): u(r) = r R(r), normalised, as a cubic Hermite spline on r_k = k h."""
    l, alphas, coefs, cut, on, n = shell

    def u_du(r):
        e = [c * np.exp(-a * r * r) for a, c in zip(alphas, coefs)]
        g, dg = sum(e), sum(-2.0 * a * r * x for a, x in zip(alphas, e))
        u = r ** (l + 1) * g
        du = (l + 1) * r ** l * g + r ** (l + 1) * dg
        if on is not None:
            x = np.clip((r - on) / (cut - on), 0.0, 1.0)
            dsw = np.where(r > on, 6.0 * (1.0 - x * x) ** 2 * -x / (cut - on), 0.0)
            du, u = du * (1.0 - x * x) ** 3 + u * dsw, u * (1.0 - x * x) ** 3
        return u, du

    fine = (np.arange(40000) + 0.5) * (cut / 40000)
    norm = 1.0 / math.sqrt(float((u_du(fine)[0] ** 2).sum()) * cut / 40000)
    h = cut / n
    u, du = (norm * x for x in u_du(np.arange(n + 1) * h))
    u[-1] = du[-1] = 0.0
    d0, d1, step = h * du[:-1], h * du[1:], u[1:] - u[:-1]
    return h, np.stack([u[:-1], d0, 3.0 * step - 2.0 * d0 - d1, d0 + d1 - 2.0 * step], axis=1)


def _rotations(gen, *shape):
    """Uniform random rotation matrices [*shape][3][3] from random unit quaternions."""
    q = torch.randn(*shape, 4, dtype=F64, device="cuda", generator=gen)
    a, b, c, d = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - a * d), 2 * (b * d + a * c),
                        2 * (b * c + a * d), 1 - 2 * (b * b + d * d), 2 * (c * d - a * b),
                        2 * (b * d - a * c), 2 * (c * d + a * b), 1 - 2 * (b * b + c * c)], dim=-1).reshape(*shape, 3, 3)


def _grid(case, R, Z, cut, n_ang, gen):
    """Points, weights, potential, owner and shell of one molecule's grid (GPU): atom-centred shells
    r_k = r_min q^k, golden-angle spheres, Becke weights over the owner and its nearest atoms; the 4 % of
    the points with the least weight are dropped, as far outside their cell."""
    n_at, n_rad = len(R), case["n_rad"]
    k = torch.arange(n_rad, dtype=F64, device="cuda")
    lnq = torch.log(cut / 1e-3) / (n_rad - 1)                                       # per atom
    r = 1e-3 * torch.exp(lnq[:, None] * k)                                          # [n_at][n_rad]
    j = torch.arange(n_ang, dtype=F64, device="cuda")
    z = 1.0 - (2.0 * j + 1.0) / n_ang
    rho, th = torch.sqrt(1.0 - z * z), j * (math.pi * (3.0 - math.sqrt(5.0)))
    sphere = torch.stack([rho * torch.cos(th), rho * torch.sin(th), z], dim=1)
    rot = _rotations(gen, n_at, n_rad)
    pts = (R[:, None, None, :] + r[:, :, None, None] * torch.einsum("jc,akdc->akjd", sphere, rot)).reshape(n_at, -1, 3)
    w = (r ** 3 * lnq[:, None] * (4.0 * math.pi / n_ang)).repeat_interleave(n_ang, dim=1)
    v = torch.empty_like(w)
    near = torch.cdist(R, R).argsort(dim=1)[:, :16]                                 # the owner first
    kk = near.shape[1]
    eye = torch.eye(kk, dtype=torch.bool, device="cuda")
    step = max(1, int(2e6) // (n_rad * n_ang))
    for a0 in range(0, n_at, step):
        N = near[a0:a0 + step]
        A = R[N]                                                                    # [a][kk][3]
        d = torch.cdist(pts[a0:a0 + step], A, compute_mode="donot_use_mm_for_euclid_dist")
        f = (torch.erf(d) - torch.erf(0.5 * d)) / d.clamp_min(1e-12)
        v[a0:a0 + step] = -(f * Z[N][:, None, :]).sum(-1)
        if kk > 1:
            rab = torch.cdist(A, A, compute_mode="donot_use_mm_for_euclid_dist").masked_fill(eye, 1.0)
            P = torch.ones_like(d)
            for c in range(kk):
                m = (d - d[..., c:c + 1]) / rab[:, c][:, None, :]
                for _ in range(3):
                    m = m * (1.5 - 0.5 * m * m)
                P *= (0.5 * (1.0 - m)).masked_fill(eye[c], 1.0)
            w[a0:a0 + step] *= P[..., 0] / P.sum(-1)
    if case["mixed_sign"]:
        v += 0.2
    owner = torch.arange(n_at, device="cuda").repeat_interleave(n_rad * n_ang)
    shell = torch.arange(n_rad, device="cuda").repeat_interleave(n_ang).repeat(n_at)
    pts, w, v = pts.reshape(-1, 3), w.reshape(-1), v.reshape(-1)
    if n_at > 1:
        keep = w.topk(len(w) - len(w) // 25, sorted=False).indices.sort().values
        pts, w, v, owner, shell = pts[keep], w[keep], v[keep], owner[keep], shell[keep]
    return pts, w, v, owner, shell, lnq


def _batches(pts, first, case, gen):
    """Order of the points and batch offsets: recursive bisection (x, y, z in turn) of each molecule's
    points, at the median or, for uneven batches, at a random quantile, until p_max points are left."""
    n = len(pts)
    order = torch.arange(n, device="cuda")
    off = torch.tensor(first, device="cuda")
    axis = 0
    while True:
        size = off[1:] - off[:-1]
        big = size > case["p_max"]
        if not bool(big.any()):
            return order, off, size
        seg = torch.arange(len(size), device="cuda").repeat_interleave(size)
        by = pts[order, axis].argsort()
        by = by[seg[by].argsort(stable=True)]
        order = order[by]
        q = torch.rand(len(size), dtype=F64, device="cuda", generator=gen) * 0.6 + 0.2 if case["uneven"] else 0.5
        cut = torch.minimum(torch.clamp_min((q * size).round().long(), case["p_min"]), size - case["p_min"])
        off = torch.cat([off, (off[:-1] + cut)[big]]).sort().values
        axis = (axis + 1) % 3


def _problem(case, seed):
    """The system of a case for one seed: basis, atoms, grid, potential; arrays on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng([11, seed])
    mols = _geometry(case)
    names = [s for s in SPECIES if any(s in m[0] for m in mols)]
    radials, species, rid = [], [], 0
    for s in names:
        ids = []
        for shell in _shells(case, s, rng):
            h, coef = _spline(shell)
            radials.append(types.SimpleNamespace(l=shell[0], h=h, coef=coef, cut=shell[3]))
            ids.append(rid)
            rid += 1
        species.append(types.SimpleNamespace(Z=SPECIES[s], radial_ids=ids, cut=max(radials[i].cut for i in ids),
                                             n_fn=sum(2 * radials[i].l + 1 for i in ids)))
    P = types.SimpleNamespace(radials=radials, species=species)
    atom_off, parts, first, rg = [0], [], [0], []
    for m, (elements, xyz) in enumerate(mols):
        sp = np.array([names.index(e) for e in elements])
        R = torch.from_numpy(xyz).cuda() @ _rotations(gen, 1)[0].T
        Z = torch.tensor([species[k].Z for k in sp], dtype=F64, device="cuda")
        cut = torch.tensor([species[k].cut for k in sp], dtype=F64, device="cuda")
        n_ang = case["n_ang"] if case["molecules"] == 1 else max(50, case["n_ang"] - 12 * (m % 8))
        pts, w, v, owner, shell, lnq = _grid(case, R, Z, cut, n_ang, gen)
        parts.append((sp, R, pts, w, v, owner + atom_off[-1], shell))
        rg.append(torch.stack([torch.full_like(lnq, 1e-3), lnq, torch.full_like(lnq, case["n_rad"])], dim=1))
        atom_off.append(atom_off[-1] + len(sp))
        first.append(first[-1] + len(w))
    cat = lambda i: torch.cat([p[i] for p in parts])  # noqa: E731
    P.atom_off, P.sp, P.R, P.rgrid = np.array(atom_off), np.concatenate([p[0] for p in parts]), cat(1), torch.cat(rg)
    order, off, size = _batches(cat(2), first, case, gen)
    P.r, P.wt, P.v, P.own, P.sh = (cat(i)[order] for i in (2, 3, 4, 5, 6))
    P.off = off.cpu().numpy()
    P.first = first
    P.bsys = (np.searchsorted(np.array(first), P.off[:-1], side="right") - 1).astype(np.int32)
    P.nfn = np.array([s.n_fn for s in species])[P.sp]
    P.fn0 = np.concatenate([[0], np.cumsum(P.nfn)])
    return P


def _stored(P, s):
    """(row, column) function of every stored value of molecule s, in order: the upper triangle by rows
    over the atom pairs closer than the sum of their cutoffs."""
    a0, a1 = P.atom_off[s], P.atom_off[s + 1]
    cut = torch.tensor([P.species[k].cut for k in P.sp[a0:a1]], dtype=F64, device="cuda")
    d = torch.cdist(P.R[a0:a1], P.R[a0:a1], compute_mode="donot_use_mm_for_euclid_dist")
    pair = d < cut[:, None] + cut[None, :]
    at = torch.from_numpy(P.nfn[a0:a1]).cuda()
    at = torch.arange(len(at), device="cuda").repeat_interleave(at)
    rows, cols = [], []
    for i0 in range(0, len(at), 2048):                                              # rows in pieces
        i = torch.arange(i0, min(i0 + 2048, len(at)), device="cuda")
        m = pair[at[i]][:, at] & (torch.arange(len(at), device="cuda")[None, :] >= i[:, None])
        r, c = m.nonzero(as_tuple=True)
        rows.append(r + i0)
        cols.append(c)
    return torch.cat(rows), torch.cat(cols)


def _density_values(P, seed):
    """Stored values of D = 2 C C^T, C orthonormal columns (0.28 of the functions; at most 512)."""
    gen = torch.Generator(device="cuda").manual_seed(seed + (1 << 40))
    out = []
    for s in range(len(P.atom_off) - 1):
        n = int(P.fn0[P.atom_off[s + 1]] - P.fn0[P.atom_off[s]])
        C = torch.randn(n, max(1, min(512, round(0.28 * n))), dtype=F64, device="cuda", generator=gen)
        C = torch.linalg.solve_triangular(torch.linalg.cholesky(C.T @ C, upper=True), C, upper=True, left=False)
        r, c = _stored(P, s)
        out.append(2.0 * (C @ C.T)[r, c])
    return torch.cat(out)


def _gradient_values(P, seed):
    """A loss's gradient with respect to the stored values of H."""
    gen = torch.Generator(device="cuda").manual_seed(seed + (1 << 41))
    n = sum(len(_stored(P, s)[0]) for s in range(len(P.atom_off) - 1))
    return torch.randn(n, dtype=F64, device="cuda", generator=gen)


# ------------------------------------------------------- what a program does
def prepare(case, seed):
    P = _problem(case, seed)
    host = types.SimpleNamespace(
        radials=P.radials, species=P.species, atom_off=P.atom_off, atom_species=P.sp, atom_xyz=P.R.cpu().numpy(),
        pts=P.r.cpu().numpy(), w=P.wt.cpu().numpy(), batch_off=P.off, batch_sys=P.bsys,
        owner=P.own.int().cpu().numpy(), shell=P.sh.int().cpu().numpy(), atom_rgrid=P.rgrid.cpu().numpy())
    s = types.SimpleNamespace(call=case["call"], l_max=case["l_max"], v=P.v)
    s.ctx = fgi.Context(0).load(host, case["precision"])
    if s.call in ("density", "step", "scf"):
        s.d = _density_values(P, seed)
    if s.call in ("adjoint", "grad"):
        s.g = _gradient_values(P, seed)
    if s.call == "grad":
        s.R = P.R
    if s.call == "hartree":                                                         # a smooth charge density
        s.n = _model_density(P)
    return s


def run(s):
    ctx = s.ctx
    if s.call == "h":
        return ctx.integrate_h(s.v)
    if s.call == "density":
        return ctx.density(s.d)
    if s.call == "step":
        n, traces = ctx.density(s.d)
        return ctx.integrate_h(s.v), n, traces
    if s.call == "adjoint":
        return ctx.adjoint(s.g, s.v)
    if s.call == "hartree":
        return ctx.hartree(s.n, s.l_max)
    if s.call == "scf":
        n, traces = ctx.density(s.d)
        vh = ctx.hartree(n, s.l_max)
        return ctx.integrate_h(s.v + vh), n, traces, vh
    v, R = s.v.clone().requires_grad_(True), s.R.clone().requires_grad_(True)       # grad
    h = fgi.integrate(ctx, v, R)
    (h * s.g).sum().backward()
    return h.detach(), v.grad, R.grad


def work(case):
    """Floating-point operations of the functions that are non-zero at each point (30 a value, n (n+1) a
    contraction with a symmetric matrix, 2 n^2 with the gradient's), and every input and output once."""
    P = _problem(case, 1)
    n_pts = len(P.wt)
    stride = max(1, n_pts // 200000)
    n1 = n2 = pairs = nnz = 0.0
    for s in range(len(P.atom_off) - 1):
        a0, a1 = P.atom_off[s], P.atom_off[s + 1]
        cut = torch.tensor([P.species[k].cut for k in P.sp[a0:a1]], dtype=F64, device="cuda")
        nfn = torch.from_numpy(P.nfn[a0:a1]).cuda().double()
        for r in P.r[P.first[s]:P.first[s + 1]:stride].split(20000):
            n = ((torch.cdist(r, P.R[a0:a1]) < cut) * nfn).sum(1)
            n1 += float(n.sum()) * stride
            n2 += float((n * (n + 1)).sum()) * stride
        pairs += float(P.first[s + 1] - P.first[s]) * float(a1 - a0)
        nnz += len(_stored(P, s)[0])
    terms = (case["l_max"] + 1) ** 2
    h = (n2 + 30.0 * n1, 8.0 * nnz + 40.0 * n_pts)
    density = (n2 + 32.0 * n1, 8.0 * nnz + 40.0 * n_pts)
    adjoint = (2.0 * n2 + 70.0 * n1, 8.0 * nnz + 48.0 * n_pts)
    hartree = ((20.0 + 4.0 * terms) * pairs + 6.0 * terms * n_pts, 56.0 * n_pts)
    parts = {"h": [h], "density": [density], "step": [h, density], "adjoint": [adjoint], "hartree": [hartree],
             "scf": [density, hartree, h], "grad": [h, adjoint]}[case["call"]]
    return {"flops": sum(p[0] for p in parts), "bytes": sum(p[1] for p in parts)}


# --------------------------------------------------------- the same in 64 bits
def _model_density(P):
    """A superposition of Gaussian charges, one on each atom, of the atom's own width and size."""
    n = torch.empty_like(P.wt)
    for s in range(len(P.atom_off) - 1):
        a0, a1 = P.atom_off[s], P.atom_off[s + 1]
        Z = torch.tensor([P.species[k].Z for k in P.sp[a0:a1]], dtype=F64, device="cuda")
        a = 0.4 + 0.1 * torch.sqrt(Z)
        for p0 in range(P.first[s], P.first[s + 1], 500000):
            p1 = min(p0 + 500000, P.first[s + 1])
            own = P.own[p0:p1] - a0
            near = torch.cdist(P.R[a0:a1], P.R[a0:a1]).argsort(dim=1)[:, :16][own]
            d2 = (P.r[p0:p1, None, :] - P.R[a0:a1][near]).square().sum(-1)
            n[p0:p1] = (Z[near] * (a[near] / math.pi) ** 1.5 * torch.exp(-a[near] * d2)).sum(1)
    return n


def _angular(l, x, y, z):
    """Real spherical harmonics of a unit vector, unit-normalised, m = -l .. l, no Condon-Shortley phase."""
    if l == 0:
        return [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if l == 1:
        c = math.sqrt(3 / (4 * math.pi))
        return [c * y, c * z, c * x]
    if l == 2:
        c = 0.5 * math.sqrt(15 / math.pi)
        return [c * x * y, c * y * z, 0.25 * math.sqrt(5 / math.pi) * (2 * z * z - x * x - y * y), c * x * z,
                0.5 * c * (x * x - y * y)]
    a, b = 0.25 * math.sqrt(35 / (2 * math.pi)), 0.25 * math.sqrt(21 / (2 * math.pi))
    c, q = 0.5 * math.sqrt(105 / math.pi), 4 * z * z - x * x - y * y
    return [a * y * (3 * x * x - y * y), c * x * y * z, b * y * q,
            0.25 * math.sqrt(7 / math.pi) * z * (2 * z * z - 3 * x * x - 3 * y * y), b * x * q,
            0.5 * c * z * (x * x - y * y), a * x * (x * x - 3 * y * y)]


def _phi(P, r, atoms, R):
    """phi [points][functions of the listed atoms] in 64 bits; differentiable in R (their positions)."""
    delta = r[:, None, :] - R[None]
    d = delta.square().sum(-1).clamp_min(1e-24).sqrt()
    x, y, z = (delta / d[..., None]).unbind(-1)
    cols, place = [], []
    first = np.concatenate([[0], np.cumsum(P.nfn[atoms])])
    for k, sp in enumerate(P.species):
        mine = np.nonzero(P.sp[atoms] == k)[0]
        if not len(mine):
            continue
        dk, xk, yk, zk = d[:, mine], x[:, mine], y[:, mine], z[:, mine]
        f = 0
        for i in sp.radial_ids:
            rad = P.radials[i]
            c = torch.from_numpy(rad.coef).cuda()
            q = dk / rad.h
            t0 = q.detach().floor().long().clamp_max(len(c) - 1)
            t, c = q - t0, c[t0]
            u = c[..., 0] + t * (c[..., 1] + t * (c[..., 2] + t * c[..., 3]))
            u = torch.where(dk < rad.h * len(rad.coef), u / dk, torch.zeros_like(u))
            for Y in _angular(rad.l, xk, yk, zk):
                cols.append(u * Y)
                place.append(first[mine] + f)
                f += 1
    inv = torch.from_numpy(np.argsort(np.concatenate(place), kind="stable")).cuda()
    return torch.cat(cols, dim=1)[:, inv]


def _pieces(P):
    """Runs of neighbouring batches of one molecule: (molecule, first point, last, atoms within reach)."""
    cut = torch.tensor([s.cut for s in P.species], dtype=F64, device="cuda")[torch.from_numpy(P.sp).cuda()]
    b = 0
    while b < len(P.bsys):
        s, e = P.bsys[b], b + 1
        while e < len(P.bsys) and P.bsys[e] == s and P.off[e + 1] - P.off[b] <= 6000:
            e += 1
        p0, p1 = int(P.off[b]), int(P.off[e])
        a0, a1 = P.atom_off[s], P.atom_off[s + 1]
        on = ((torch.cdist(P.r[p0:p1], P.R[a0:a1]) < cut[a0:a1]).any(0)).cpu().numpy()
        if on.any():
            yield s, p0, p1, a0 + np.nonzero(on)[0]
        b = e


def _functions(P, s, atoms):
    f0 = P.fn0[P.atom_off[s]]
    return torch.from_numpy(np.concatenate([np.arange(P.fn0[a], P.fn0[a + 1]) for a in atoms]) - f0).cuda()


def _exact_h(P, v):
    n = [int(P.fn0[P.atom_off[s + 1]] - P.fn0[P.atom_off[s]]) for s in range(len(P.atom_off) - 1)]
    H = [torch.zeros(m, m, dtype=F64, device="cuda") for m in n]
    for s, p0, p1, atoms in _pieces(P):
        phi, f = _phi(P, P.r[p0:p1], atoms, P.R[atoms]), _functions(P, s, atoms)
        H[s][f[:, None], f[None, :]] += (phi * (P.wt[p0:p1] * v[p0:p1])[:, None]).T @ phi
    return torch.cat([H[s][_stored(P, s)] for s in range(len(n))])


def _matrices(P, values, offdiag):
    out, k = [], 0
    for s in range(len(P.atom_off) - 1):
        n = int(P.fn0[P.atom_off[s + 1]] - P.fn0[P.atom_off[s]])
        r, c = _stored(P, s)
        x = values[k:k + len(r)] * torch.where(r == c, 1.0, offdiag)
        M = torch.zeros(n, n, dtype=F64, device="cuda")
        M[r, c] = x
        M[c, r] = x
        out.append(M)
        k += len(r)
    return out


def _exact_density(P, values):
    D, n = _matrices(P, values, 1.0), torch.zeros_like(P.wt)
    for s, p0, p1, atoms in _pieces(P):
        phi, f = _phi(P, P.r[p0:p1], atoms, P.R[atoms]), _functions(P, s, atoms)
        n[p0:p1] = ((phi @ D[s][f[:, None], f[None, :]]) * phi).sum(1)
    return n, torch.stack([(P.wt * n)[a:b].sum() for a, b in zip(P.first[:-1], P.first[1:])])


def _exact_adjoint(P, g, v):
    G, dv, dR = _matrices(P, g, 0.5), torch.zeros_like(P.wt), torch.zeros_like(P.R)
    for s, p0, p1, atoms in _pieces(P):
        R = P.R[atoms].clone().requires_grad_(True)
        phi, f = _phi(P, P.r[p0:p1], atoms, R), _functions(P, s, atoms)
        E = phi.detach() @ G[s][f[:, None], f[None, :]]
        dv[p0:p1] = P.wt[p0:p1] * (E * phi.detach()).sum(1)
        (2.0 * (P.wt[p0:p1] * v[p0:p1])[:, None] * E * phi).sum().backward()
        dR[atoms] += R.grad
    return dv, dR


def _legendre(l_max, x, y, z):
    """Real spherical harmonics up to l_max of unit vectors by the Legendre recurrences, [l*l + l + m]."""
    out = [None] * (l_max + 1) ** 2
    c, s, pmm = torch.ones_like(x), torch.zeros_like(x), 1.0
    for m in range(l_max + 1):
        if m:
            c, s, pmm = c * x - s * y, c * y + s * x, pmm * (2 * m - 1)
        p2, p1 = None, torch.full_like(x, pmm)
        for l in range(m, l_max + 1):
            if l == m + 1:
                p2, p1 = p1, (2 * m + 1) * z * p1
            elif l > m:
                p2, p1 = p1, ((2 * l - 1) * z * p1 - (l + m - 1) * p2) / (l - m)
            k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m) * (2 if m else 1))
            out[l * l + l + m] = k * p1 * c
            if m:
                out[l * l + l - m] = k * p1 * s
    return out


def _exact_hartree(P, n, l_max):
    """Multipoles on each atom's shells, the radial Poisson equation in ln r (cubic interval rule), and
    4-point interpolation between the shells, the exterior field beyond them, V(r_0) (d/r_0)^l inside."""
    N, L, n_at = int(P.rgrid[0, 2]), (l_max + 1) ** 2, len(P.R)
    lnq = P.rgrid[:, 1]
    r = P.rgrid[:, :1] * torch.exp(lnq[:, None] * torch.arange(N, dtype=F64, device="cuda"))
    rho = torch.zeros(n_at * N, L, dtype=F64, device="cuda")
    for p0 in range(0, len(n), 2000000):
        q = slice(p0, p0 + 2000000)
        own, k = P.own[q], P.sh[q]
        delta = P.r[q] - P.R[own]
        delta = delta / delta.norm(dim=1, keepdim=True)
        x = P.wt[q] / (r[own, k] ** 3 * lnq[own]) * n[q]
        rho.index_add_(0, own * N + k, x[:, None] * torch.stack(_legendre(l_max, *delta.unbind(1)), dim=1))
    rho = rho.reshape(n_at, N, L)
    l = torch.tensor([k for k in range(l_max + 1) for _ in range(2 * k + 1)], dtype=F64, device="cuda")
    h, rk = lnq[:, None, None], r[:, :, None]

    def intervals(f):
        mid = h * (-f[:, :-3] + 13 * f[:, 1:-2] + 13 * f[:, 2:-1] - f[:, 3:]) / 24
        lo = h * (9 * f[:, :1] + 19 * f[:, 1:2] - 5 * f[:, 2:3] + f[:, 3:4]) / 24
        hi = h * (f[:, -4:-3] - 5 * f[:, -3:-2] + 19 * f[:, -2:-1] + 9 * f[:, -1:]) / 24
        return torch.cat([lo, mid, hi], dim=1)

    f, g = rho * rk ** (l + 3), rho * rk ** (2 - l)
    zero = torch.zeros_like(f[:, :1])
    inner = torch.cat([zero, intervals(f).cumsum(1)], dim=1) + f[:, :1] / (l + 3)
    outer = torch.cat([intervals(g).flip(1).cumsum(1).flip(1), zero], dim=1)
    pref = 4 * math.pi / (2 * l + 1)
    V = pref * (rk ** -(l + 1) * inner + rk ** l * outer)                           # [n_at][N][L]
    Q = pref * inner[:, -1]
    vh = torch.zeros_like(n)
    for s in range(len(P.atom_off) - 1):
        for a in range(P.atom_off[s], P.atom_off[s + 1]):
            for p0 in range(P.first[s], P.first[s + 1], 8000000):
                p1 = min(p0 + 8000000, P.first[s + 1])
                delta = P.r[p0:p1] - P.R[a]
                d = delta.norm(dim=1)
                Y = _legendre(l_max, *(delta / d.clamp_min(1e-300)[:, None]).unbind(1))
                out = torch.zeros_like(d)
                rl = 1.0 / d
                for k in range(l_max + 1):
                    out += rl * sum(Q[a, i] * Y[i] for i in range(k * k, (k + 1) ** 2))
                    rl = rl / d
                near = (d < r[a, -1]).nonzero()[:, 0]
                dn, Yn = d[near], torch.stack([y[near] for y in Y], dim=1)
                x = torch.log(dn / r[a, 0]) / lnq[a]
                i0 = (x.floor().long() - 1).clamp(0, N - 4)
                t = x - i0
                val = sum(wt[:, None] * V[a, i0 + j] for j, wt in enumerate(
                    (-(t - 1) * (t - 2) * (t - 3) / 6, t * (t - 2) * (t - 3) / 2, -t * (t - 1) * (t - 3) / 2,
                     t * (t - 1) * (t - 2) / 6)))
                val = torch.where((dn <= r[a, 0])[:, None], V[a, 0] * (dn / r[a, 0])[:, None] ** l, val)
                out[near] = (val * Yn).sum(1)
                vh[p0:p1] += out
    return vh


def exact(case, seed):
    if case["atoms"] > 500:
        return None                                                                 # minutes in 64 bits
    P = _problem(case, seed)
    call, v = case["call"], P.v
    largest = max(int(P.fn0[b] - P.fn0[a]) for a, b in zip(P.atom_off[:-1], P.atom_off[1:]))
    if call != "hartree" and len(P.wt) * min(largest, 2000) ** 2 > 3.2e12:
        return None
    if call == "h":
        return _exact_h(P, v)
    if call == "density":
        return _exact_density(P, _density_values(P, seed))
    if call == "step":
        n, traces = _exact_density(P, _density_values(P, seed))
        return _exact_h(P, v), n, traces
    if call == "adjoint":
        return _exact_adjoint(P, _gradient_values(P, seed), v)
    if call == "hartree":
        return _exact_hartree(P, _model_density(P), case["l_max"])
    if call == "scf":
        n, traces = _exact_density(P, _density_values(P, seed))
        vh = _exact_hartree(P, n, case["l_max"])
        return _exact_h(P, v + vh), n, traces, vh
    return (_exact_h(P, v),) + _exact_adjoint(P, _gradient_values(P, seed), v)
