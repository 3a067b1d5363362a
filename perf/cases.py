"""The work whose speed is watched: calls of the package as an MD or SCF program makes them.

Every case is one pass of one kind of call sequence on one seeded QM/MM system:

  step    one MD step: qmmm_set_positions, qmmm_vpot, qmmm_energy, qmmm_forces (forward and backward)
  grad    the same step through the autograd Function, forward and backward, dE/dgamma included
  scf     one SCF iteration at a fixed geometry: multipoles, E_II and the Fock term of a new density,
          the total energy and dE/dgamma
  rcut    the octupole error of the multipole truncation over a grid of region-I radii
  images  the QM-QM periodic images: energy, gradient and Fock matrix
  batch   V, energy and gradient of several uneven MD frames through one recorded graph

Systems are drawn as the benchmark's are: QM atoms in a sphere (or a cluster of waters) with a seeded
contracted Cartesian basis, rigid three-site waters on a jittered lattice as MM charges.  The handle is
created at a nearby geometry and the pass moves it to the state's own, as an MD step does.

The mixed-precision path holds 1e-6 of each result, no more than single precision carries; the
programs that ask for it keep its results in single precision, and so do the cases that use it.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2408_03273_gb300 as q

BOHR = 0.52917721092  # Angstrom
DEV = "cuda"
ZNUC = {"H": 1.0, "C": 6.0, "N": 7.0, "O": 8.0}
MIX = (("C", 20), ("N", 4), ("O", 6), ("H", 30))  # the active site's elements
# shells per element of the basis recipes: heavy atoms, hydrogen
BASIS = {"small": ("3s2p1d", "2s1p"), "site": ("6s4p3d", "4s2p1d"), "site_f": ("6s4p3d2f", "3s1p1d"),
         "spdf": ("1s1p1d1f", "1s1p")}


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
WATER = dict(natm=3, qm="water", basis="small", nprim=3, waters=215, box=18.6, aspect=1.0, cutoff=9.0, alpha=0.35,
             kmax=7, sigma=0.2, points=0.0)
SITE = dict(natm=60, qm="sphere", basis="site", nprim=0, waters=20000, box=58.0, aspect=1.0, cutoff=12.0, alpha=0.3,
            kmax=16, sigma=0.2, points=0.0)
LARGE = dict(natm=150, qm="sphere", basis="site_f", nprim=0, waters=66667, box=86.0, aspect=1.0, cutoff=12.0,
             alpha=0.3, kmax=24, sigma=0.2, points=0.0)


def listed():
    return [
        # a QM water in a small water box, driven by autograd as a torch program does: the smallest
        # calls, where latency and launches count
        dict(WATER, name="water_grad_fp64", kind="grad", mixed=False),
        # the same system's MD step in mixed precision
        dict(WATER, name="water_step_mixed", kind="step", mixed=True),
        # an uneven middle size: ragged box, f shells, half the MM charges bare points
        dict(name="ragged_step_fp64", kind="step", mixed=False, natm=17, qm="sphere", basis="spdf", nprim=0,
             waters=1931, box=39.0, aspect=1.13, cutoff=10.5, alpha=0.32, kmax=11, sigma=0.2, points=0.5),
        # an enzyme active site, the ordinary MD step in both precisions
        dict(SITE, name="site_step_fp64", kind="step", mixed=False),
        dict(SITE, name="site_step_mixed", kind="step", mixed=True),
        # an SCF iteration of the active site
        dict(SITE, name="site_scf_fp64", kind="scf", mixed=False),
        # the choice of the region-I radius from the predicted density, made once per MD step
        dict(SITE, name="site_rcut_fp64", kind="rcut", mixed=False),
        # the periodic images of the active site, added in small cells
        dict(SITE, name="site_images_fp64", kind="images", mixed=False),
        # the large site with f shells: the largest step, in both precisions
        dict(LARGE, name="large_step_fp64", kind="step", mixed=False),
        dict(LARGE, name="large_step_mixed", kind="step", mixed=True),
        # uneven MD frames (QM water clusters of 21 to 120 atoms) through one recorded graph
        dict(name="frames_batch_mixed", kind="batch", mixed=True, frames=8, natm=120, qm="water", basis="small",
             nprim=3, waters=39500, box=105.7, aspect=1.0, cutoff=12.0, alpha=0.3, kmax=30, sigma=0.2, points=0.0),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["step", "step", "step", "step", "grad", "scf", "rcut", "images", "batch"])
    mixed = kind == "batch" or (kind == "step" and rng.random() < 0.5)
    natm = int(round(log(3, 120)))
    qm = "water" if kind == "batch" or rng.random() < 0.3 else "sphere"
    basis = "small" if qm == "water" else rng.choice(["small", "site", "site_f", "spdf"])
    waters = int(round(log(200, 40000)))
    if qm == "water":
        natm = max(3, natm // 3 * 3)
    if kind == "batch":  # the frames of one run: the size is the largest frame's
        natm, waters = max(21, natm), max(2000, waters)
    aspect = rng.choice([1.0, 1.0, round(rng.uniform(0.9, 1.2), 3)])
    box = round((3 * waters / 0.1003) ** (1 / 3) * rng.uniform(0.98, 1.1), 2)
    box = max(box, 2 * (3.0 + qm_radius(natm, qm)) / 0.9, 18.2)
    cutoff = round(min(rng.uniform(8.5, 12.5), 0.49 * 0.9 * box), 2)
    alpha = round(3.6 / cutoff, 3)
    kmax = max(5, int(math.ceil(16 * box / 58.0)) + rng.randint(-1, 1))
    c = dict(kind=kind, mixed=mixed, natm=natm, qm=qm, basis=basis, nprim=rng.choice([0, 3]), waters=waters,
             box=round(box, 2), aspect=aspect, cutoff=cutoff, alpha=alpha, kmax=kmax,
             sigma=rng.choice([0.2, round(rng.uniform(0.15, 0.5), 3)]), points=rng.choice([0.0, 0.0, 0.5, 1.0]))
    if kind == "batch":
        c["frames"] = rng.randint(2, 8)
    return c


# ------------------------------------------------------------------------------------------------
# seeded systems (numpy)
# ------------------------------------------------------------------------------------------------
def qm_radius(natm, qm):
    """Radius (Angstrom) of the QM sphere: the active site's density, or water's."""
    if qm == "water":
        return max(3.0, (natm / 3 / 0.0334 * 3 / (4 * math.pi)) ** (1 / 3)) if natm > 3 else 1.0
    return 10.0 * (natm / 60.0) ** (1 / 3)


def rotations(rng, n):
    u = rng.standard_normal((4, n))
    w, x, y, z = u / np.linalg.norm(u, axis=0)
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                     [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                     [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]]).transpose(2, 0, 1)


def water_sites():
    r, th = 0.9572, math.radians(104.52)
    return np.array([[0.0, 0.0, 0.0], [r * math.sin(th / 2), r * math.cos(th / 2), 0.0],
                     [-r * math.sin(th / 2), r * math.cos(th / 2), 0.0]])


def points_in_sphere(rng, n, radius, dmin):
    pts = np.zeros((0, 3))
    while len(pts) < n:
        for p in rng.uniform(-radius, radius, (256, 3)):
            if p @ p <= radius * radius and (len(pts) == 0 or ((pts - p) ** 2).sum(1).min() >= dmin * dmin):
                pts = np.vstack([pts, p])
                if len(pts) == n:
                    break
        radius *= 1.01  # a crowded sphere grows until all atoms fit
    return pts


def system(case, seed):
    """Geometry, basis and charges in bohr, laid out as qmmm_create takes them."""
    rng = np.random.default_rng([seed, 2408])
    natm, radius = case["natm"], qm_radius(case["natm"], case["qm"])
    if case["qm"] == "water":
        o = points_in_sphere(rng, natm // 3, radius, 2.6) if natm > 3 else np.zeros((1, 3))
        qm = (o[:, None] + np.einsum("nij,kj->nki", rotations(rng, len(o)), water_sites())).reshape(-1, 3)
        elems = ["O", "H", "H"] * (natm // 3)
    else:
        qm = points_in_sphere(rng, natm, radius, 1.0)
        pool = [e for e, n in MIX for _ in range(n)]
        elems = [pool[i % 60] for i in rng.permutation(natm)]
    heavy, light = BASIS[case["basis"]]
    atom, ang, nprim, exps, coef = [], [], [], [], []
    for a, e in enumerate(elems):
        spec = light if e == "H" else heavy
        for count, l in zip(spec[::2], spec[1::2]):
            for _ in range(int(count)):
                n = case["nprim"] or int(rng.integers(1, 6))
                atom.append(a), ang.append("spdf".index(l)), nprim.append(n)
                exps.append(np.exp(rng.uniform(math.log(0.1), math.log(50.0), n)))
                coef.append(rng.uniform(0.1, 1.0, n))
    box = np.array([case["box"], case["box"] / case["aspect"], case["box"]])
    n_side = int(math.ceil((case["waters"] - 1e-9) ** (1 / 3)))
    while True:  # the coarsest lattice with enough sites 2 Angstrom clear of every QM atom
        site = np.stack(np.meshgrid(*[np.arange(n_side)] * 3, indexing="ij"), -1).reshape(-1, 3)
        site = (site + 0.5) * (box / n_side) - box / 2 + rng.uniform(-0.3, 0.3, site.shape)
        near = np.nonzero(((site - qm.mean(0)) ** 2).sum(1) < (np.sqrt(((qm - qm.mean(0)) ** 2).sum(1).max()) + 2.0) ** 2)[0]
        clear = np.ones(len(site), bool)
        clear[near] = (((site[near][:, None] - qm[None]) ** 2).sum(-1).min(1)) >= 4.0
        if clear.sum() >= case["waters"]:
            break
        n_side += 1
    site = site[np.sort(rng.choice(np.nonzero(clear)[0], case["waters"], replace=False))]
    mol = site[:, None] + np.einsum("nij,kj->nki", rotations(rng, len(site)), water_sites())
    nmm = 3 * len(mol)
    sigma = np.full(nmm, case["sigma"] / BOHR)
    sigma.reshape(-1, 3)[rng.random(len(mol)) < case["points"]] = 0.0
    nprim = np.array(nprim, np.int32)
    return SimpleNamespace(
        elems=elems, atom_xyz=qm / BOHR, atom_Z=np.array([ZNUC[e] for e in elems]),
        shell_atom=np.array(atom, np.int32), shell_l=np.array(ang, np.int32), shell_nprim=nprim,
        shell_prim_offset=(np.cumsum(nprim) - nprim).astype(np.int32), prim_exp=np.concatenate(exps),
        prim_coeff=np.concatenate(coef), mm_xyz=mol.reshape(-1, 3) / BOHR,
        mm_q=np.tile([-0.834, 0.417, 0.417], len(mol)), mm_sigma=sigma, box=box / BOHR, cutoff=case["cutoff"] / BOHR,
        ewald_alpha=case["alpha"] * BOHR, kmax=(case["kmax"],) * 3, ewald_rcut=0.0,
        nao=sum((l + 1) * (l + 2) // 2 for l in ang))


def moved(s, seed):
    """The geometry of the state's own step: every site up to 0.03 bohr from where the handle was made."""
    rng = np.random.default_rng([seed, 7])
    return (s.atom_xyz + rng.uniform(-0.03, 0.03, s.atom_xyz.shape),
            s.mm_xyz + rng.uniform(-0.03, 0.03, s.mm_xyz.shape))


def density(s, seed, device):
    """Random symmetric positive density matrix with the trace of the nuclear charge."""
    g = torch.Generator(device=device).manual_seed(seed)
    x = torch.randn(s.nao, s.nao, dtype=torch.float64, device=device, generator=g)
    d = x @ x.T
    return (d + d.T) * (0.5 * float(s.atom_Z.sum()) / float(d.diagonal().sum()))


def frames_of(case):
    """The single frames of a batch: sizes spread from the largest down to about a sixth of it."""
    n, out = case["frames"], []
    for f in range(n):
        w = 1.0 - 0.83 * f / max(1, n - 1)
        waters = max(200, int(case["waters"] * w))
        box = max(case["box"] * (waters / case["waters"]) ** (1 / 3), 2 * case["cutoff"] * 1.01 * max(case["aspect"], 1))
        natm = max(21, int(case["natm"] * w) // 3 * 3)
        out.append({**case, "natm": min(natm, case["natm"]), "waters": waters, "box": box,
                    "kmax": max(5, min(case["kmax"], int(math.ceil(16 * box / 58.0))))})
    return out


# ------------------------------------------------------------------------------------------------
# the calls
# ------------------------------------------------------------------------------------------------
R_LO, R_STEP, R_N = 10.0, 0.5, 25  # region-I radii (bohr) of the octupole error scan


def prepare_one(case, seed):
    s = system(case, seed)
    st = SimpleNamespace(kind=case["kind"], mixed=case["mixed"], nmm=len(s.mm_q))
    st.handle = q.Handle(s, precision=q.QMMM_MIXED if case["mixed"] else q.QMMM_FP64)
    qm, mm = moved(s, seed)
    st.qm, st.mm, st.q = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (qm, mm, s.mm_q))
    st.dm = density(s, seed, DEV)
    if case["kind"] in ("scf", "rcut", "images", "batch"):  # at the step's geometry already
        st.handle.set_positions(st.qm, st.mm, st.q)
    if case["kind"] == "scf":
        st.handle.vpot(like=st.dm)
    return st


def prepare(case, seed):
    if case["kind"] != "batch":
        return prepare_one(case, seed)
    fs = [prepare_one(c, 1000 * seed + i) for i, c in enumerate(frames_of(case))]
    new = lambda *shape: torch.empty(shape, dtype=torch.float64, device=DEV)  # noqa: E731
    st = SimpleNamespace(kind="batch", mixed=case["mixed"], frames=fs, dm=[f.dm for f in fs])
    st.batch = q.Batch([f.handle for f in fs])
    st.V = [new(*f.dm.shape) for f in fs]
    st.E = [new(4) for f in fs]
    st.gq = [new(*f.qm.shape) for f in fs]
    st.gm = [new(*f.mm.shape) for f in fs]
    st.gc = [new(f.nmm) for f in fs]
    return st


def run(st):
    if st.kind == "batch":  # the next MD step's frames
        for f in st.frames:
            f.handle.set_positions(f.qm, f.mm, f.q)
        st.batch.run(st.dm, st.V, st.E, st.gq, st.gm, st.gc)
        out = {k: getattr(st, k) for k in ("V", "E", "gq", "gm", "gc")}
        return {k: [x.float() for x in v] for k, v in out.items()} if st.mixed else out
    h, dm = st.handle, st.dm
    if st.kind == "step":
        h.set_positions(st.qm, st.mm, st.q)
        V, Enuc = h.vpot(like=dm)
        E = h.energy(dm)
        gq, gm, gc = h.forces(dm)
        out = {"V": V, "Enuc": Enuc, "E": E, "gq": gq, "gm": gm, "gc": gc}
    elif st.kind == "grad":
        x = [t.detach().requires_grad_() for t in (dm, st.qm, st.mm, st.q)]
        E = q.QMMMEnergy.apply(h, *x)
        E.backward()
        out = {"E": E.detach(), "gdm": x[0].grad, "gq": x[1].grad, "gm": x[2].grad, "gc": x[3].grad}
    elif st.kind == "scf":
        EII, M, F = h.ewald(dm, want_F=True)
        out = {"EII": EII, "M": M, "F": F, "E": h.energy(dm), "G": h.density_gradient(dm)}
    elif st.kind == "rcut":
        err, octu = h.octupole_error(dm, R_LO, R_STEP, R_N, want_octupoles=True)
        out = {"err": err, "oct": octu}
    else:
        E, g, F = h.qm_images(dm, want_F=True)
        out = {"E": E, "gq": g, "F": F}
    return {k: v.float() for k, v in out.items()} if st.mixed else out


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------
def work(case):
    if case["kind"] == "batch":
        w = [work({**c, "kind": "step"}) for c in frames_of(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    s = system(case, 0)
    natm, nmm, n2, k = case["natm"], len(s.mm_q), s.nao * s.nao, case["kmax"]
    b = basis_of(s, "cpu")
    nI = nmm * 4 / 3 * math.pi * s.cutoff ** 3 / float(np.prod(s.box))
    sweep = moments = 0.0
    for la, lb, i, j in b.pairs(s.atom_xyz, 1e-14):
        L, n = la + lb, len(i)
        c3, c4, c5 = (math.comb(L + m, 3 if m == 3 else 4) for m in (3, 4, 5))
        # Hermite integrals and their gradient against every region-I charge
        sweep += n * nI * ((40 + 3 * L + 2 * c4 + 2 * c3) + (75 + 3 * L + 2 * c5 + 10 * c3))
        moments += n * 40.0 * ((la + 1) * (la + 2) // 2) * ((lb + 1) * (lb + 2) // 2)
    grid = (k + 1) * (2 * k + 1) ** 2
    # reciprocal sums by separable phases: the MM structure factor, and the charge and force sums
    recip = 8.0 * (2 * k + 1) * (k + 1) * (2 * nmm + 8 * nmm) + 60.0 * grid * natm
    near = 200.0 * natm * nI
    return {"step": {"bytes": 8.0 * (3 * n2 + 8 * nmm), "flops": sweep + recip + near + 2 * moments},
            "grad": {"bytes": 8.0 * (3 * n2 + 8 * nmm), "flops": sweep + recip + near + 3 * moments},
            "scf": {"bytes": 8.0 * 4 * n2, "flops": 2 * moments},
            "rcut": {"bytes": 8.0 * (n2 + 4 * nmm), "flops": moments + 100.0 * natm * nI},
            "images": {"bytes": 8.0 * 2 * n2, "flops": 2 * moments + 20.0 * natm * natm * grid}}[case["kind"]]


# ------------------------------------------------------------------------------------------------
# the same results by plain torch in 64 bits: Hermite integrals over all screened primitive pairs with
# autograd for the gradients, Ewald sums by separable phases
# ------------------------------------------------------------------------------------------------
def carts(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def odd_fact(n):
    return math.prod(range(2 * n - 1, 0, -2)) if n > 0 else 1


def basis_of(s, device):
    """Primitives with normalised coefficients, and the screened pair lists per (l_a >= l_b)."""
    b = SimpleNamespace()
    prim_shell = np.repeat(np.arange(len(s.shell_l)), s.shell_nprim)
    l, a = s.shell_l[prim_shell], s.prim_exp
    c = s.prim_coeff * (2 * a / math.pi) ** 0.75 * (4 * a) ** (l / 2) / np.sqrt([odd_fact(k) for k in l])
    for sh in range(len(s.shell_l)):
        m = slice(s.shell_prim_offset[sh], s.shell_prim_offset[sh] + s.shell_nprim[sh])
        p, ll = a[m][:, None] + a[m], int(s.shell_l[sh])
        c[m] /= math.sqrt((np.outer(c[m], c[m]) * odd_fact(ll) / (2 * p) ** ll * (math.pi / p) ** 1.5).sum())
    ao = np.cumsum([0] + [(k + 1) * (k + 2) // 2 for k in s.shell_l])[:-1]
    t = lambda x: torch.as_tensor(x, device=device)  # noqa: E731
    b.exp, b.coef, b.shell, b.l = t(a), t(c), t(prim_shell), t(l.astype(np.int64))
    b.atom, b.ao = t(s.shell_atom[prim_shell].astype(np.int64)), t(ao[prim_shell])

    def pairs(xyz, tol):
        x = torch.as_tensor(xyz, device=device)
        vals = []
        top = 0.0
        for la in range(int(l.max()) + 1):
            for lb in range(la + 1):
                ia, ib = (torch.nonzero(b.l == k)[:, 0] for k in (la, lb))
                if len(ia) == 0 or len(ib) == 0:
                    continue
                p = b.exp[ia, None] + b.exp[ib]
                ab = torch.cdist(x[b.atom[ia]], x[b.atom[ib]], compute_mode="donot_use_mm_for_euclid_dist")
                v = (b.coef[ia, None] * b.coef[ib]).abs() * (math.pi / p) ** 1.5
                v *= torch.exp(-b.exp[ia, None] * b.exp[ib] / p * ab * ab)
                v *= (b.exp[ib] / p * ab + p ** -0.5) ** la * (b.exp[ia, None] / p * ab + p ** -0.5) ** lb
                if la == lb:  # each shell pair once
                    v[b.shell[ia][:, None] > b.shell[ib]] = 0.0
                top = max(top, float(v.max()))
                vals.append((la, lb, ia, ib, v))
        for la, lb, ia, ib, v in vals:
            i, j = torch.nonzero(v >= tol * top, as_tuple=True)
            if len(i):
                yield la, lb, ia[i], ib[j]

    b.pairs = pairs
    return b


class Boys(torch.autograd.Function):
    """F_0 .. F_m of T, stacked; the derivative of F_k is -F_{k+1}."""

    @staticmethod
    def forward(ctx, T, m):
        F = torch.empty((m + 2,) + T.shape, dtype=T.dtype, device=T.device)
        e, big = torch.exp(-T), T.clamp(min=30.0)
        F[0] = 0.5 * torch.sqrt(math.pi / big) * torch.erf(torch.sqrt(big))
        for k in range(m + 1):
            F[k + 1] = ((2 * k + 1) * F[k] - e) / (2 * big)
        small = torch.nonzero(T < 30.0, as_tuple=True)
        t, et = T[small], e[small]
        term = torch.full_like(t, 1.0 / (2 * m + 3))
        f = term.clone()
        for k in range(1, 160):
            term = term * (2 * t / (2 * m + 3 + 2 * k))
            f += term
        f *= et
        for k in range(m + 1, -1, -1):
            F[k][small] = f
            f = (2 * t * f + et) / (2 * k - 1) if k else f
        ctx.save_for_backward(F)
        return F[:-1].clone()

    @staticmethod
    def backward(ctx, g):
        (F,) = ctx.saved_tensors
        return -(g * F[1:]).sum(0), None


def hermite_r(T, rho, d, L):
    """R_tuv of all charges and pairs, as a dict."""
    F = Boys.apply(T, L)
    lev = {(0, 0, 0): F[L] * (-2 * rho) ** L}
    for n in range(L - 1, -1, -1):
        new = {(0, 0, 0): F[n] * (-2 * rho) ** n}
        for k in range(1, L - n + 1):
            for tuv in carts(k):
                ax = next(a for a in range(3) if tuv[a])
                m1 = tuple(x - (a == ax) for a, x in enumerate(tuv))
                r = d[ax] * lev[m1]
                if m1[ax] > 0:
                    r = r + m1[ax] * lev[tuple(x - (a == ax) for a, x in enumerate(m1))]
                new[tuv] = r
        lev = new
    return lev


def hermite_e(la, lb, pa, pb, p):
    """E[i][j][t] of one direction."""
    E = {(0, 0, 0): torch.ones_like(p)}
    get = lambda i, j, t: E.get((i, j, t))  # noqa: E731
    for i in range(la + 1):
        for j in range(lb + 1):
            if i == j == 0:
                continue
            (pi, pj), x = ((i - 1, j), pa) if i else ((i, j - 1), pb)
            for t in range(i + j + 1):
                parts = [(get(pi, pj, t - 1), 0.5 / p), (get(pi, pj, t), x), (get(pi, pj, t + 1), t + 1.0)]
                E[i, j, t] = sum(e * f for e, f in parts if e is not None)
    return E


def pair_geometry(b, i, j, xyz):
    a, c = b.exp[i], b.exp[j]
    A, B, p = xyz[b.atom[i]], xyz[b.atom[j]], a + c
    P = (a[:, None] * A + c[:, None] * B) / p[:, None]
    pref = b.coef[i] * b.coef[j] * torch.exp(-a * c / p * ((A - B) ** 2).sum(1))
    return A, B, p, P, pref


def block_index(b, i, j, la, lb, nao):
    """Flat indices of the AO blocks of the pairs and of their mirrors, and which have a mirror."""
    r = (b.ao[i][:, None] + torch.arange(len(carts(la)), device=i.device))[:, :, None]
    c = (b.ao[j][:, None] + torch.arange(len(carts(lb)), device=i.device))[:, None, :]
    return r * nao + c, c * nao + r, b.shell[i] != b.shell[j]


def region(s, qm, mm):
    """Region-I images: index and position shift."""
    d = mm - qm.mean(0)
    shift = -torch.round(d / s.tbox) * s.tbox
    return torch.nonzero(((d + shift) ** 2).sum(1) < s.cutoff ** 2)[:, 0], shift


def electronic(s, b, qm, mm, ch, dm, grads):
    """V of region I; the gradients of sum(dm V) go into the leaves' .grad if asked."""
    idx, shift = region(s, qm.detach(), mm.detach())
    V = torch.zeros(s.nao * s.nao, dtype=torch.float64, device=dm.device)
    kap = torch.where(s.tsigma[idx] > 0, s.tsigma[idx].clamp(min=1e-30) ** -2, torch.zeros_like(s.tsigma[idx]))
    flat = dm.reshape(-1)

    def charge_sums(i, j, L):
        """W_tuv of the pairs (i, j), stacked over carts(0..L)."""
        _, _, p, P, _ = pair_geometry(b, i, j, qm)
        C = mm[idx] + shift[idx]
        f = torch.where(kap > 0, kap / (p[:, None] + kap), torch.ones_like(p[:, None] + kap))
        d = [P[:, a, None] - C[:, a] for a in range(3)]
        R = hermite_r(p[:, None] * f * (d[0] ** 2 + d[1] ** 2 + d[2] ** 2), p[:, None] * f, d, L)
        w = -ch[idx] * f.sqrt() * (2 * math.pi / p)[:, None]
        return torch.stack([(w * R[t]).sum(1) for k in range(L + 1) for t in carts(k)])

    for la, lb, I, J in b.pairs(qm.detach(), 1e-16):
        L, step = la + lb, max(1, int(1e7 / (la + lb + 1)) // max(1, len(idx)))
        chunks = [(I[k:k + step], J[k:k + step]) for k in range(0, len(I), step)]
        with torch.no_grad():
            W = torch.cat([charge_sums(i, j, L) for i, j in chunks], 1)
        with torch.set_grad_enabled(grads):
            W.requires_grad_(grads)
            Wd = dict(zip([t for k in range(L + 1) for t in carts(k)], W))
            A, B, p, P, pref = pair_geometry(b, I, J, qm)
            E = [hermite_e(la, lb, P[:, a] - A[:, a], P[:, a] - B[:, a], p) for a in range(3)]
            blk = torch.stack([
                sum(E[0][x[0], y[0], t] * E[1][x[1], y[1], u] * E[2][x[2], y[2], v] * Wd[t, u, v]
                    for t in range(x[0] + y[0] + 1) for u in range(x[1] + y[1] + 1) for v in range(x[2] + y[2] + 1))
                for x in carts(la) for y in carts(lb)], 1).reshape(len(I), len(carts(la)), len(carts(lb)))
            blk = pref[:, None, None] * blk
            n1, n2, two = block_index(b, I, J, la, lb, s.nao)
            if grads:
                g = torch.where(two[:, None, None], flat[n1] + flat[n2], flat[n1])
                (g * blk).sum().backward()
        if grads:
            done = 0
            for i, j in chunks:
                (charge_sums(i, j, L) * W.grad[:, done:done + len(i)]).sum().backward()
                done += len(i)
        V.index_add_(0, n1.reshape(-1), blk.detach().reshape(-1))
        V.index_add_(0, n2[two].reshape(-1), blk.detach()[two].reshape(-1))
    return V.reshape(s.nao, s.nao)


def nuclear(s, qm, mm, ch):
    idx, shift = region(s, qm.detach(), mm.detach())
    r = (qm[:, None] - (mm[idx] + shift[idx])[None]).norm(dim=-1)
    sg = s.tsigma[idx]
    f = torch.where(sg > 0, torch.erf(r / torch.where(sg > 0, sg, torch.ones_like(sg))), torch.ones_like(r)) / r
    return (s.tZ[:, None] * ch[idx] * f).sum()


def fold_moments(s, b, qm, dm, order, want=None):
    """Per-atom sums m[atom, e] = sum_{mu on atom} sum_nu dm <mu|(r - R)^e|nu>; with want[atom, e] the matrix
    X_{mu nu} = sum_e want[atom of mu, e] <mu|(r - R)^e|nu> instead of the sums."""
    comps = [e for k in range(order + 1) for e in carts(k)]
    out = torch.zeros(len(s.atom_Z), len(comps), dtype=torch.float64, device=dm.device)
    X = torch.zeros(s.nao * s.nao, dtype=torch.float64, device=dm.device)
    flat = dm.reshape(-1)
    for la, lb, I, J in b.pairs(qm.detach(), 1e-16):
        step = 400000 // (len(carts(la)) * len(carts(lb)))
        for k in range(0, len(I), step):
            i, j = I[k:k + step], J[k:k + step]
            A, B, p, P, pref = pair_geometry(b, i, j, qm)
            pref = pref * (math.pi / p) ** 1.5
            S = [hermite_e(la + order, lb + order, P[:, a] - A[:, a], P[:, a] - B[:, a], p) for a in range(3)]
            n1, n2, two = block_index(b, i, j, la, lb, s.nao)
            for side in (0, 1):  # moments about the first shell's atom, then about the second's
                g = flat[n1] if side == 0 else torch.where(two[:, None, None], flat[n2], torch.zeros_like(flat[n2]))
                n = n1 if side == 0 else n2
                at = b.atom[i] if side == 0 else b.atom[j]
                xs = 0.0
                for ie, e in enumerate(comps):
                    blk = torch.stack([
                        S[0][x[0] + e[0] * (side == 0), y[0] + e[0] * (side == 1), 0] *
                        S[1][x[1] + e[1] * (side == 0), y[1] + e[1] * (side == 1), 0] *
                        S[2][x[2] + e[2] * (side == 0), y[2] + e[2] * (side == 1), 0]
                        for x in carts(la) for y in carts(lb)],
                        1).reshape(len(i), len(carts(la)), len(carts(lb))) * pref[:, None, None]
                    if want is None:
                        one = torch.zeros(len(s.atom_Z), dtype=torch.float64, device=dm.device)
                        col = torch.zeros(len(comps), dtype=torch.float64, device=dm.device)
                        col[ie] = 1.0
                        out = out + one.index_add(0, at, (g * blk).sum((1, 2)))[:, None] * col
                    else:
                        xs = xs + want[at, ie][:, None, None] * blk
                if want is not None:
                    keep = torch.ones_like(two) if side == 0 else two
                    X.index_add_(0, n[keep].reshape(-1), xs[keep].reshape(-1))
    return out if want is None else X.reshape(s.nao, s.nao)


W10 = (1.0, 1, 1, 1, 1, 2, 2, 1, 2, 1)  # weights of the stored (Q, mu, theta) components


def radial(r2, beta):
    """f, f'/r, (f'/r)'/r and once more, of 1/r (beta 0) or erfc(beta r)/r."""
    r = r2.sqrt()
    point = beta == 0
    e = torch.where(point, torch.zeros_like(r), torch.exp(-beta * beta * r2) * 2 * beta / math.sqrt(math.pi))
    f = torch.where(point, 1 / r, torch.erfc(beta * r) / r)
    g1 = -(f + e) / r2
    g2 = (-3 * g1 + 2 * beta ** 2 * e) / r2
    g3 = (-5 * g2 - 4 * beta ** 4 * e) / r2
    return f, g1, g2, g3


def tensor_energy(M, qi, d, beta):
    """sum of q_i M_j . T(R_j - R_i) over pairs; M [n, 10], d [n, 3]."""
    f, g1, g2, _ = radial((d * d).sum(1), beta)
    x, y, z = d.unbind(1)
    quad = M[:, 4] * (g1 + x * x * g2) + M[:, 7] * (g1 + y * y * g2) + M[:, 9] * (g1 + z * z * g2)
    quad = quad + 2 * (M[:, 5] * x * y + M[:, 6] * x * z + M[:, 8] * y * z) * g2
    return (qi * (M[:, 0] * f + (M[:, 1] * x + M[:, 2] * y + M[:, 3] * z) * g1 + 0.5 * quad)).sum()


def near_pairs(s, qm, mm, rmax):
    """(atom, charge, shift) with minimum-image distance below rmax[charge]."""
    out = []
    for j in range(len(qm)):
        d = qm[j] - mm
        shift = torch.round(d / s.tbox) * s.tbox
        i = torch.nonzero(((d - shift) ** 2).sum(1) < rmax ** 2)[:, 0]
        out.append((torch.full_like(i, j), i, shift[i]))
    return tuple(torch.cat(x) for x in zip(*out))


def multipole_energy(s, M, qm, mm, ch):
    """E_II of the real-space and background terms (Ewald, minus bare T over region I, minus screened T over II)."""
    z = torch.zeros_like(s.tsigma)
    j, i, sh = near_pairs(s, qm.detach(), mm.detach(), torch.full_like(z, s.cutoff))
    E = tensor_energy(M[j], ch[i], qm[j] - mm[i] - sh, torch.full_like(z[i], s.ewald_alpha))
    idx, shift = region(s, qm.detach(), mm.detach())
    n = len(qm)
    j, i = torch.arange(n, device=qm.device).repeat_interleave(len(idx)), idx.repeat(n)
    E = E - tensor_energy(M[j], ch[i], qm[j] - mm[i] - shift[i], z[i])
    inside = torch.zeros_like(z, dtype=torch.bool)
    inside[idx] = True
    j, i, sh = near_pairs(s, qm.detach(), mm.detach(), 9 * s.tsigma)
    d = qm.detach()[j] - mm.detach()[i] - sh  # an image of region II: not the region-I image itself
    same = inside[i] & ((mm.detach()[i] + sh - mm.detach()[i] - shift[i]).abs().sum(1) < 1e-6)
    j, i, sh = j[~same], i[~same], sh[~same]
    if len(d) and len(j):
        E = E - tensor_energy(M[j], ch[i], qm[j] - mm[i] - sh, 1 / s.tsigma[i])
    return E - math.pi / (s.vol * s.ewald_alpha ** 2) * ch.sum() * M[:, 0].sum()


def gvectors(s):
    k = [torch.arange(-n, n + 1, device=s.tbox.device, dtype=torch.float64) for n in s.kmax]
    return [2 * math.pi * k[a] / s.tbox[a] for a in range(3)]


def structure(s, mm, ch):
    """S(G) = sum q exp(iG.R) and, for field A(G), the sums on the charges; by separable phases."""
    gx, gy, gz = gvectors(s)
    S = torch.zeros(len(gx), len(gy) * len(gz), dtype=torch.complex128, device=mm.device)
    for k in range(0, len(mm), 16384):
        x, y, z = mm[k:k + 16384].unbind(1)
        px, py, pz = (torch.exp(1j * g * t[:, None]) for g, t in ((gx, x), (gy, y), (gz, z)))
        S += (px * ch[k:k + 16384, None]).T @ (py[:, :, None] * pz[:, None, :]).reshape(len(x), -1)
    return S.reshape(len(gx), len(gy), len(gz))


def on_charges(s, mm, ch, A):
    """dE/dq and dE/dR on the charges of E = sum_G Re(conj(S) A)."""
    gx, gy, gz = gvectors(s)
    C = [A, gx[:, None, None] * A, gy[None, :, None] * A, gz[None, None, :] * A]
    C = torch.cat([c.reshape(len(gx), -1) for c in C]).T.contiguous()
    out = []
    for k in range(0, len(mm), 16384):
        x, y, z = mm[k:k + 16384].unbind(1)
        px, py, pz = (torch.exp(-1j * g * t[:, None]) for g, t in ((gx, x), (gy, y), (gz, z)))
        T = ((py[:, :, None] * pz[:, None, :]).reshape(len(x), -1) @ C).reshape(len(x), 4, len(gx))
        out.append((T * px[:, None]).sum(2))
    T = torch.cat(out)
    return T[:, 0].real, ch[:, None] * T[:, 1:].imag


def recip_field(s, M, qm):
    """A(G) = g(G) sum_j (Q + iG.mu - G.theta.G/2...) exp(iG.R_j)."""
    gx, gy, gz = gvectors(s)
    g2 = gx[:, None, None] ** 2 + gy[None, :, None] ** 2 + gz[None, None, :] ** 2
    w = torch.where(g2 > 0, 4 * math.pi / s.vol * torch.exp(-g2 / (4 * s.ewald_alpha ** 2)) / g2.clamp(min=1e-300),
                    torch.zeros_like(g2))
    A = 0.0
    X, Y, Z = gx[:, None, None], gy[None, :, None], gz[None, None, :]
    for j in range(len(qm)):
        ph = [torch.exp(1j * g * qm[j, a]) for a, g in enumerate((gx, gy, gz))]
        m = M[j]
        re = m[0] - 0.5 * (m[4] * X * X + m[7] * Y * Y + m[9] * Z * Z) - m[5] * X * Y - m[6] * X * Z - m[8] * Y * Z
        im = m[1] * X + m[2] * Y + m[3] * Z
        A = A + torch.complex(re, im) * (ph[0][:, None, None] * ph[1][None, :, None] * ph[2][None, None, :])
    return w * A


def recip_on_atoms(s, M, qm, mm, ch, grads):
    """Reciprocal part of E_II: its value and, through the leaves M and qm, its gradients, atom by atom."""
    S = structure(s, mm.detach(), ch.detach())
    total = 0.0
    for j in range(len(qm)):
        with torch.set_grad_enabled(grads):
            E = (torch.view_as_real(recip_field(s, M[j:j + 1], qm[j:j + 1])) * torch.view_as_real(S)).sum()
            if grads:
                E.backward()
        total += E.item()
    return total


def leaf(x):
    return x.detach().clone().requires_grad_()


def context(case, seed):
    s = system(case, seed)
    qm, mm = (torch.from_numpy(x).to(DEV) for x in moved(s, seed))
    ch = torch.from_numpy(s.mm_q).to(DEV)
    s.tbox, s.tsigma, s.tZ = (torch.from_numpy(x).to(DEV) for x in (s.box, s.mm_sigma, s.atom_Z))
    s.vol = float(np.prod(s.box))
    return s, basis_of(s, DEV), qm, mm, ch, density(s, seed, DEV)


def multipoles(s, b, qm, dm):
    m = -fold_moments(s, b, qm, dm, 2)
    return m + torch.nn.functional.pad(s.tZ[:, None], (0, 9))


def energy_II(s, M, qm, mm, ch):
    """E_II with v[atom, 10] = dE_II/dM over the weights, and its gradients at fixed multipoles."""
    m, x, y, c = leaf(M), leaf(qm), leaf(mm), leaf(ch)
    E = multipole_energy(s, m, x, y, c)
    E.backward()
    total = E.item() + recip_on_atoms(s, m, x, y, c, True)
    with torch.no_grad():
        dq, dR = on_charges(s, mm, ch, recip_field(s, M, qm))
    return total, m.grad, x.grad, y.grad + dR, c.grad + dq


def fock(s, b, qm, dm, v):
    """-(X + X^T)/2 with X the moments weighted by dE/dM (which holds the components' weights)."""
    X = fold_moments(s, b, qm, dm, 2, want=v)
    return -0.5 * (X + X.T)


def exact_step(case, seed):
    s, b, qm, mm, ch, dm = context(case, seed)
    x, y, c = leaf(qm), leaf(mm), leaf(ch)
    V = electronic(s, b, x, y, c, dm, True)
    En = nuclear(s, x, y, c)
    En.backward()
    M = multipoles(s, b, qm, dm)
    EII, v, gq, gm, gc = energy_II(s, M, qm, mm, ch)
    (multipoles(s, b, x, dm) * v).sum().backward()  # the multipoles move with the basis
    EI, En = (dm * V).sum(), En.detach()
    grads = {"gq": x.grad + gq, "gm": y.grad + gm, "gc": c.grad + gc}
    if case["kind"] == "grad":
        return {"E": EI + En + EII, "gdm": V + fock(s, b, qm, dm, v), **grads}
    return {"V": V, "Enuc": En.reshape(1), "E": torch.stack([EI + En + EII, EI, En, 0 * En + EII]), **grads}


def exact_scf(case, seed):
    s, b, qm, mm, ch, dm = context(case, seed)
    V = electronic(s, b, qm, mm, ch, dm, False)
    En = nuclear(s, qm, mm, ch)
    M = multipoles(s, b, qm, dm)
    EII, v = energy_II(s, M, qm, mm, ch)[:2]
    F, EI = fock(s, b, qm, dm, v), (dm * V).sum()
    return {"EII": (0 * En + EII).reshape(1), "M": M, "F": F, "E": torch.stack([EI + En + EII, EI, En, 0 * En + EII]),
            "G": V + F}


def exact_rcut(case, seed):
    """The octupoles; the errors are sums over region II that this file does not restate."""
    s, b, qm, _, _, dm = context(case, seed)
    return {"err": None, "oct": -fold_moments(s, b, qm, dm, 3)[:, 10:]}


def image_energy(s, M, qm):
    """Eq. 5 summed by Ewald: the QM multipoles with all their periodic images."""
    alpha, n = s.ewald_alpha, len(qm)
    X, Y, Z = (g.reshape([-1 if a == b else 1 for b in range(3)]) for a, g in enumerate(gvectors(s)))
    g2 = X * X + Y * Y + Z * Z
    w = torch.where(g2 > 0, 4 * math.pi / s.vol * torch.exp(-g2 / (4 * alpha ** 2)) / g2.clamp(min=1e-300), 0 * g2)
    a0 = a1 = a2 = 0.0
    for j in range(n):
        ph = [torch.exp(1j * g * qm[j, a]) for a, g in enumerate((X, Y, Z))]
        ph, m = ph[0] * ph[1] * ph[2], M[j]
        quad = 0.5 * (m[4] * X * X + m[7] * Y * Y + m[9] * Z * Z) + m[5] * X * Y + m[6] * X * Z + m[8] * Y * Z
        a0, a1, a2 = a0 + m[0] * ph, a1 + 1j * (m[1] * X + m[2] * Y + m[3] * Z) * ph, a2 - quad * ph
    E = 0.5 * (w * ((a0.conj() * (a0 + 2 * a1 + 2 * a2)).real + (a1.conj() * a1).real)).sum()

    def pairs(d, j, i, beta):
        f, g1, h, _ = radial((d * d).sum(1), torch.full_like(d[:, 0], beta))
        mj, mi = M[j], M[i]
        x, y, z = d.unbind(1)
        pj, pi = ((m[:, 1:4] * d).sum(1) for m in (mj, mi))
        quad = mj[:, 4] * (g1 + x * x * h) + mj[:, 7] * (g1 + y * y * h) + mj[:, 9] * (g1 + z * z * h)
        quad = quad + 2 * (mj[:, 5] * x * y + mj[:, 6] * x * z + mj[:, 8] * y * z) * h
        dip = (mj[:, 1:4] * mi[:, 1:4]).sum(1) * g1 + pj * pi * h
        return 0.5 * (mi[:, 0] * (mj[:, 0] * f + 2 * pj * g1 + quad) - dip).sum()

    j, i = torch.arange(n, device=qm.device).repeat_interleave(n), torch.arange(n, device=qm.device).repeat(n)
    for sx in (-1, 0, 1):
        for sy in (-1, 0, 1):
            for sz in (-1, 0, 1):
                sh = torch.tensor([sx, sy, sz], device=qm.device) * s.tbox
                r2 = ((qm.detach()[j] - qm.detach()[i] + sh) ** 2).sum(1)
                k = torch.nonzero((r2 < s.cutoff ** 2) & (r2 > 1e-12))[:, 0]
                E = E + pairs(qm[j[k]] - qm[i[k]] + sh, j[k], i[k], alpha)
    k = torch.nonzero(i != j)[:, 0]
    E = E - pairs(qm[j[k]] - qm[i[k]], j[k], i[k], 0.0)
    f0, h0 = -2 * alpha / math.sqrt(math.pi), 4 / 3 * alpha ** 3 / math.sqrt(math.pi)
    trace = M[:, 4] + M[:, 7] + M[:, 9]
    E = E + 0.5 * (M[:, 0] ** 2 * f0 + M[:, 0] * trace * h0 - (M[:, 1:4] ** 2).sum(1) * h0).sum()
    return E - math.pi / (2 * s.vol * alpha ** 2) * M[:, 0].sum() ** 2


def exact_images(case, seed):
    s, b, qm, _, _, dm = context(case, seed)
    with torch.no_grad():
        M = multipoles(s, b, qm, dm)
    m, x = leaf(M), leaf(qm)
    E = image_energy(s, m, x)
    E.backward()
    (multipoles(s, b, x, dm) * m.grad).sum().backward()
    return {"E": E.detach().reshape(1), "gq": x.grad, "F": fock(s, b, qm, dm, m.grad)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        outs = [exact_step({**c, "kind": "step"}, 1000 * seed + i) for i, c in enumerate(frames_of(case))]
        return {k: [o[k] for o in outs] for k in ("V", "E", "gq", "gm", "gc")}
    one = {"step": exact_step, "grad": exact_step, "scf": exact_scf, "rcut": exact_rcut, "images": exact_images}
    return one[kind](case, seed)
