"""Performance cases of the long-range planewave Coulomb build.

Each case is one call that a periodic-SCF program makes in every iteration:
density matrices D^k in, Coulomb matrices J^k and energies E_J out (or forces),
on a plan made once for the geometry.  Listed are the smallest and the largest
systems and the forms users choose between: the FP64 build (the default), the
split-precision walks, the tensor-core contraction for orthorhombic cells,
per-pair cutoffs, the compact/diffuse classification, host buffers, nuclear
gradients, and batches of uneven cells.

exact() is an independent FP64 evaluation in plain torch (Obara-Saika
recurrences in G space over ordered primitive pairs).
"""
import math

import numpy as np
import torch

EPS_G = 1e-14          # kernel floor exp(-G^2/4w^2) of the G sphere
PAIR_THRESH = 1e-12    # overlap screen of primitive pairs
CUTOFF_EPS = 1e-12     # screening threshold of the per-pair cutoffs

#: (l, smallest exponent, largest exponent, count): even-tempered uncontracted shells
BASIS = {
    "H": [(0, 0.1, 80.0, 5), (1, 0.2, 1.8, 3)],
    "C": [(0, 0.1, 8.0e3, 8), (1, 0.15, 10.0, 4), (2, 0.3, 1.2, 2)],
    "O": [(0, 0.15, 1.5e4, 8), (1, 0.2, 30.0, 4), (2, 0.4, 1.6, 2)],
    "Mg": [(0, 0.08, 2.0e4, 8), (1, 0.1, 50.0, 4), (2, 0.5, 0.5, 1)],
    "X": [(0, 0.2, 10.0, 3), (1, 0.3, 1.0, 2)],
}


def _case(name, system, form, call, k, omega, ndens=1, **more):
    c = dict(name=name, system=system, form=form, call=call, k1=k[0], k2=k[1], k3=k[2], omega=omega, ndens=ndens,
             geometry=0)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call there is: two atoms at the Gamma point, where launches are all of the time
        _case("dimer-fp64", "dimer", "fp64", "build", (1, 1, 1), 0.3),
        # a small low-symmetry unit cell with an uneven k-mesh, as in a screening run over structures
        _case("triclinic-5-split", "random", "split", "build", (2, 1, 3), 0.37, centres=5, ortho=False, geometry=3),
        # a molecular unit cell of the same kind in the default FP64 form
        _case("triclinic-14-fp64", "random", "fp64", "build", (3, 2, 1), 0.41, centres=14, ortho=False, geometry=7),
        # the everyday solid: a cubic diamond-like cell, dense k-mesh, in the default and in the fast form
        _case("diamond-fp64", "diamond", "fp64", "build", (4, 4, 4), 0.4),
        _case("diamond-split", "diamond", "split", "build", (4, 4, 4), 0.4),
        # the same solid from an SCF program that keeps its matrices in pinned host memory
        _case("diamond-host", "diamond", "split", "host", (4, 4, 4), 0.4),
        # a surface slab with vacuum in the default form: many small G per line, 34 centres
        _case("slab-fp64", "slab", "fp64", "build", (3, 3, 1), 0.4, layers=4),
        # forces on that slab, one step of a geometry optimisation
        _case("slab-gradient", "slab", "split", "gradient", (3, 3, 1), 0.4, layers=4),
        # the largest system: a molecular crystal with two spin densities, in the fastest form it has
        _case("crystal-tensor", "rings", "tensor", "build", (2, 2, 2), 0.5, ndens=2, rings=4),
        # the same with diffuse-diffuse pairs on the real-space grid, as an all-electron run classifies them
        _case("crystal-classified", "rings", "classified", "build", (2, 2, 2), 0.5, ndens=2, rings=4),
        # and with per-pair G cutoffs in the walks
        _case("crystal-cutoffs", "rings", "cutoffs", "build", (2, 2, 2), 0.5, ndens=2, rings=4),
        # an uneven set of low-symmetry cells built together in each iteration, replayed as one graph
        _case("batch-16-split", "cells", "split", "batch", (0, 0, 0), 0.0, cells=16),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    geometry = rng.randrange(1, 1 << 20)
    omega = round(rng.uniform(0.3, 0.5), 3)
    k = tuple(rng.randint(1, 3) for _ in range(3))
    ndens = rng.choice((1, 1, 2))
    kind = rng.choice(("fp64", "split", "tensor", "classified", "cutoffs", "gradient", "host", "batch", "rings",
                       "diamond"))
    c = None
    if kind == "fp64":
        c = _case("", "random", "fp64", "build", k, omega, ndens, centres=_spread(rng, 2, 14),
                  ortho=rng.random() < 0.4)
    elif kind in ("split", "cutoffs", "host"):
        c = _case("", "random", "cutoffs" if kind == "cutoffs" else "split", "host" if kind == "host" else "build", k,
                  omega, ndens, centres=_spread(rng, 2, 24), ortho=rng.random() < 0.4)
    elif kind in ("tensor", "classified"):
        c = _case("", "random", kind, "build", k, omega, ndens, centres=_spread(rng, 2, 24), ortho=True)
    elif kind == "gradient":
        c = _case("", "random", rng.choice(("fp64", "split", "split")), "gradient", k, omega, 1,
                  centres=_spread(rng, 2, 10), ortho=rng.random() < 0.4)
    elif kind == "batch":
        c = _case("", "cells", "split", "batch", (0, 0, 0), 0.0, cells=rng.randint(2, 14))
    elif kind == "rings":
        c = _case("", "rings", rng.choice(("tensor", "classified", "cutoffs")), "build",
                  tuple(rng.randint(1, 2) for _ in range(3)), omega, rng.choice((1, 2)), rings=rng.randint(1, 3))
    else:
        c = _case("", "diamond", rng.choice(("fp64", "split", "tensor")), rng.choice(("build", "host")),
                  tuple(rng.randint(1, 4) for _ in range(3)), omega, ndens)
    c["geometry"] = geometry
    del c["name"]
    return c


# ---- the systems ---------------------------------------------------------------


def _cell_matrix(rng, ortho, volume):
    """A random cell of at least `volume`: edges 6-16 bohr, angles 60-120 degrees unless orthorhombic."""
    while True:
        a, b, c = rng.uniform(6.0, 16.0, 3)
        if ortho:
            A = np.diag([a, b, c])
        else:
            al, be, ga = np.radians(rng.uniform(60.0, 120.0, 3))
            cx, cy = math.cos(be), (math.cos(al) - math.cos(be) * math.cos(ga)) / math.sin(ga)
            cz2 = 1.0 - cx * cx - cy * cy
            if cz2 < 0.1:
                continue
            A = np.array([[a, 0, 0], [b * math.cos(ga), b * math.sin(ga), 0], [c * cx, c * cy, c * math.sqrt(cz2)]])
        if abs(np.linalg.det(A)) >= volume:
            return A


def _scattered(rng, A, n):
    """n fractional sites at least 1.5 bohr apart (nearest images of the rounded difference)."""
    sites = []
    while len(sites) < n:
        f = rng.uniform(0, 1, 3)
        d = np.array(sites).reshape(-1, 3) - f
        d -= np.round(d)
        if not len(sites) or np.linalg.norm(d @ A, axis=1).min() >= 1.5:
            sites.append(f)
    return np.array(sites) @ A


class System:
    """One cell: lattice rows A, centres xyz, element of each centre, k-mesh and range-separation parameter."""

    def __init__(self, A, xyz, kinds, kmesh, omega):
        self.A, self.xyz, self.kinds = np.asarray(A, float), np.asarray(xyz, float), list(kinds)
        self.kmesh, self.omega, self.cartesian = tuple(int(v) for v in kmesh), float(omega), "X" in kinds
        self.shells = []  # (centre, l, exponent)
        for i, kind in enumerate(self.kinds):
            for l, lo, hi, n in BASIS[kind]:
                ratio = (hi / lo) ** (1.0 / max(1, n - 1))
                self.shells += [(i, l, lo * ratio ** q) for q in range(n)]
        self.widths = [(l + 1) * (l + 2) // 2 if self.cartesian else 2 * l + 1 for _, l, _ in self.shells]
        self.nao, self.nk = sum(self.widths), int(np.prod(self.kmesh))


def _random_system(rng, centres, ortho, kmesh, omega):
    A = _cell_matrix(rng, ortho, 40.0 * centres)
    xyz = _scattered(rng, A, centres)
    return System(A, xyz, rng.choice(["H", "C", "O", "Mg"], size=centres), kmesh, omega)


def _systems(case):
    """The cells of a case (one, or several for a batch)."""
    rng = np.random.default_rng(case["geometry"])
    kmesh, omega = (case["k1"], case["k2"], case["k3"]), case["omega"]
    kind = case["system"]
    if kind == "dimer":
        return [System(np.eye(3) * 8.0, [[0, 0, 0], [1.4, 0, 0]], ["X", "X"], kmesh, omega)]
    if kind == "random":
        return [_random_system(rng, case["centres"], case["ortho"], kmesh, omega)]
    if kind == "cells":
        return [_random_system(rng, int(rng.integers(2, 25)), False, rng.integers(1, 4, 3),
                               float(rng.uniform(0.3, 0.5))) for _ in range(case["cells"])]
    if kind == "diamond":
        A = np.eye(3) * 6.74
        fcc = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
        return [System(A, np.vstack([fcc, fcc + 0.25]) @ A, ["C"] * 8, kmesh, omega)]
    if kind == "rings":
        A = np.diag([14.0, 17.8, 12.9])
        sites = (np.array([[0, 0, 0], [.5, .5, 0], [0, .5, .5], [.5, 0, .5]]) @ A)[:case["rings"]]
        ang = np.arange(6) * (math.pi / 3.0)
        ring = np.stack([np.cos(ang), np.sin(ang), np.zeros(6)], axis=1)
        cs, hs = [], []
        for s in sites:
            Q, R = np.linalg.qr(rng.normal(size=(3, 3)))
            Q = Q * np.sign(np.diag(R))
            cs.append(2.64 * ring @ Q.T + s)
            hs.append((2.64 + 2.05) * ring @ Q.T + s)
        n = 6 * len(sites)
        return [System(A, np.vstack(cs + hs), ["C"] * n + ["H"] * n, kmesh, omega)]
    if kind == "slab":  # rock-salt (001) layers, 8 sites each, and a CO molecule above the top one
        d, layers = 3.98, case["layers"]
        A = np.diag([2.0 * math.sqrt(2.0) * d] * 2 + [(layers - 1) * d + 20.0])
        xyz, kinds = [], []
        for z in range(layers):
            for i in range(4):
                for j in range(4):
                    if (i + j) % 2 == 0:
                        xyz.append([i * A[0, 0] / 4, j * A[1, 1] / 4, z * d])
                        kinds.append("Mg" if (i + z) % 2 == 0 else "O")
        top = [p for p, q in zip(xyz, kinds) if q == "Mg" and p[2] == (layers - 1) * d][0]
        xyz += [[top[0], top[1], top[2] + 4.3], [top[0], top[1], top[2] + 4.3 + 2.13]]
        return [System(A, xyz, kinds + ["C", "O"], kmesh, omega)]
    raise ValueError(kind)


def _partner(kmesh):
    """Index of -k for every k of the Gamma-centred mesh."""
    g = np.indices(kmesh).reshape(3, -1).T
    m = (-g) % np.array(kmesh)
    return (m[:, 0] * kmesh[1] + m[:, 1]) * kmesh[2] + m[:, 2]


def _densities(s, ndens, seed, device):
    """D^k = C C^dagger of random occupied orbitals, Hermitian, with D^{-k} = conj D^k."""
    gen = torch.Generator(device=device).manual_seed(int(seed))
    nocc, partner = max(1, s.nao // 12), _partner(s.kmesh)
    pk = torch.from_numpy(partner).to(device)
    shape = (ndens, s.nk, s.nao, nocc)
    re, im = (torch.randn(shape, dtype=torch.float64, device=device, generator=gen) * 0.35 for _ in range(2))
    C = torch.complex(re, im)
    C = torch.where((torch.arange(s.nk, device=device) <= pk).view(1, -1, 1, 1), C, C[:, pk].conj())
    self_conj = (torch.arange(s.nk, device=device) == pk).view(1, -1, 1, 1)
    C = torch.where(self_conj, (C.real * math.sqrt(2.0)).to(C.dtype), C)
    D = C @ C.mH
    D = 0.5 * (D + D.mH)
    D = torch.where((torch.arange(s.nk, device=device) <= pk).view(1, -1, 1, 1), D, D[:, pk].conj())
    return torch.where(self_conj, D.real.to(D.dtype), D).contiguous()


# ---- the calls -------------------------------------------------------------------


def prepare(case, seed):
    from paper_2509_16460_gb300 import ftcj
    from paper_2509_16460_gb300.workloads import Shell, Workload

    dev = torch.device("cuda")
    systems = _systems(case)

    def shells(s):
        return [Shell(c, l, not s.cartesian, np.array([e]), np.array([1.0])) for c, l, e in s.shells]

    form = case["form"]
    precision = ftcj.FTCJ_PREC_FP64 if form == "fp64" else ftcj.FTCJ_PREC_SPLIT
    Dk = [_densities(s, case["ndens"], seed * 64 + i, dev) for i, s in enumerate(systems)]
    if case["call"] == "batch":
        batch = ftcj.Batch([Workload("cell", s.A, s.xyz, shells(s), s.kmesh, s.omega, D, EPS_G, 0.0, PAIR_THRESH)
                            for s, D in zip(systems, Dk)], precision=precision)
        Jk, EJ = batch.outputs_like(Dk)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        batch.capture(Dk, Jk, EJ, stream)
        return {"call": "batch", "batch": batch, "Dk": Dk, "Jk": Jk, "EJ": EJ}
    s, D = systems[0], Dk[0]
    plan = ftcj.Plan(s.A, s.xyz, shells(s), s.kmesh, s.omega, eps_g=EPS_G, pair_thresh=PAIR_THRESH,
                     precision=precision, max_dens=case["ndens"],
                     pair_gcut_eps=CUTOFF_EPS if form == "cutoffs" else 0.0,
                     contraction=ftcj.FTCJ_CONTRACT_TC if form in ("tensor", "classified") else
                     ftcj.FTCJ_CONTRACT_WALK, classify=form == "classified")
    state = {"call": case["call"], "plan": plan}
    if case["call"] == "host":
        state["Dk"] = torch.empty(D.shape, dtype=D.dtype, pin_memory=True).copy_(D)
        state["Jk"] = torch.empty(D.shape, dtype=D.dtype, pin_memory=True)
        state["EJ"] = torch.empty(case["ndens"], dtype=torch.float64, pin_memory=True)
    elif case["call"] == "gradient":
        state["Dk"] = D
    else:
        state["Dk"], state["Jk"] = D, torch.empty_like(D)
        state["EJ"] = torch.empty(case["ndens"], dtype=torch.float64, device=dev)
    return state


def run(state):
    call = state["call"]
    if call == "batch":
        state["batch"].replay()
        return {"Jk": state["Jk"], "EJ": state["EJ"]}
    if call == "host":
        Jk, EJ = state["plan"].jbuild_host(state["Dk"], state["Jk"], state["EJ"])
        return {"Jk": Jk, "EJ": EJ}
    if call == "gradient":
        EJ, grad = state["plan"].grad(state["Dk"])
        return {"EJ": EJ, "grad": grad}
    Jk, EJ = state["plan"].jbuild(state["Dk"], state["Jk"], state["EJ"])
    return {"Jk": Jk, "EJ": EJ}


# ---- pairs and the G sphere --------------------------------------------------------


def _half_sphere(s, dev):
    """Half of the reciprocal vectors with 0 < |G| < G_cut, Cartesian."""
    B = 2.0 * math.pi * np.linalg.inv(s.A).T
    gcut = 2.0 * s.omega * math.sqrt(math.log(1.0 / EPS_G))
    top = [int(gcut * np.linalg.norm(a) / (2.0 * math.pi)) + 1 for a in s.A]
    n = np.stack(np.meshgrid(*(np.arange(-t, t + 1) for t in top), indexing="ij"), -1).reshape(-1, 3)
    n = n[(n[:, 2] > 0) | ((n[:, 2] == 0) & ((n[:, 1] > 0) | ((n[:, 1] == 0) & (n[:, 0] > 0))))]
    g2 = np.einsum("ni,ij,nj->n", n, B @ B.T, n)
    return torch.from_numpy(n[g2 < gcut * gcut] @ B).to(dev)


def _pairs(s, dev):
    """Ordered screened primitive-shell pairs (a in the home cell, b in cell L): index arrays a, b and L."""
    alpha = torch.tensor([e for _, _, e in s.shells], dtype=torch.float64, device=dev)
    cen = torch.tensor([c for c, _, _ in s.shells], device=dev)
    X = torch.from_numpy(s.xyz).to(dev)[cen]
    p = alpha[:, None] + alpha[None, :]
    mu = alpha[:, None] * alpha[None, :] / p
    r2 = (1.5 * torch.log(2.0 * torch.sqrt(alpha[:, None] * alpha[None, :]) / p) - math.log(PAIR_THRESH)) / mu
    A = torch.from_numpy(s.A).to(dev)
    reach = float(r2.max().clamp_min(0).sqrt())
    diff = X[:, None] - X[None, :]
    heights = 1.0 / np.linalg.norm(np.linalg.inv(s.A), axis=0)
    frac = np.abs((s.xyz[:, None] - s.xyz[None]) @ np.linalg.inv(s.A)).reshape(-1, 3).max(0)
    top = [int(math.ceil(reach / h + f)) for h, f in zip(heights, frac)]
    ia, ib, il = [], [], []
    for l1 in range(-top[0], top[0] + 1):
        for l2 in range(-top[1], top[1] + 1):
            for l3 in range(-top[2], top[2] + 1):
                L = torch.tensor([l1, l2, l3], dtype=torch.float64, device=dev)
                a, b = torch.nonzero(((diff - L @ A) ** 2).sum(-1) < r2, as_tuple=True)
                ia.append(a)
                ib.append(b)
                il.append(torch.tensor([[l1, l2, l3]], device=dev).expand(len(a), 3))
    return torch.cat(ia), torch.cat(ib), torch.cat(il)


def work(case):
    """Two passes of 4L + 14 flops (L = l_a + l_b: Horner steps, prefactor, accumulation) for a quarter of the
    ordered pair x G products (+-G and mirror symmetry), D^k read and J^k (or the forces) written."""
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    flops = nbytes = 0.0
    for s in _systems(case):
        a, b, L = _pairs(s, dev)
        ls = torch.tensor([l for _, l, _ in s.shells], dtype=torch.float64, device=dev)
        g = _half_sphere(s, dev).shape[0]
        per_point = 4.0 * (ls[a] + ls[b]) + 14.0
        share = torch.full_like(per_point, 1.0)
        if case["form"] == "cutoffs":  # points where e^{-G^2 (1/4w^2 + 1/4p)} K is above the threshold, by volume
            al = torch.tensor([e for _, _, e in s.shells], dtype=torch.float64, device=dev)
            p = al[a] + al[b]
            reach = -math.log(CUTOFF_EPS) / (0.25 / s.omega ** 2 + 0.25 / p)
            share = (reach.sqrt() / (2.0 * s.omega * math.sqrt(-math.log(EPS_G)))).clamp_max(1.0) ** 3
        flops += 2.0 * case["ndens"] * float((per_point * share).sum()) / 2.0 * g
        matrix = 16.0 * case["ndens"] * s.nk * s.nao ** 2
        nbytes += matrix + (24.0 * len(s.xyz) if case["call"] == "gradient" else matrix)
    return {"bytes": nbytes, "flops": flops}


# ---- the independent FP64 evaluation -------------------------------------------------


def _monomials(l):
    return [(i, j, l - i - j) for i in range(l, -1, -1) for j in range(l - i, -1, -1)]


def _to_cartesian(l, cartesian, dev):
    """Rows: basis functions of a shell over its Cartesian monomials, per unit (2a/pi)^{3/4} (4a)^{l/2}."""
    mono = _monomials(l)
    if cartesian:
        fact = [math.sqrt(math.prod(max(1, math.prod(range(2 * n - 1, 0, -2))) for n in m)) for m in mono]
        T = np.diag([1.0 / f for f in fact])
    elif l < 2:
        T = np.eye(len(mono))
    else:  # xy, yz, z^2, xz, x^2 - y^2 over xx, xy, xz, yy, yz, zz
        r = 1.0 / (2.0 * math.sqrt(3.0))
        T = np.array([[0, 1, 0, 0, 0, 0], [0, 0, 0, 0, 1, 0], [-r, 0, 0, -r, 0, 2 * r], [0, 0, 1, 0, 0, 0],
                      [0.5, 0, 0, -0.5, 0, 0]])
    return torch.from_numpy(T).to(dev)


def _pair_transforms(la, lb, A, B, alpha, beta, G):
    """(mu nu|G) of n primitive pairs over Cartesian monomials: yields ((ca, cb), [n, g] complex)."""
    p = alpha + beta
    P = (alpha[:, None] * A + beta[:, None] * B) / p[:, None]
    K = torch.exp(-alpha * beta / p * ((A - B) ** 2).sum(-1)) * (math.pi / p) ** 1.5
    norm = ((2 * alpha / math.pi) ** 0.75 * (4 * alpha) ** (la / 2) * (2 * beta / math.pi) ** 0.75 *
            (4 * beta) ** (lb / 2))
    head = torch.polar((K * norm)[:, None] * torch.exp(-(G * G).sum(-1)[None] / (4 * p[:, None])), -(P @ G.T))
    h = (0.5 / p)[:, None]
    f = []
    for x in range(3):
        iG = torch.complex(torch.zeros_like(G[:, x]), -G[:, x])[None] * h
        up_a, up_b = iG + (P - A)[:, x, None], iG + (P - B)[:, x, None]
        t = {(0, 0): None}  # None stands for 1
        for i in range(la + 1):
            for j in range(lb + 1):
                if i == j == 0:
                    continue
                ii, jj, up = (i - 1, j, up_a) if i else (i, j - 1, up_b)
                v = up if t[ii, jj] is None else up * t[ii, jj]
                for c, low in ((ii, (ii - 1, jj)), (jj, (ii, jj - 1))):
                    if c:
                        v = v + (c * h if t[low] is None else c * h * t[low])
                t[i, j] = v
        f.append(t)
    for ca, m in enumerate(_monomials(la)):
        for cb, q in enumerate(_monomials(lb)):
            v = head
            for x in range(3):
                w = f[x][m[x], q[x]]
                v = v if w is None else v * w
            yield (ca, cb), v


class _Exact:
    """Pairs of one system in blocks of one (l_a, l_b), with the steps of the build over them."""

    def __init__(self, s, dev, limit):
        self.s, self.dev = s, dev
        self.G = _half_sphere(s, dev)
        self.a, self.b, self.L = _pairs(s, dev)
        self.alpha = torch.tensor([e for _, _, e in s.shells], dtype=torch.float64, device=dev)
        self.cen = torch.tensor([c for c, _, _ in s.shells], device=dev)
        self.l = torch.tensor([l for _, l, _ in s.shells], device=dev)
        self.ao = torch.tensor(np.concatenate([[0], np.cumsum(s.widths)[:-1]]), device=dev)
        km = torch.tensor(s.kmesh, device=dev)
        n = self.L % km
        self.cell = (n[:, 0] * km[1] + n[:, 1]) * km[2] + n[:, 2]
        self.X = torch.from_numpy(s.xyz).to(dev)
        self.latt = torch.from_numpy(s.A).to(dev)
        self.T = [_to_cartesian(l, s.cartesian, dev) for l in range(3)]
        ng = self.G.shape[0]
        self.blocks = []
        for la in range(3):
            for lb in range(3):
                idx = torch.nonzero((self.l[self.a] == la) & (self.l[self.b] == lb)).ravel()
                if len(idx):
                    self.blocks += [(la, lb, i) for i in torch.split(idx, max(1, limit // max(1, ng)))]

    def phases(self):
        m = torch.from_numpy(np.indices(self.s.kmesh).reshape(3, -1).T.astype(float)).to(self.dev)
        return torch.polar(torch.ones(self.s.nk, self.s.nk, dtype=torch.float64, device=self.dev),
                           2.0 * math.pi * (m @ (m / torch.tensor(self.s.kmesh, device=self.dev)).T))

    def place(self, la, lb, i):
        """AO rows and columns of a block's functions, [n, wa, 1] and [n, 1, wb]."""
        wa, wb = self.T[la].shape[0], self.T[lb].shape[0]
        return (self.ao[self.a[i]][:, None, None] + torch.arange(wa, device=self.dev)[None, :, None],
                self.ao[self.b[i]][:, None, None] + torch.arange(wb, device=self.dev)[None, None, :])

    def transforms(self, la, lb, i, X):
        A = X[self.cen[self.a[i]]]
        B = X[self.cen[self.b[i]]] + self.L[i].double() @ self.latt
        return _pair_transforms(la, lb, A, B, self.alpha[self.a[i]], self.alpha[self.b[i]], self.G)

    def block_density(self, D0n, la, lb, i):
        r, c = self.place(la, lb, i)
        D = D0n[:, self.cell[i][:, None, None], r, c]
        return torch.einsum("dnij,ix,jy->dnxy", D, self.T[la], self.T[lb]).to(torch.complex128)

    def rho(self, D0n, keep):
        out = torch.zeros(D0n.shape[0], self.G.shape[0], dtype=torch.complex128, device=self.dev)
        for la, lb, i in self.blocks:
            i = i[keep[i]]
            if len(i):
                D = self.block_density(D0n, la, lb, i)
                for (ca, cb), v in self.transforms(la, lb, i, self.X):
                    out += D[:, :, ca, cb] @ v
        return out

    def back(self, W, keep, J0n):
        for la, lb, i in self.blocks:
            i = i[keep[i]]
            if len(i):
                wa, wb = self.T[la].shape[1], self.T[lb].shape[1]
                J = torch.zeros(W.shape[0], len(i), wa, wb, dtype=torch.float64, device=self.dev)
                for (ca, cb), v in self.transforms(la, lb, i, self.X):
                    J[:, :, ca, cb] = (v @ W.T).real.T
                J = torch.einsum("dnxy,ix,jy->dnij", J, self.T[la], self.T[lb])
                r, c = self.place(la, lb, i)
                flat = ((self.cell[i][:, None, None] * self.s.nao + r) * self.s.nao + c).reshape(-1)
                J0n.view(W.shape[0], -1).index_add_(1, flat, J.reshape(W.shape[0], -1))

    def gradient(self, D0n, W):
        """dE_J/dR with W = 2 v conj(rho) held: the derivative of Re sum_G W rho, density by density."""
        out = torch.zeros(D0n.shape[0], len(self.s.xyz), 3, dtype=torch.float64, device=self.dev)
        for la, lb, i in self.blocks:
            D = self.block_density(D0n, la, lb, i)
            for d in range(D0n.shape[0]):
                X = self.X.clone().requires_grad_(True)
                e = 0.0
                for (ca, cb), v in self.transforms(la, lb, i, X):
                    e = e + (D[d, :, ca, cb].real * (v @ W[d]).real).sum()
                out[d] += torch.autograd.grad(e, X)[0]
        return out


def _exact_one(case, s, Dk, dev):
    e = _Exact(s, dev, 2_000_000 if case["call"] == "gradient" else 12_000_000)
    F = e.phases()
    D0n = torch.einsum("nk,dkab->dnab", F.conj() / s.nk, Dk).real.contiguous()
    g2 = (e.G * e.G).sum(-1)
    full = 4.0 * math.pi / (abs(np.linalg.det(s.A)) * g2)
    long_range = full * torch.exp(-g2 / (4.0 * s.omega ** 2))
    every = torch.ones(len(e.a), dtype=torch.bool, device=dev)
    J0n = torch.zeros_like(D0n)
    if case["form"] == "classified":  # pairs of two diffuse primitives take the full kernel in every integral
        diffuse = e.alpha < 0.5 * s.omega ** 2
        dd = diffuse[e.a] & diffuse[e.b]
        rc, rd = e.rho(D0n, ~dd), e.rho(D0n, dd)
        EJ = (long_range * rc.abs() ** 2 + full * (2.0 * (rc * rd.conj()).real + rd.abs() ** 2)).sum(-1)
        e.back(2.0 * (long_range * rc.conj() + full * rd.conj()), ~dd, J0n)
        e.back(2.0 * full * (rc + rd).conj(), dd, J0n)
    else:
        rho = e.rho(D0n, every)
        EJ = (long_range * rho.abs() ** 2).sum(-1)
        W = 2.0 * long_range * rho.conj()
        if case["call"] == "gradient":
            return None, EJ, e.gradient(D0n, W)
        e.back(W, every, J0n)
    return torch.einsum("kn,dnab->dkab", F, J0n.to(torch.complex128)), EJ, None


def exact(case, seed):
    """The case's outputs in FP64, by definition (cutoffs: of the whole sphere, which they approximate)."""
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    systems = _systems(case)
    got = [_exact_one(case, s, _densities(s, case["ndens"], seed * 64 + i, dev), dev) for i, s in enumerate(systems)]
    if case["call"] == "batch":
        return {"Jk": [g[0] for g in got], "EJ": [g[1] for g in got]}
    Jk, EJ, grad = got[0]
    return {"EJ": EJ, "grad": grad} if case["call"] == "gradient" else {"Jk": Jk, "EJ": EJ}
