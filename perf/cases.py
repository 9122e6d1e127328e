"""The library's work as its users call it, in sizes from the smallest molecule to the largest system.

A case is a molecule (or a batch of them) with the settings it is run at.  Four kinds:

* ``step``: one MD step through ``sim_step_host``, the call of a program that keeps positions and
  velocities on the host (an integrator, a sampler, a driver of several replicas); the electronic
  state stays on the device.  ``graph`` steps through the captured CUDA graphs, as the server does.
  With ``read`` the program also takes the density matrix and the orbital energies of the step.
* ``point``: a ground state from nothing (``sim_create`` with its SCF), energy, forces and density
  taken, the handle given back: single points, and what every new trajectory of the server begins with.
* ``batch``: one step of many molecules at once (``sim_batch_run``), thermostatted.
* ``product``: the allocation-free product of two small matrices in device memory.

Molecules are alkane-like strands with N and O in the chain (odd basis sizes, hydrogen and heavy
atoms mixed) and clusters of C60 cages (60 to 840 atoms), parameters a synthetic H/C/N/O table.

``SIM_PREC_FP64`` results are kept in double precision.  ``SIM_PREC_MIXED`` multiplies matrices cut
into 24 and 32 bits, and a program that asks for it keeps its trajectory in single precision, as
trajectory files do; energies come as plain numbers either way.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2303_00689_gb300 as kx

# raw parameters, rows H, C, N, O: Z, orbitals, principal quantum number, core charge, mass, U_ss, U_pp,
# zeta_s, zeta_p, beta_s, beta_p, G_ss, G_sp, G_pp, G_p2, H_sp, alpha, two core-core Gaussians (a, b, c)
TABLE = np.array([
    [1, 1, 1, 1, 1.008, -12.76152, 0, 1.25153, 0, -6.61451, 0, 13.50967, 0, 0, 0, 0, 2.56038,
     0.2443, 5.90034, 1.58747, 0.17008, 4.08369, 1.26967],
    [6, 4, 2, 4, 12.011, -52.56881, -39.8196, 1.84753, 1.66513, -15.74281, -7.54201, 12.40523, 11.93765,
     10.76134, 9.80223, 2.39221, 2.50305, 0.19621, 7.00013, 2.15192, 0.15893, 4.07955, 1.57071],
    [7, 4, 2, 5, 14.007, -71.38707, -57.97188, 2.24802, 2.02899, -20.73632, -18.1144, 13.15281, 12.08377,
     11.97212, 10.20138, 2.78564, 2.91039, 0.16749, 6.33152, 1.64793, 0.16222, 5.21842, 2.06895],
    [8, 4, 2, 6, 15.999, -97.48555, -77.85125, 2.85004, 2.68388, -28.51237, -28.38616, 15.42013, 14.71134,
     14.36776, 12.60403, 3.98746, 3.18533, 0.26965, 5.85744, 1.81212, 0.30098, 5.32859, 2.0978]])
ROW = {1: 0, 6: 1, 7: 2, 8: 3}
KB, ACCEL, E2, BOHR = 8.617333262e-5, 9.648533212e-3, 14.399645, 0.52917721090
DT = 0.5          # fs
SCF_STEPS = 14    # linear mixing brings the density to about 1e-4 and better, what dynamics starts from

# Work limits of a drawn case: basis functions, by precision
MAX_N = {"fp64": 1680, "mixed": 3360}


def listed():
    def step(name, mol, size, precision, m=4, Te=1000.0, graph=False, read=False):
        return dict(name=name, kind="step", mol=mol, size=size, precision=precision, m=m, Te=Te, graph=graph,
                    read=read)

    return [
        # a serving process's inner product, one launch deep
        dict(name="product_250", kind="product", size=250, terms=10),
        # the plain method on a molecule of 14 atoms, everything read back: latency and launches
        step("strand_4_fp64", "strand", 4, "fp64", read=True),
        # a molecule of the organic batch on its own (62 atoms, 131 basis functions), replayed from graphs
        step("strand_23_mixed_graph", "strand", 23, "mixed", graph=True),
        # a larger organic system in the default precision (274 atoms)
        step("strand_100_fp64", "strand", 100, "fp64", read=True),
        # one cage: the smallest request of the server; analysis reads density and orbital energies
        step("c60_mixed_read", "cages", 1, "mixed", Te=5000.0, read=True),
        # two cages: the energy-conservation runs
        step("c120_mixed_graph", "cages", 2, "mixed", Te=5000.0, graph=True),
        # a mid-size request of the server (420 atoms)
        step("c420_mixed_graph", "cages", 7, "mixed", Te=5000.0, graph=True),
        # the same system in double precision
        step("c420_fp64", "cages", 7, "fp64", Te=5000.0),
        # the largest system, rank 6
        step("c840_mixed", "cages", 14, "mixed", m=6, Te=3000.0),
        # single points
        dict(name="c60_point", kind="point", mol="cages", size=1, precision="mixed", m=4, Te=5000.0),
        # batches of cages of 60 to 180 atoms, Langevin at 300 K
        dict(name="batch_16", kind="batch", mol="cages", size=16, precision="mixed", m=4, Te=5000.0),
    ]


def draw(rng):
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step"] * 8 + ["point", "batch", "product"])
    if kind == "product":
        return dict(kind=kind, size=between(2, 256), terms=rng.choice([1, 3, 6, 10]))
    if kind == "batch":
        return dict(kind=kind, mol="cages", size=between(2, 16), precision="mixed", m=rng.randint(2, 6), Te=5000.0)
    precision = rng.choice(["fp64", "mixed", "mixed"])
    if kind == "point":
        mol, size = rng.choice([("strand", between(2, 60)), ("cages", between(1, 3))])
    elif rng.random() < 0.5:
        mol, size = "strand", between(2, 120 if precision == "fp64" else 250)
    else:
        mol, size = "cages", between(1, MAX_N[precision] // 240)
    case = dict(kind=kind, mol=mol, size=size, precision=precision, m=rng.randint(2, 6 if precision == "mixed" else 4),
                Te=1000.0 if mol == "strand" else rng.choice([3000.0, 5000.0]))
    if kind == "step":
        case.update(graph=rng.random() < 0.5, read=size <= (100 if mol == "strand" else 2) and rng.random() < 0.5)
    return case


# ---- molecules ------------------------------------------------------------------------------------------
def strand(heavy):
    """Zigzag strands of at most 24 heavy atoms side by side, N and O at fixed places in the chain, H saturated."""
    Z, R = [], []
    dx, dy = 1.53 * math.sqrt(2.0 / 3.0), 1.53 * math.sqrt(1.0 / 3.0)
    for s, first in enumerate(range(0, heavy, 24)):
        k = min(24, heavy - first)
        at = np.array([0.0, 5.0 * (s % 4), 5.0 * (s // 4)])
        for i in range(k):
            up = 1.0 if i % 2 else -1.0
            z = 8 if i % 7 == 3 and i < k - 1 else 7 if i % 7 == 5 and i < k - 1 else 6
            p = at + np.array([i * dx, 0.5 * up * dy, 0.0])
            Z.append(z)
            R.append(p)
            out = [np.array([0.0, up * math.sqrt(1.0 / 3.0), w * math.sqrt(2.0 / 3.0)]) for w in (1.0, -1.0)]
            ends = [np.array([w * dx, -up * dy, 0.0]) / 1.53 for w in (-1.0, 1.0)]
            bonds = out[:{6: 2, 7: 1, 8: 0}[z]] + [e for e, end in zip(ends, (i == 0, i == k - 1)) if end]
            for b in bonds:
                Z.append(1)
                R.append(p + 1.09 * b)
    return np.array(Z, dtype=np.int32), np.array(R)


def cages(count, first=0):
    """C60 cages on a cubic grid 11.5 Angstrom apart."""
    g = (1.0 + 5.0 ** 0.5) / 2.0
    unit = set()
    for v in ((0.0, 1.0, 3 * g), (1.0, 2.0 + g, 2 * g), (g, 2.0, 2 * g + 1.0)):
        for sign in np.ndindex(2, 2, 2):
            w = [x * (1 - 2 * s) for x, s in zip(v, sign)]
            unit.update(tuple(round(w[(k + j) % 3], 12) + 0.0 for j in range(3)) for k in range(3))
    unit = np.array(sorted(unit)) * (1.60 / 2.0)
    side = math.ceil(count ** (1.0 / 3.0) - 1e-9)
    R = [unit + 11.5 * np.array([c % side, c // side % side, c // side ** 2]) for c in range(count)]
    return np.full(60 * count, 6, dtype=np.int32), np.concatenate(R)


def molecule(mol, size, seed):
    """Atoms, positions (0.02 Angstrom off the ideal ones) and Maxwell-Boltzmann velocities at 300 K."""
    Z, R = (strand if mol == "strand" else cages)(size)
    rng = np.random.default_rng([seed, len(Z)])
    R = R + 0.02 * rng.normal(size=R.shape)
    mass = TABLE[[ROW[int(z)] for z in Z], 4]
    V = rng.normal(size=R.shape) * np.sqrt(KB * 300.0 * ACCEL / mass)[:, None]
    V -= (mass[:, None] * V).sum(axis=0) / mass.sum()
    return Z, R, V


# ---- what a program holds -------------------------------------------------------------------------------
class Handles:
    """Handles (and the batch over them), given back with this object."""

    def __init__(self):
        self.h, self.batch = [], None

    def __del__(self):
        if self.batch:
            kx.sim_batch_destroy(self.batch)
        for h in self.h:
            kx.sim_destroy(h)


def config(case, **more):
    return kx.sim_config_default(
        Te=case["Te"], dt=DT, m_max=case["m"], m_min=case["m"],
        precision=kx.SIM_PREC_FP64 if case["precision"] == "fp64" else kx.SIM_PREC_MIXED,
        scf_tol=1e-12, scf_max=SCF_STEPS, scf_accept=1, **more)


def single(case):
    """How the program keeps arrays (see the top of this file)."""
    return np.float32 if case["precision"] == "mixed" else np.float64


def batch_members(case, seed):
    return [molecule("cages", 1 + i % 3, seed + 1000 * i) for i in range(case["size"])]


def prepare(case, seed):
    if case["kind"] == "product":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        n = case["size"]
        A, B = (torch.linalg.qr(torch.randn(n, n, generator=gen, device="cuda", dtype=torch.float64))[0].contiguous()
                for _ in range(2))
        return dict(case=case, A=A, B=B, C=torch.empty_like(A))
    table = kx.param_table(TABLE)
    if case["kind"] == "point":
        Z, R, V = molecule(case["mol"], case["size"], seed)
        return dict(case=case, cfg=config(case), table=table, Z=Z, R=R)
    own = Handles()
    if case["kind"] == "batch":
        sizes = []
        for i, (Z, R, V) in enumerate(batch_members(case, seed)):
            cfg = config(case, langevin_gamma=0.01, langevin_T=300.0, langevin_seed=seed + i)
            own.h.append(kx.sim_create(cfg, table, Z, R, V=V))
            sizes.append(len(Z))
        own.batch = kx.sim_batch_create(own.h)
        return dict(case=case, own=own, sizes=sizes)
    Z, R, V = molecule(case["mol"], case["size"], seed)
    own.h.append(kx.sim_create(config(case), table, Z, R, V=V))
    if case["graph"]:
        kx.sim_enable_graphs(own.h[0])
    return dict(case=case, own=own, R=R, V=V, out=[np.empty_like(R) for _ in range(3)], record=kx.sim_step_result())


def energies(r):
    return dict(E_kin=r["E_kin"], U=r["U"], E_tot=r["E_tot"], rank=r["rank"])


def run(state):
    case = state["case"]
    if case["kind"] == "product":
        rc = kx.sim_tc_gemm_noalloc(case["size"], state["A"].data_ptr(), state["B"].data_ptr(), case["terms"], False,
                                    state["C"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != kx.SIM_OK:
            raise RuntimeError("sim_tc_gemm_noalloc: status %d" % rc)
        return state["C"]
    as_kept = single(case)
    if case["kind"] == "point":
        h = kx.sim_create(state["cfg"], state["table"], state["Z"], state["R"])
        try:
            _, _, F, D = kx.sim_get_state(h, len(state["Z"]))
            r = kx.sim_last_result(h)
            return dict(F=F.astype(as_kept), D=D.astype(as_kept), U=r["U"])
        finally:
            kx.sim_destroy(h)
    if case["kind"] == "batch":
        kx.sim_batch_run(state["own"].batch, 1)
        out = []
        for h, natoms in zip(state["own"].h, state["sizes"]):
            R, V, F = (np.empty((natoms, 3)) for _ in range(3))
            rc = kx.lib().sim_get_state(h, *(a.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for a in (R, V, F)), None)
            if rc != kx.SIM_OK:
                raise kx.SimError(rc, kx.sim_last_error())
            out.append((R, V, F, energies(kx.sim_last_result(h))))
        return dict(R=np.concatenate([o[0] for o in out]).astype(as_kept),
                    V=np.concatenate([o[1] for o in out]).astype(as_kept),
                    F=np.concatenate([o[2] for o in out]).astype(as_kept),
                    E_tot=np.array([o[3]["E_tot"] for o in out]).astype(as_kept),
                    U=np.array([o[3]["U"] for o in out]).astype(as_kept))
    h, rec = state["own"].h[0], state["record"]
    kx.sim_step_host(h, state["R"], state["V"], *state["out"], rec)
    R, V, F = (a.astype(as_kept) for a in state["out"])
    answer = dict(R=R, V=V, F=F, E=dict(E_kin=rec.E_kin, U=rec.U, E_tot=rec.E_tot, rank=rec.rank))
    if case["read"]:
        answer["D"] = kx.sim_get_state(h, len(R))[3].astype(as_kept)
        answer["eps"] = kx.sim_get_vector(h, 0)
    return answer


# ---- bytes and operations of one pass -------------------------------------------------------------------
def evaluation(N, n, m):
    """One evaluation: eigenpairs (4/3 n^3 + 2 n^3), density (n^3), m responses of 6 n^3, 425 + 1100 multiply-adds a
    pair; the pair blocks and the matrices F, D0, X and its history once."""
    pairs = N * (N - 1) // 2
    return dict(bytes=8.0 * (467.0 * pairs + (12.0 + 2.0 * m) * n * n),
                flops=(13.0 / 3.0 + 6.0 * m) * float(n) ** 3 + 2.0 * (425.0 * (m + 1) + 1100.0) * pairs)


def work(case):
    if case["kind"] == "product":
        return dict(bytes=24.0 * case["size"] ** 2, flops=2.0 * case["terms"] * case["size"] ** 3)

    def of(mol, size):
        Z, _ = (strand if mol == "strand" else cages)(size)
        return len(Z), int(TABLE[[ROW[int(z)] for z in Z], 1].sum())

    if case["kind"] == "batch":
        each = [evaluation(*of("cages", 1 + i % 3), case["m"]) for i in range(case["size"])]
        return {k: sum(e[k] for e in each) for k in each[0]}
    N, n = of(case["mol"], case["size"])
    w = evaluation(N, n, case["m"])
    if case["kind"] == "point":
        one = evaluation(N, n, 0)
        w = {k: w[k] + SCF_STEPS * one[k] for k in w}
    return w


# ---- the same in 64 bits, plain torch --------------------------------------------------------------------
# orbital products on one atom, and the product of every orbital pair
PRODUCTS = [(0, 0), (0, 1), (0, 2), (0, 3), (1, 1), (2, 2), (3, 3), (1, 2), (1, 3), (2, 3)]
INDEX = [[next(i for i, p in enumerate(PRODUCTS) if p in ((a, b), (b, a))) for b in range(4)] for a in range(4)]
KAPPA, ORBITALS = 1.84, np.arange(4)


def root(fn):
    lo, hi = 1e-8, 1e3
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if fn(mid) > 0.0 else (lo, mid)
    return 0.5 * (lo + hi)


def derived(row):
    """Multipole lengths D1, D2 and additive terms rho_0, rho_1, rho_2 of one element."""
    gss, gpp, gp2, hsp, nq, zs, zp = row[11], row[13], row[14], row[15], row[2], row[7], row[8]
    r0 = E2 / (2.0 * gss)
    if row[1] == 1:
        return [0.0, 0.0, r0, r0, r0]
    D1 = (2 * nq + 1) * (4 * zs * zp) ** (nq + 0.5) / ((zs + zp) ** (2 * nq + 2) * math.sqrt(3.0)) * BOHR
    D2 = math.sqrt((4 * nq * nq + 6 * nq + 2) / 20.0) / zp * BOHR
    r1 = root(lambda r: 0.25 * E2 * (1 / r - 1 / math.sqrt(D1 * D1 + r * r)) - hsp)
    r2 = root(lambda r: 0.125 * E2 * (1 / r - 2 / math.sqrt(D2 * D2 + r * r) + 1 / math.sqrt(2 * D2 * D2 + r * r))
              - 0.5 * (gpp - gp2))
    return [D1, D2, r0, r1, r2]


class Reference:
    """NDDO energy, forces, density and Krylov kernel of one molecule in 64 bits, straight from the equations."""

    def __init__(self, Z, Te):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        f64 = dict(dtype=torch.float64, device=self.dev)
        rows = np.array([ROW[int(z)] for z in Z])
        self.N, self.par = len(Z), torch.tensor(TABLE[rows], **f64)
        self.der = torch.tensor(np.array([derived(r) for r in TABLE])[rows], **f64)
        self.has = torch.tensor((ORBITALS[None] < TABLE[rows, 1][:, None]).astype(float), **f64)      # N x 4
        self.orb = torch.nonzero(self.has.reshape(-1))[:, 0]
        self.n, self.nocc = len(self.orb), int(round(TABLE[rows, 3].sum())) // 2
        self.beta, self.kT = 1.0 / (KB * Te), KB * Te
        self.A, self.B = torch.triu_indices(self.N, self.N, 1, device=self.dev)
        self.U = torch.where(torch.arange(4, device=self.dev)[None] == 0, self.par[:, 5:6], self.par[:, 6:7]) * self.has
        self.bet = torch.where(torch.arange(4, device=self.dev)[None] == 0, self.par[:, 9:10], self.par[:, 10:11]) * self.has
        one = np.zeros((4, 4, 4, 4, 4))                                    # element, mu nu lam sig
        for e, r in enumerate(TABLE):
            gss, gsp, gpp, gp2, hsp = r[11:16]
            for (a, b, c, d) in np.ndindex(4, 4, 4, 4):
                if a == b and c == d:
                    one[e, a, b, c, d] = gss if a == c == 0 else gsp if 0 in (a, c) else gpp if a == c else gp2
                elif a != b and sorted((a, b)) == sorted((c, d)):
                    one[e, a, b, c, d] = hsp if 0 in (a, b) else 0.5 * (gpp - gp2)
            if r[1] == 1:
                one[e].reshape(-1)[1:] = 0.0
        self.one = torch.tensor(one[rows], **f64)

    def charges(self, at):
        """Charges q (10 x 4), places (pairs x 10 x 4 x 3) and additive terms (pairs x 10 x 4) in the pair's frame."""
        D1, D2, r = self.der[at, 0], self.der[at, 1], self.der[at, 2:5]
        q, where, kind = np.zeros((10, 4)), np.zeros((10, 4, 3, 2)), np.zeros((10, 4), dtype=int)
        for p, (a, b) in enumerate(PRODUCTS):
            if b == 0:
                q[p, 0] = 1.0
            elif a == 0:
                for i, s in enumerate((1, -1)):
                    q[p, i], kind[p, i], where[p, i, b - 1, 0] = 0.5 * s, 1, s
            elif a == b:
                q[p], kind[p, 1:] = (1.0, 0.25, 0.25, -0.5), 2
                where[p, 1, a - 1, 1], where[p, 2, a - 1, 1] = 2.0, -2.0
            else:
                for i, (s, t) in enumerate(((1, 1), (-1, -1), (1, -1), (-1, 1))):
                    q[p, i], kind[p, i] = 0.25 * s * t, 2
                    where[p, i, a - 1, 1], where[p, i, b - 1, 1] = s, t
        w = torch.tensor(where, dtype=torch.float64, device=self.dev)
        place = w[..., 0] * D1[:, None, None, None] + w[..., 1] * D2[:, None, None, None]
        return torch.tensor(q, dtype=torch.float64, device=self.dev), place, r[:, torch.tensor(kind, device=self.dev)]

    def overlaps(self, R, A, B):
        """ss, (s)(sigma), (sigma)(s), (sigma)(sigma), (pi)(pi) Slater overlaps, by quadrature that is exact for them:
        Gauss-Laguerre in xi (a polynomial times e^(-p xi)), 48-point Gauss-Legendre in eta."""
        f64 = dict(dtype=torch.float64, device=self.dev)
        gx, gw = (torch.tensor(v, **f64) for v in np.polynomial.laguerre.laggauss(12))
        ex, ew = (torch.tensor(v, **f64) for v in np.polynomial.legendre.leggauss(48))
        h = 0.5 * R / BOHR
        out = []
        for ka, kb in ((0, 0), (0, 1), (1, 0), (1, 1), (2, 2)):
            za, zb = self.par[A, 7 + min(ka, 1)], self.par[B, 7 + min(kb, 1)]
            na, nb = self.par[A, 2], self.par[B, 2]
            skip = ((za == 0) | (zb == 0))
            za, zb = torch.where(skip, torch.ones_like(za), za), torch.where(skip, torch.ones_like(zb), zb)
            p, q = h * (za + zb), h * (za - zb)
            xi = (1.0 + gx[None] / p[:, None])[:, :, None]
            eta = ex[None, None]
            ra, rb = xi + eta, xi - eta
            # radial factors r^(n-1); a sigma p takes r^(n-2) (r cos theta), a pi p r^(n-2) (r sin theta)
            fa = torch.where((na == 1)[:, None, None], torch.ones_like(ra), ra) if ka == 0 else 1.0 + xi * eta
            fb = torch.where((nb == 1)[:, None, None], torch.ones_like(rb), rb) if kb == 0 else xi * eta - 1.0
            body = (xi * xi - 1.0) * (1.0 - eta * eta) if ka == 2 else fa * fb
            val = (xi * xi - eta * eta) * body * torch.exp(-q[:, None, None] * eta)
            s = torch.einsum("pxe,x,e->p", val, gw, ew) * torch.exp(-p) / p
            ang = [1.0 / math.sqrt(4 * math.pi), math.sqrt(3.0 / (4 * math.pi))]
            norm = [(2 * z) ** (k + 0.5) / torch.sqrt(torch.exp(torch.lgamma(2 * k + 1))) for z, k in ((za, na), (zb, nb))]
            phi = math.pi if ka == 2 else 2.0 * math.pi
            s = s * norm[0] * norm[1] * ang[min(ka, 1)] * ang[min(kb, 1)] * phi * h ** (na + nb + 1)
            out.append(torch.where(skip, torch.zeros_like(s), s))
        return out

    def blocks(self, R, A, B):
        """Two-centre integrals (p x 4 x 4 x 4 x 4), overlaps (p x 4 x 4) and core-core energies of pairs A, B."""
        d = R[B] - R[A]
        r = d.square().sum(1).sqrt()
        u = d / r[:, None]
        ref = torch.nn.functional.one_hot(u.detach().abs().argmin(1), 3).to(u)
        ex = ref - (ref * u).sum(1, keepdim=True) * u
        ex = ex / ex.square().sum(1, keepdim=True).sqrt()
        ey = torch.linalg.cross(u, ex)
        T = torch.nn.functional.pad(torch.stack([ex, ey, u], 2), (1, 0, 1, 0))
        T = T + torch.diag(torch.tensor([1.0, 0, 0, 0], dtype=T.dtype, device=T.device))
        (q, xa, ra), (_, xb, rb) = self.charges(A), self.charges(B)
        xb = xb + torch.nn.functional.pad(r[:, None], (2, 0))[:, None, None]
        dist = (xa[:, :, None, :, None] - xb[:, None, :, None, :]).square().sum(-1)
        dist = dist + (ra[:, :, None, :, None] + rb[:, None, :, None, :]).square()
        I = E2 * torch.einsum("pijab,ia,jb->pij", dist.rsqrt(), q, q)
        xy = torch.zeros(10, 10, dtype=torch.bool, device=self.dev)
        xy[7, 7] = True                        # (xy|xy) = [(xx|xx) - (xx|yy)] / 2: the frame's x is arbitrary
        I = torch.where(xy, (0.5 * (I[:, 4, 4] - I[:, 4, 5]))[:, None, None], I)
        gss = I[:, 0, 0]
        ix = torch.tensor(INDEX, device=self.dev)
        W = torch.einsum("pai,pbj,pijkl->pabkl", T, T, I[:, ix][:, :, :, ix])
        W = torch.einsum("pck,pdl,pabkl->pabcd", T, T, W)
        ma, mb = self.has[A], self.has[B]
        W = W * torch.einsum("pa,pb,pc,pd->pabcd", ma, ma, mb, mb)
        ss, s_s, sg_s, sgg, pipi = self.overlaps(r, A, B)
        zero = torch.zeros_like(ss)
        loc = torch.stack([ss, zero, zero, s_s, zero, pipi, zero, zero, zero, zero, pipi, zero, sg_s, zero, zero, sgg], 1)
        S = torch.einsum("pai,pij,pbj->pab", T, loc.reshape(-1, 4, 4), T) * ma[:, :, None] * mb[:, None]
        zz = self.par[A, 3] * self.par[B, 3]
        E = zz * gss * (1.0 + torch.exp(-self.par[A, 16] * r) + torch.exp(-self.par[B, 16] * r))
        for at in (A, B):
            for k in (17, 20):
                E = E + zz / r * self.par[at, k] * torch.exp(-self.par[at, k + 1] * (r - self.par[at, k + 2]) ** 2)
        return W, S, E

    def pad(self, M):
        P = torch.zeros(4 * self.N, 4 * self.N, dtype=M.dtype, device=M.device)
        P[self.orb[:, None], self.orb[None]] = M
        return P.reshape(self.N, 4, self.N, 4)

    def at(self, R):
        """Pair blocks at R, kept for the Fock builds there."""
        self.R = R
        parts = [self.blocks(R, A, B) for A, B in zip(self.A.split(4096), self.B.split(4096))]
        self.W, self.S, self.E = (torch.cat(v) for v in zip(*parts))
        N, A, B, zc = self.N, self.A, self.B, self.par[:, 3]
        diag = torch.diag_embed(self.U)
        diag = diag.index_add(0, A, -zc[B][:, None, None] * self.W[:, :, :, 0, 0])
        diag = diag.index_add(0, B, -zc[A][:, None, None] * self.W[:, 0, 0])
        self.h = self.assemble(diag, 0.5 * (self.bet[A][:, :, None] + self.bet[B][:, None]) * self.S)

    def assemble(self, diag, off):
        M = torch.zeros(self.N, self.N, 4, 4, dtype=off.dtype, device=off.device)
        M[self.A, self.B], M[self.B, self.A] = off, off.transpose(1, 2)
        M[range(self.N), range(self.N)] = diag
        return M.permute(0, 2, 1, 3).reshape(4 * self.N, -1)[self.orb[:, None], self.orb[None]]

    def G(self, P):
        Pb = self.pad(P).permute(0, 2, 1, 3)
        Pd = Pb[range(self.N), range(self.N)]
        diag = 2 * torch.einsum("amnls,als->amn", self.one, Pd) - torch.einsum("amlns,als->amn", self.one, Pd)
        diag = diag.index_add(0, self.A, 2 * torch.einsum("pmnls,pls->pmn", self.W, Pd[self.B]))
        diag = diag.index_add(0, self.B, 2 * torch.einsum("pmnls,pmn->pls", self.W, Pd[self.A]))
        return self.assemble(diag, -torch.einsum("pmnls,pns->pml", self.W, Pb[self.A, self.B]))

    def density(self, F):
        eps, Q = torch.linalg.eigh(F)
        lo, hi = eps[0] - 40 * self.kT, eps[-1] + 40 * self.kT
        for _ in range(200):
            mu = 0.5 * (lo + hi)
            over = self.occupations(eps, mu).sum() > self.nocc
            lo, hi = torch.where(over, lo, mu), torch.where(over, mu, hi)
        f = self.occupations(eps, mu)
        return (Q * f) @ Q.T, eps, Q, f, mu

    def occupations(self, eps, mu):
        return 0.5 * (1.0 - torch.tanh(0.5 * self.beta * (eps - mu)))

    def scf(self, R, mix):
        """Linear mixing from the valence electrons spread over each atom's orbitals; the P with the smallest residual."""
        self.at(R)
        P = torch.diag((0.5 * self.par[:, 3:4] / self.par[:, 1:2]).expand(-1, 4).reshape(-1)[self.orb])
        P = P * self.nocc / P.trace()
        best, kept = math.inf, None
        for _ in range(SCF_STEPS):
            D = self.density(self.h + self.G(P))[0]
            err = float((D - P).abs().max())
            if err < best:
                best, kept = err, P
            P = mix * P + (1.0 - mix) * D
        return kept

    def evaluate(self, R, X, m):
        """D0, U, forces at fixed D0 and X, and the rank-m Krylov kernel of D0 - X."""
        self.at(R)
        G = self.G(X)
        D, eps, Q, f, mu = self.density(self.h + G)
        ent = -KB * (torch.special.xlogy(f, f) + torch.special.xlogy(1 - f, 1 - f)).sum()
        U = 2 * (self.h * D).sum() + ((2 * D - X) * G).sum() + self.E.sum() - 2 * self.kT / KB * ent
        F = torch.zeros(self.N, 3, dtype=torch.float64, device=self.dev)
        Db, Xb = self.pad(D).permute(0, 2, 1, 3), self.pad(X).permute(0, 2, 1, 3)
        Yb = 2 * Db - Xb
        for A, B in zip(self.A.split(2048), self.B.split(2048)):
            x = R.clone().requires_grad_(True)
            W, S, E = self.blocks(x, A, B)
            e = E.sum() - 2 * torch.einsum("p,pmn,pmn->", self.par[B, 3], W[:, :, :, 0, 0], Db[A, A])
            e = e - 2 * torch.einsum("p,pmn,pmn->", self.par[A, 3], W[:, 0, 0], Db[B, B])
            e = e + 2 * ((self.bet[A][:, :, None] + self.bet[B][:, None]) * S * Db[A, B]).sum()
            e = e + 2 * torch.einsum("pmnls,pmn,pls->", W, Yb[A, A], Xb[B, B])
            e = e + 2 * torch.einsum("pmnls,pmn,pls->", W, Xb[A, A], Yb[B, B])
            e = e - 2 * torch.einsum("pmnls,pml,pns->", W, Yb[A, B], Xb[A, B])
            F -= torch.autograd.grad(e, x)[0]
        # Krylov kernel: divided differences, responses of trace zero, least squares on W0
        de = eps[:, None] - eps[None]
        mid = self.occupations(0.5 * (eps[:, None] + eps[None]), mu)
        tie = self.beta * de.abs() < 1e-5
        Lam = torch.where(tie, -self.beta * mid * (1 - mid), (f[:, None] - f[None]) / torch.where(tie, torch.ones_like(de), de))
        W0, Vs, Ws, v = D - X, [], [], D - X
        for _ in range(m):
            for _ in range(2):
                for k in Vs:
                    v = v - (k * v).sum() * k
            v = v / v.norm()
            F1, ld = Q.T @ self.G(v) @ Q, Lam.diagonal()
            dmu = (ld * F1.diagonal()).sum() / ld.sum() if float(ld.sum().abs()) > 1e-300 else 0.0
            Vs.append(v)
            v = Q @ (Lam * (F1 - dmu * torch.eye(self.n, dtype=F1.dtype, device=F1.device))) @ Q.T - v
            Ws.append(v)
        if m:
            w = torch.stack([x.reshape(-1) for x in Ws])
            c = torch.linalg.solve(w @ w.T, w @ W0.reshape(-1))
        K = sum((c[i] * Vs[i] for i in range(m)), torch.zeros_like(D))
        return dict(D=D, eps=eps, U=float(U), F=F, K=K)


def exact(case, seed):
    if case["kind"] == "product":
        s = prepare(case, seed)
        return s["A"] @ s["B"].T if case["terms"] == 10 else None
    if case["kind"] == "batch" or case["size"] > (120 if case["mol"] == "strand" else 4):
        return None                                      # too long in 64 bits
    Z, R, V = molecule(case["mol"], case["size"], seed)
    ref = Reference(Z, case["Te"])
    R, V = (torch.tensor(v, dtype=torch.float64, device=ref.dev) for v in (R, V))
    X = ref.scf(R, 0.1)
    now = ref.evaluate(R, X, case["m"])
    if case["kind"] == "point":
        return dict(F=now["F"], D=now["D"], U=now["U"])
    mass = ref.par[:, 4:5]
    V = V + 0.5 * DT * ACCEL * now["F"] / mass
    R = R + DT * V
    now = ref.evaluate(R, X - KAPPA * now["K"], 0)
    V = V + 0.5 * DT * ACCEL * now["F"] / mass
    kin = float((0.5 * mass * V * V).sum() / ACCEL)
    answer = dict(R=R, V=V, F=now["F"], E=dict(E_kin=kin, U=now["U"], E_tot=kin + now["U"], rank=None))
    if case["read"]:
        answer.update(D=now["D"], eps=now["eps"])
    return answer
