"""Workloads of the r-z implicit PIC/MC library: what a program that uses it has it do, from
the smallest reactors, where launches and latency count, to the largest, where particles do.

  solve   one stand-alone field solve on device arrays (pic_field_solve)
  step    timesteps of one reactor (pic_step) and the averages of them on the device
          (pic_moments), as a program that follows a discharge does call after call
  batch   one timestep of several reactors together (pic_batch_step) and their averages
  window  the collisionless window's functional and its gradient (pic_window)

Argon discharges with the synthetic cross sections of the repository's benchmark; its reactors
are c1 (33 x 65 nodes, 1e5 particles per species), c2 (129 x 513, 1e7), c3 (257 x 1025, 1e8),
the batch sweep (33 x 65 to 129 x 513) and the window's c5 (65 x 257).  Weight splitting
(every rf period) is off, so that every pass of a case does the same work.

exact() computes the same step in plain PyTorch, FP64: Philox draws, load, deposit, a direct
field solve, the merged particle pass with its Monte Carlo collisions.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch

from paper_1001_2969_gb300 import pic

QE, ME, AMU = 1.602176634e-19, 9.1093837015e-31, 1.66053906660e-27
M_AR, KB, EPS0 = 39.948 * AMU, 1.380649e-23, 8.8541878128e-12
F_RF = 13.56e6
N_E = 1001  # points of a cross-section table


# ---- the cases ----

def listed():
    return [
        # the field alone: c1's mesh, one whose rows are no multiple of a warp, c2's in FP64, c3's
        dict(name="solve small mixed", kind="solve", precision="mixed", nz=33, nr=65, face="max", chi=0.3),
        dict(name="solve ragged mixed", kind="solve", precision="mixed", nz=65, nr=300, face="mean", chi=3.0),
        dict(name="solve c2 fp64", kind="solve", precision="fp64", nz=129, nr=513, face="max", chi=1.1),
        dict(name="solve c3 mixed", kind="solve", precision="mixed", nz=257, nr=1025, face="max", chi=0.22),
        # one reactor: c1; a medium one in FP64; c2 (the benchmark's); c3
        dict(name="step c1 mixed", kind="step", precision="mixed", nz=33, nr=65, n=100_000, n0=1e15, p=4.0,
             amp=100.0, per=400, steps=1),
        dict(name="step medium fp64", kind="step", precision="fp64", nz=65, nr=257, n=1_000_000, n0=1e15, p=4.0,
             amp=100.0, per=200, steps=1),
        dict(name="step c2 mixed", kind="step", precision="mixed", nz=129, nr=513, n=10_000_000, n0=5e15, p=4.0,
             amp=300.0, per=200, steps=1),
        dict(name="step c3 mixed", kind="step", precision="mixed", nz=257, nr=1025, n=100_000_000, n0=5e15, p=8.0,
             amp=200.0, per=100, freq=60e6, steps=1),
        # a run continued from stored particles (accelerations, uneven weights), the X-Y-Z pusher,
        # z-r weighting, the mean face rule, isotropic scattering; odd sizes
        dict(name="step restart options", kind="step", precision="mixed", nz=65, nr=200, n=777_777, n0=2e15, p=20.0,
             amp=250.0, per=200, steps=1, restart=True, pusher="xyz", weighting="zr", face="mean",
             scatter="isotropic"),
        # ions every fourth step, a blocking capacitor before the electrode; four steps a call
        dict(name="steps subcycle circuit", kind="step", precision="mixed", nz=65, nr=257, n=1_500_001, n0=5e15,
             p=10.0, amp=200.0, per=200, steps=4, subcycle=4, circuit=1e-9),
        # a parameter sweep: reactors of different meshes and sizes side by side
        dict(name="batch of 8 mixed", kind="batch", precision="mixed", reactors=8, n_lo=50_000, n_hi=2_000_000,
             draw=4),
        # the gradient of the ion density's average (c5's mesh)
        dict(name="window gradient", kind="window", precision="mixed", nz=65, nr=257, n=300_000, n0=1e15, amp=100.0,
             per=200, steps=16, ckpt=4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "step", "step", "step", "step", "batch", "window"])
    nz = rng.choice([17, 33, 65, 129, 257])
    nr = min(1025, int(_log(rng, max(40, nz), 8 * nz + 1)))
    precision = rng.choice(["mixed", "mixed", "fp64"])
    face = rng.choice(["max", "max", "mean"])
    if kind == "solve":
        return dict(kind=kind, precision=precision, nz=nz, nr=nr, face=face, chi=round(_log(rng, 0.1, 20.0), 3))
    amp, per, p = round(rng.uniform(50.0, 500.0), 1), rng.choice([100, 200, 400]), round(_log(rng, 1.0, 100.0), 2)
    n0 = float("%.2e" % _log(rng, 3e14, 1e16))
    if kind == "step":
        least = max(20_000, 8 * (nz - 1) * (nr - 1))  # a plasma has particles in every cell
        n = int(_log(rng, least, max(2 * least, 30_000_000 if precision == "mixed" else 2_000_000)))
        c = dict(kind=kind, precision=precision, nz=nz, nr=nr, n=n, n0=n0, p=p, amp=amp, per=per, steps=1, face=face)
        if n <= 2_000_000 and rng.random() < 0.5:
            c.update(restart=True, pusher=rng.choice(["local", "xyz"]), weighting=rng.choice(["zr2", "zr"]),
                     scatter=rng.choice(["vs", "isotropic"]))
        return c
    if kind == "batch":
        return dict(kind=kind, precision="mixed", reactors=rng.randint(3, 8), n_lo=20_000,
                    n_hi=int(_log(rng, 200_000, 3_000_000)), draw=rng.randrange(1000))
    nz, nr = rng.choice([33, 65]), rng.randint(100, 257)
    steps = rng.choice([8, 12, 16])
    return dict(kind=kind, precision=precision, nz=nz, nr=nr, n=int(_log(rng, 50_000, 300_000)), n0=1e15, amp=amp,
                per=per, steps=steps, ckpt=rng.choice([2, 4]))


# ---- a program's configuration of a reactor ----

def _sigma(E, collisions):
    def rise(thr, e_peak, s_peak):
        s = np.where((E > thr) & (E <= e_peak), s_peak * (E - thr) / (e_peak - thr), 0.0)
        return np.where(E > e_peak, s_peak * e_peak / np.maximum(E, e_peak), s)
    e = np.stack([np.full_like(E, 1e-19), rise(11.5, 25.0, 2e-20), rise(15.76, 100.0, 3e-20)])
    i = np.full((1, len(E)), 5e-19)
    return e * collisions, i * collisions


def config(c, seed, collisions=True):
    """The library's configuration of a case: c2's cell sizes, the case's mesh and particles."""
    nz, nr, amp = c["nz"], c["nr"], c.get("amp", 100.0)
    E = np.linspace(0.0, 4.0 * amp, N_E)
    se, si = _sigma(E, 1.0 if collisions else 0.0)
    n = c.get("n", 0)
    cap = int(n * (1.2 if n > 30_000_000 else 1.5)) + 4096
    freq = c.get("freq", F_RF)
    return dict(
        R=0.20 * (nr - 1) / 512, L=0.025 * (nz - 1) / 128, nz=nz, nr=nr,
        species=[dict(q=-QE, m=ME, n0=c.get("n0", 1e15), T_eV=3.0, n_init=n, capacity=cap),
                 dict(q=QE, m=M_AR, n0=c.get("n0", 1e15), T_eV=0.026, n_init=n, capacity=cap)],
        xsec=[dict(n_e=N_E, E_max=4.0 * amp, sigma=se, threshold=np.array([0.0, 11.5, 15.76]),
                   kind=["elastic", "excite", "ionize"], B_eV=10.0),
              dict(n_e=N_E, E_max=4.0 * amp, sigma=si, threshold=np.array([0.0]), kind=["cx"], B_eV=10.0)],
        rf=dict(amp=[amp], freq=[freq], phase=[0.0]), gas=dict(p_Pa=c.get("p", 4.0), T_K=300.0, m_gas=M_AR),
        dt=1.0 / freq / c.get("per", 200), seed=_key(seed), precision=c["precision"],
        weighting=c.get("weighting", "zr2"), chi_face=c.get("face", "max"), scatter=c.get("scatter", "vs"),
        pusher=c.get("pusher", "local"), split_every=0, mg_max_cycles=50, mg_tol=1e-10, eedf_bins=200,
        eedf_emax=100.0, ion_subcycle=c.get("subcycle", 1), circuit_C=c.get("circuit", 0.0))


def _key(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 0x1234567) & ((1 << 63) - 1)


def _first_step(c, seed):
    # somewhere in the second quarter of an rf period, on a period of the subcycling
    K = c.get("subcycle", 1)
    return (c["per"] // 4 + int(seed) % (c["per"] // 4)) // K * K


def _generator(seed, salt, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed((int(seed) * 1_000_003 + salt) % (1 << 62))
    return g


def _stored_particles(c, cfg, s, seed):
    """Particles of a stored run: uniform in (z, r^2), warm, with accelerations and weights
    within a factor of four, ids in no order."""
    sp, n, g = cfg["species"][s], c["n"], _generator(seed, 11 + s, "cpu")
    u = lambda: torch.rand(n, generator=g, dtype=torch.float64)  # noqa: E731
    v = lambda k: k * torch.randn(n, generator=g, dtype=torch.float64)  # noqa: E731
    sig = math.sqrt(sp["T_eV"] * QE / sp["m"]) * (1.5 if s == 0 else 1.0)
    acc = QE / sp["m"] * 1e3
    vol = math.pi * cfg["R"] ** 2 * cfg["L"]
    z, r = cfg["L"] * (0.001 + 0.998 * u()), cfg["R"] * 0.999 * torch.sqrt(u())
    w = sp["n0"] * vol / n * 4.0 ** (u() - 0.5)
    p = dict(r=r, z=z, vr=v(sig), vt=v(sig), vz=v(sig), ar=v(acc), az=v(acc), w=w)
    p = {k: x.numpy() for k, x in p.items()}
    p["id"] = torch.randperm(n, generator=g).numpy().astype(np.uint64)
    p["at"] = v(acc).numpy() if c.get("pusher") == "xyz" else np.zeros(n)
    return p


class _Averages:
    """Device buffers for a reactor's averages, and their reading (pic_moments) with a reset.  A
    program on the mixed path, whose particles and decisions are FP32, keeps its history in FP32."""

    def __init__(self, cfg):
        nz, nr, nb, self.mixed = cfg["nz"], cfg["nr"], cfg["eedf_bins"], cfg["precision"] == "mixed"
        ng = nz * nr
        self.buf = torch.zeros(5 * ng + nb, dtype=torch.float64, device="cuda")
        self.kept = self.buf.float() if self.mixed else self.buf
        self.views = {k: self.kept[i * ng:(i + 1) * ng].view(nz, nr) for i, k in enumerate(("ne", "ni", "phi", "Er", "Ez"))}
        self.views["eedf"] = self.kept[5 * ng:]
        self.counters = np.zeros(pic.PIC_NCOUNT, dtype=np.int64)
        # what the particles did (collisions, births, losses) and how many were moved; the
        # solver's own iteration count is no result of the discharge
        self.which = [k for k in range(pic.PIC_NCOUNT) if k not in (pic.PIC_C_MGCYC, pic.PIC_C_STEPS)]
        self.charge = np.zeros(3)
        dp = ctypes.POINTER(ctypes.c_double)
        at = lambda k: ctypes.cast(self.buf.data_ptr() + 8 * k, dp)  # noqa: E731
        self.out = pic.pic_moments_out(
            *[at(i * ng) for i in range(6)], self.counters.ctypes.data_as(ctypes.POINTER(ctypes.c_int64)),
            self.charge.ctypes.data_as(dp), 0, 1)

    def read(self, h):
        pic.pic_moments_into(h, self.out, True)
        counts, charge = self.counters[self.which], self.charge
        if self.mixed:
            self.kept.copy_(self.buf)
            counts, charge = counts.astype(np.float32), charge.astype(np.float32)
        return dict(self.views, charge=charge, counters=counts)


def _reactor(c, seed):
    cfg = config(c, seed)
    h = pic.pic_init(cfg, load=not c.get("restart"))
    if c.get("restart"):
        for s in (0, 1):
            pic.pic_set_particles(h, s, _stored_particles(c, cfg, s, seed))
    pic.pic_set_step(h, _first_step(c, seed))
    avg = _Averages(cfg)
    if _before(c):
        pic.pic_step(h, _before(c))
        avg.read(h)
    return h, avg


def _before(c):
    """Steps taken before the first pass: a run under way, but for one that starts from stored particles."""
    return 0 if c.get("restart") else c.get("subcycle", 1)


def _sweep(c):
    """The reactors of a batch, as cases of their own."""
    r, out = random.Random(c["draw"]), []
    for _ in range(c["reactors"]):
        nz = r.choice([33, 65, 129])
        nr = r.choice([x for x in (65, 129, 257, 513) if x >= 2 * nz - 1])
        out.append(dict(kind="step", precision=c["precision"], nz=nz, nr=nr, n=int(_log(r, c["n_lo"], c["n_hi"])),
                        n0=5e15, p=_log(r, 1.0, 100.0), amp=r.uniform(50.0, 500.0), per=200, steps=1))
    return out


def _charge_and_chi(c, seed):
    """A discharge's charge and susceptibility: a bulk, sheaths, and the noise of its particles."""
    nz, nr, g = c["nz"], c["nr"], _generator(seed, 3)
    z = torch.linspace(0.0, 1.0, nz, dtype=torch.float64, device="cuda")[:, None]
    r = torch.linspace(0.0, 1.0, nr, dtype=torch.float64, device="cuda")[None, :]
    a = torch.rand(4, generator=g, dtype=torch.float64, device="cuda")
    bulk = torch.sin(math.pi * (0.02 + 0.96 * z)) ** 0.5 * (1.05 - r ** (2.0 + 4.0 * a[0]))
    noise = lambda k: k * torch.randn(nz, nr, generator=g, dtype=torch.float64, device="cuda")  # noqa: E731
    chi = (c["chi"] * bulk * (1.0 + noise(0.05))).clamp_min(0.0)
    n0 = c["chi"] * 5e15
    sheath = torch.exp(-z * (12.0 + 10.0 * a[1])) + torch.exp(-(1.0 - z) * (12.0 + 10.0 * a[2]))
    rho = QE * n0 * (0.02 * sheath * bulk + noise(0.03) * bulk)
    return rho.contiguous(), chi.contiguous(), 50.0 + 250.0 * float(a[3])


def prepare(case, seed):
    c = case
    if c["kind"] == "solve":
        h = pic.pic_init(config(c, seed), load=False)
        rho, chi, V = _charge_and_chi(c, seed)
        return dict(kind="solve", h=h, rho=rho, chi=chi, V=V, phi=torch.zeros_like(rho))
    if c["kind"] == "step":
        h, avg = _reactor(c, seed)
        return dict(kind="step", h=h, avg=avg, steps=c["steps"])
    if c["kind"] == "batch":
        rs = [_reactor(x, seed * 100 + k) for k, x in enumerate(_sweep(c))]
        hs = [h for h, _ in rs]
        return dict(kind="batch", hs=hs, avgs=[a for _, a in rs], batch=pic.pic_batch_init(hs))
    cfg = config(c, seed, collisions=False)
    h = pic.pic_init(cfg)
    pic.pic_set_step(h, _first_step(c, seed))
    return dict(kind="window", h=h, steps=c["steps"], ckpt=c["ckpt"], w=_weight(cfg), amp=c["amp"],
                dtype=np.float32 if c["precision"] == "mixed" else np.float64)


def _weight(cfg):
    z = np.linspace(0.0, cfg["L"], cfg["nz"])[:, None]
    r = np.linspace(0.0, cfg["R"], cfg["nr"])[None, :]
    return np.exp(-((r - 0.3 * cfg["R"]) ** 2 + (z - 0.5 * cfg["L"]) ** 2) / (2.0 * (0.25 * cfg["L"]) ** 2))


def run(state):
    s = state
    if s["kind"] == "solve":
        pic.pic_field_solve_device(s["h"], s["rho"].data_ptr(), s["chi"].data_ptr(), s["V"], s["phi"].data_ptr())
        return s["phi"]
    if s["kind"] == "step":
        pic.pic_step(s["h"], s["steps"])
        return s["avg"].read(s["h"])
    if s["kind"] == "batch":
        pic.pic_batch_step(s["batch"], 1)
        return [a.read(h) for h, a in zip(s["hs"], s["avgs"])]
    J, dA, dP = pic.pic_window(s["h"], s["steps"], s["ckpt"], s["w"], s["amp"])
    return {k: np.asarray(v, dtype=s["dtype"]) for k, v in (("J", J), ("dJ_damp", dA), ("dJ_dphi", dP))}


def work(case):
    c = case
    if c["kind"] == "batch":
        w = [work(x) for x in _sweep(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    ng = c["nz"] * c["nr"]
    if c["kind"] == "solve":
        # rho and chi in, phi out; one application of the operator and one sweep of the lines
        return dict(bytes=24.0 * ng, flops=30.0 * ng)
    rec = 44.0 if c["precision"] == "mixed" else 76.0
    moved = c["n"] * (c["steps"] + math.ceil(c["steps"] / c.get("subcycle", 1)))  # electrons and ions
    grids = 8.0 * ng * 10  # deposit and potential in and out, the averages
    b, f = 2.0 * rec * moved + grids * c["steps"], 230.0 * moved
    if c["kind"] == "window":  # the forward and its reverse
        b, f = 3.0 * b, 3.0 * f
    return dict(bytes=b, flops=f)


# ---- the same in plain PyTorch, FP64 ----

class _Mesh:
    def __init__(self, cfg, dev):
        self.nz, self.nr = cfg["nz"], cfg["nr"]
        self.dz, self.dr = cfg["L"] / (self.nz - 1), cfg["R"] / (self.nr - 1)
        self.zr2, self.mean = cfg["weighting"] == "zr2", cfg["chi_face"] == "mean"
        t = dict(dtype=torch.float64, device=dev)
        j = torch.arange(self.nr, **t)
        rp, rm = (j + 0.5) * self.dr, (j - 0.5).clamp_min(0.0) * self.dr
        self.area = math.pi * (rp * rp - rm * rm)      # z faces of node j's ring
        self.side = 2.0 * math.pi * rp * self.dz       # r face between j and j + 1
        # node volumes: the integral of the deposit's shape factor over the domain
        r, lo, hi = j * self.dr, (j - 1).clamp_min(0.0) * self.dr, (j + 1).clamp_max(self.nr - 1) * self.dr
        if self.zr2:
            v = math.pi / 2.0 * (hi * hi - lo * lo)
        else:
            v = math.pi / 3.0 * ((hi - r) * (2.0 * r + hi) + (r - lo) * (2.0 * r + lo))
        h = torch.full((self.nz,), self.dz, **t)
        h[0] = h[-1] = 0.5 * self.dz
        self.V = h[:, None] * v[None, :]

    def shapes(self, zc, rc):
        i, j = zc.detach().floor().long(), rc.detach().floor().long()
        s1, o = zc - i, rc - j
        r1 = o * (2.0 * j + o) / (2.0 * j + 1.0) if self.zr2 else o
        return i, j, (1.0 - s1, s1), (1.0 - r1, r1)

    def corners(self, zc, rc):
        i, j, sz, sr = self.shapes(zc, rc)
        return [((i + a) * self.nr + (j + b), sz[a] * sr[b]) for a in (0, 1) for b in (0, 1)]

    def deposit(self, N, zc, rc, w):
        for k, s in self.corners(zc, rc):
            N = N.index_add(0, k, w * s)
        return N

    def solve(self, rho, chi, bottom, top):
        """div[(1 + chi) grad phi] = -rho / eps0, potentials `bottom` and `top` on the z ends, 0 at
        r = R: columns of the interior eliminated one after another (block Thomas)."""
        nz, nr = self.nz, self.nr
        face = (lambda a, b: 0.5 * (a + b)) if self.mean else (lambda a, b: torch.where(a > b, a, b))
        cz = (1.0 + face(chi[:-1], chi[1:])) * self.area / self.dz
        cr = (1.0 + face(chi[:, :-1], chi[:, 1:])) * self.side[:-1] / self.dr
        n = nr - 1
        A, C, Rr = cz[:-1, :n], cz[1:, :n], cr[1:-1]  # below, above, right of the interior nodes
        D = A + C + Rr + torch.nn.functional.pad(Rr[:, :-1], (1, 0))
        b = rho[1:-1, :n] * self.area[:n] * self.dz / EPS0
        ends = torch.zeros_like(b)
        ends = torch.cat([A[:1] * bottom[:n], ends[1:]]) + torch.cat([ends[1:], C[-1:] * top[:n]])
        b = b + ends
        inv, y = [], []
        for j in range(n):
            T = torch.diag(D[:, j])
            if nz > 3:
                T = T - torch.diag(C[:-1, j], 1) - torch.diag(A[1:, j], -1)
            bj = b[:, j]
            if j:
                e = Rr[:, j - 1]
                T = T - e[:, None] * inv[-1] * e[None, :]
                bj = bj + e * (inv[-1] @ y[-1])
            inv.append(torch.linalg.inv(T))
            y.append(bj)
        x = [None] * n
        x[-1] = inv[-1] @ y[-1]
        for j in range(n - 2, -1, -1):
            x[j] = inv[j] @ (y[j] + Rr[:, j] * x[j + 1])
        inner = torch.nn.functional.pad(torch.stack(x, 1), (0, 1))
        wall = torch.ones(nr, dtype=rho.dtype, device=rho.device)
        wall[-1] = 0.0
        return torch.cat([(bottom * wall)[None], inner, top[None]])

    def field(self, phi):
        """-grad phi: central inside, one-sided on the Dirichlet rows and at r = R, E_r = 0 on the axis."""
        dz, dr = self.dz, self.dr
        Ez = torch.cat([(phi[:1] - phi[1:2]) / dz, (phi[:-2] - phi[2:]) / (2 * dz), (phi[-2:-1] - phi[-1:]) / dz])
        Er = torch.cat([torch.zeros_like(phi[:, :1]), (phi[:, :-2] - phi[:, 2:]) / (2 * dr),
                        (phi[:, -2:-1] - phi[:, -1:]) / dr], 1)
        return Ez, Er

    def wall(self, zc, rc):
        w = torch.full_like(zc, -1, dtype=torch.long)
        w = torch.where(rc >= self.nr - 1, 2, w)
        w = torch.where(zc >= self.nz - 1, 1, w)
        return torch.where(zc <= 0, 0, w)


def _mulhilo(a, b):
    """High and low words of the product of two 32-bit words held in int64."""
    a0, a1, b0, b1 = a & 0xFFFF, a >> 16, b & 0xFFFF, b >> 16
    lo = a0 * b0
    mid = a1 * b0 + (lo >> 16)
    mid2 = a0 * b1 + (mid & 0xFFFF)
    return a1 * b1 + (mid >> 16) + (mid2 >> 16), ((mid2 & 0xFFFF) << 16) | (lo & 0xFFFF)


def _philox(ids, step, stream, s, key):
    """Philox4x32-10 of (id, step, 2 stream + s): four words per particle."""
    c = [ids & 0xFFFFFFFF, ids >> 32, torch.full_like(ids, step & 0xFFFFFFFF), torch.full_like(ids, 2 * stream + s)]
    k0, k1 = key & 0xFFFFFFFF, (key >> 32) & 0xFFFFFFFF
    for _ in range(10):
        h0, l0 = _mulhilo(c[0], 0xD2511F53)
        h1, l1 = _mulhilo(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _u(x):
    return (x.double() + 0.5) * 2.0 ** -32


def _normals(a, b):
    rad = torch.sqrt(-2.0 * torch.log(_u(a)))
    return rad * torch.cos(2 * math.pi * _u(b)), rad * torch.sin(2 * math.pi * _u(b))


FIELDS = ("zc", "rc", "vr", "vt", "vz", "ar", "at", "az", "w")


class _Exact:
    """One reactor of a case in plain PyTorch."""

    def __init__(self, c, cfg, seed, dev, particles=None):
        self.c, self.cfg, self.dev, self.seed = c, cfg, dev, seed
        self.m = _Mesh(cfg, dev)
        self.step = _first_step(c, seed)
        self.dt, self.key = cfg["dt"], cfg["seed"]
        self.stored = particles
        self.ng = cfg["gas"]["p_Pa"] / (KB * cfg["gas"]["T_K"])
        self.v_gas = math.sqrt(KB * cfg["gas"]["T_K"] / M_AR)
        self.sig = [torch.tensor(np.asarray(x["sigma"]), dtype=torch.float64, device=dev) for x in cfg["xsec"]]
        self.nu = [self._nu_max(s) for s in (0, 1)]

    def _nu_max(self, s):
        x, m = self.cfg["xsec"][s], self.cfg["species"][s]["m"]
        tot = np.asarray(x["sigma"]).sum(0)
        E = np.linspace(0.0, x["E_max"], x["n_e"])
        best = (tot * np.sqrt(2.0 * E * QE / m)).max()
        beta = np.diff(tot) / np.diff(E)
        alpha = tot[:-1] - beta * E[:-1]
        fall = beta < 0.0
        Es = -alpha[fall] / (3.0 * beta[fall])
        ok = (Es > E[:-1][fall]) & (Es < E[1:][fall])
        if ok.any():
            best = max(best, ((alpha[fall] + beta[fall] * Es) * np.sqrt(2.0 * Es * QE / m))[ok].max())
        return self.ng * best * (1.0 + 1e-6)

    def chunks(self, s, size=4_000_000):
        """The reactor's particles before the step: the loaded ones (evenly over the cells, z and
        r^2 uniform within a cell, Maxwellian) or the stored ones."""
        sp, m = self.cfg["species"][s], self.m
        n, ncz = self.c["n"], m.nz - 1
        for a in range(0, n, size):
            b = min(n, a + size)
            if self.stored:
                p = {k: torch.as_tensor(v[a:b].astype(np.int64) if k == "id" else v[a:b]).to(self.dev)
                     for k, v in self.stored[s].items()}
                p["zc"], p["rc"] = p.pop("z") / m.dz, p.pop("r") / m.dr
                yield p
                continue
            ids = torch.arange(a, b, device=self.dev)
            base, rem = divmod(n, ncz * (m.nr - 1))
            cell = torch.where(ids < rem * (base + 1), ids // (base + 1),
                               rem + (ids - rem * (base + 1)) // max(base, 1))
            ppc = base + (cell < rem).long()
            i, j = cell % ncz, (cell // ncz).double()
            x, y = _philox(ids, 0xFFFFFFFF, 3, s, self.key), _philox(ids, 0xFFFFFFFF, 4, s, self.key)
            t = _u(x[1]) * (2.0 * j + 1.0)
            sig = math.sqrt(sp["T_eV"] * QE / sp["m"])
            vr, vt = _normals(x[2], x[3])
            vz, _ = _normals(y[0], y[1])
            w = sp["n0"] * math.pi * (2.0 * j + 1.0) * m.dr ** 2 * m.dz / ppc
            zero = torch.zeros_like(w)
            yield dict(zc=i + _u(x[0]), rc=j + t / (torch.sqrt(j * j + t) + j), vr=sig * vr, vt=sig * vt,
                       vz=sig * vz, ar=zero, at=zero, az=zero, w=w, id=ids)

    def deposits(self, parts):
        N = [torch.zeros(self.m.nz * self.m.nr, dtype=torch.float64, device=self.dev) for _ in (0, 1)]
        for s in (0, 1):
            for p in parts[s]:
                N[s] = self.m.deposit(N[s], p["zc"], p["rc"], p["w"])
        return N

    def potential(self, N, step, amp=None, top=None):
        sp, m = self.cfg["species"], self.m
        n = [x.view(m.nz, m.nr) / m.V for x in N]
        rho = sp[0]["q"] * n[0] + sp[1]["q"] * n[1]
        chi = sum(sp[s]["q"] ** 2 * self.dt ** 2 / (2 * EPS0 * sp[s]["m"]) * n[s] for s in (0, 1))
        rf = self.cfg["rf"]
        one = torch.ones(m.nr, dtype=torch.float64, device=self.dev)
        V = (rf["amp"][0] if amp is None else amp) * math.sin(2 * math.pi * rf["freq"][0] * (step + 1) * self.dt)
        return m.solve(rho, chi, V * one, 0.0 * one if top is None else top)

    def final_push(self, s, p, Ez, Er):
        sp, m, dt = self.cfg["species"][s], self.m, self.dt
        qm = sp["q"] / sp["m"]
        at = m.corners(p["zc"], p["rc"])
        ez = sum(w * Ez.reshape(-1)[k] for k, w in at)
        er = sum(w * Er.reshape(-1)[k] for k, w in at)
        p = dict(p, zc=p["zc"] + 0.5 * qm * dt * dt / m.dz * ez, rc=p["rc"] + 0.5 * qm * dt * dt / m.dr * er,
                 vz=p["vz"] + 0.5 * qm * dt * ez, vr=p["vr"] + 0.5 * qm * dt * er,
                 az=0.5 * (qm * ez + p["az"]), ar=0.5 * (qm * er + p["ar"]), at=0.5 * p["at"])
        thru = p["rc"] < 0
        p["rc"] = torch.where(thru, -p["rc"], p["rc"])
        if self.cfg["pusher"] == "xyz":
            for k in ("vr", "ar", "vt", "at"):
                p[k] = torch.where(thru, -p[k], p[k])
        else:
            for k in ("vr", "ar"):
                p[k] = torch.where(thru, p[k].abs(), p[k])
        return p

    def first_push(self, p):
        m, dt, xyz = self.m, self.dt, self.cfg["pusher"] == "xyz"
        vx = p["vr"] + 0.5 * p["ar"] * dt
        vy = p["vt"] + (0.5 * p["at"] * dt if xyz else 0.0)
        vz = p["vz"] + 0.5 * p["az"] * dt
        x, y = p["rc"] * m.dr + vx * dt, vy * dt
        q2 = x * x + y * y
        r = torch.sqrt(torch.where(q2 > 0, q2, torch.ones_like(q2)))
        c, sn = torch.where(q2 > 0, x / r, torch.ones_like(x)), torch.where(q2 > 0, y / r, torch.zeros_like(y))
        r = torch.where(q2 > 0, r, torch.zeros_like(r))
        ar = p["ar"] * c + (p["at"] * sn if xyz else 0.0)
        at = -p["ar"] * sn + p["at"] * c if xyz else p["at"]
        return dict(p, zc=p["zc"] + vz * dt / m.dz, rc=r / m.dr, vr=vx * c + vy * sn, vt=-vx * sn + vy * c, vz=vz,
                    ar=ar, at=at)

    def _cos_chi(self, e, R):
        iso = 1.0 - 2.0 * R
        if self.cfg["scatter"] == "isotropic":
            return iso
        ee = e.clamp_min(1e-6)
        return torch.where(e < 1e-6, iso, (2.0 + ee - 2.0 * (1.0 + ee) ** R) / ee).clamp(-1.0, 1.0)

    @staticmethod
    def _turn(u, cc, phi):
        """The unit vectors u turned by the angle of cosine cc at azimuth 2 pi phi about them."""
        sc, cp, sp_ = torch.sqrt((1.0 - cc * cc).clamp_min(0.0)), torch.cos(2 * math.pi * phi), torch.sin(2 * math.pi * phi)
        s2 = u[0] ** 2 + u[1] ** 2
        s = torch.sqrt(s2.clamp_min(1e-24))
        out = (cc * u[0] + sc * (cp * u[1] + sp_ * u[0] * u[2]) / s,
               cc * u[1] + sc * (-cp * u[0] + sp_ * u[1] * u[2]) / s, cc * u[2] - sc * sp_ * s2 / s)
        along = (sc * cp, sc * sp_ * u[2], cc * u[2])
        return [torch.where(s2 < 1e-24, a, o) for a, o in zip(along, out)]

    def collide(self, s, p):
        """Null-collision Monte Carlo in place; the births as (species, particles)."""
        sp, xs = self.cfg["species"], self.cfg["xsec"][s]
        m_s, births = sp[s]["m"], []
        x = _philox(p["id"], self.step, 0, s, self.key)
        t_null = math.ceil((1.0 - math.exp(-self.nu[s] * self.dt)) * 2.0 ** 32 - 0.5)
        k = torch.nonzero(x[0] < t_null).flatten()
        if not len(k):
            return births
        x, ids = [v[k] for v in x], p["id"][k]
        v = [p[f][k] for f in ("vr", "vt", "vz")]
        gas = [torch.zeros_like(v[0])] * 3
        if s == 1:
            y = _philox(ids, self.step, 1, 1, self.key)
            gas = [self.v_gas * t for t in (*_normals(y[0], y[1]), _normals(y[2], y[3])[0])]
        g3 = [a - b for a, b in zip(v, gas)]
        g = torch.sqrt(sum(t * t for t in g3))
        E = 0.5 * m_s / QE * g * g
        pos = (E / xs["E_max"] * (N_E - 1))
        b = pos.long().clamp(0, N_E - 2)
        inside = self.sig[s][:, b] + (pos - b) * (self.sig[s][:, b + 1] - self.sig[s][:, b])
        beyond = self.sig[s][:, -1:] * (xs["E_max"] / E.clamp_min(1e-30))
        nu = self.ng * g * torch.where(E >= xs["E_max"], beyond, inside)
        ch = (_u(x[1]) * self.nu[s] >= nu.cumsum(0)).sum(0)
        thr = torch.tensor(np.append(np.asarray(xs["threshold"], dtype=float), np.inf), device=self.dev)
        real = (ch < len(nu)) & ((ch == 0) | (E > thr[ch]))
        if s == 1:
            for f, t in zip(("vr", "vt", "vz"), gas):
                p[f][k[real]] = t[real]
            return births
        for kind in range(3):
            q = torch.nonzero(real & (ch == kind)).flatten()
            if not len(q):
                continue
            at, e, gg = k[q], E[q], g[q]
            u, ux, uphi = [t[q] / gg for t in g3], _u(x[2][q]), _u(x[3][q])
            if kind == 0:
                cc = self._cos_chi(e, ux)
                speed = gg * torch.sqrt(1.0 - 2.0 * m_s / M_AR * (1.0 - cc))
            elif kind == 1:
                cc = self._cos_chi(e - thr[1], ux)
                speed = torch.sqrt(2.0 * QE / m_s * (e - thr[1]))
            else:
                y, zz = _philox(ids[q], self.step, 1, 0, self.key), _philox(ids[q], self.step, 2, 0, self.key)
                B = xs["B_eV"]
                ej = B * torch.tan(_u(y[0]) * torch.atan((e - thr[2]) / (2.0 * B)))
                esc = (e - thr[2] - ej).clamp_min(0.0)
                cc, speed = self._cos_chi(esc, ux), torch.sqrt(2.0 * QE / m_s * esc)
                w = self._turn(u, self._cos_chi(ej, _u(y[1])), _u(y[2]))
                vej = torch.sqrt(2.0 * QE / m_s * ej)
                par = {f: p[f][at].clone() for f in (*FIELDS, "id")}  # the parent's id orders the newborns
                births.append((0, dict(par, vr=vej * w[0], vt=vej * w[1], vz=vej * w[2])))
                k3 = [self.v_gas * t for t in (*_normals(zz[0], zz[1]), _normals(zz[2], zz[3])[0])]
                f = sp[1]["q"] * sp[0]["m"] / (sp[0]["q"] * sp[1]["m"])
                births.append((1, dict(par, vr=k3[0], vt=k3[1], vz=k3[2], ar=f * par["ar"], at=f * par["at"],
                                       az=f * par["az"])))
            for f, t in zip(("vr", "vt", "vz"), self._turn(u, cc, uphi)):
                p[f][at] = speed * t
        return births

    def averages(self):
        """What pic_moments gives after the first pass's step."""
        parts = [list(self.chunks(s)) for s in (0, 1)]
        self.next_id = [self.c["n"]] * 2
        for _ in range(_before(self.c) + 1):
            parts, out = self.one_step(parts)
            self.step += 1
        return out

    def one_step(self, parts):
        m, cfg = self.m, self.cfg
        phi = self.potential(self.deposits(parts), self.step)
        Ez, Er = m.field(phi)
        eedf = torch.zeros(cfg["eedf_bins"], dtype=torch.float64, device=self.dev)
        charge = torch.zeros(3, dtype=torch.float64, device=self.dev)

        def settle(s, p):  # the walls' charge; the particles that are left
            wall = m.wall(p["zc"], p["rc"])
            charge.index_add_(0, wall.clamp_min(0), torch.where(wall >= 0, p["w"] * cfg["species"][s]["q"], 0.0))
            return {k: v[wall < 0] for k, v in p.items()}

        kept, born = [[], []], [[], []]
        for s in (0, 1):
            while parts[s]:
                p = settle(s, self.final_push(s, parts[s].pop(0), Ez, Er))
                births = self.collide(s, p)
                if s == 0:
                    E = 0.5 * ME / QE * (p["vr"] ** 2 + p["vt"] ** 2 + p["vz"] ** 2) * (cfg["eedf_bins"] / cfg["eedf_emax"])
                    ok = E < cfg["eedf_bins"]
                    eedf.index_add_(0, E[ok].long(), p["w"][ok])
                kept[s].append(settle(s, self.first_push(p)))
                for t, q in births:
                    born[t].append(settle(t, self.first_push(q)))
        for t in (0, 1):
            if born[t]:  # numbered in the order of their parents
                q = {f: torch.cat([x[f] for x in born[t]]) for f in born[t][0]}
                rank = torch.empty_like(q["id"])
                rank[torch.argsort(q["id"])] = torch.arange(len(rank), device=self.dev)
                kept[t].append(dict(q, id=self.next_id[t] + rank))
                self.next_id[t] += len(rank)
        n = [x.view(m.nz, m.nr) / m.V for x in self.deposits(kept)]
        return kept, dict(ne=n[0], ni=n[1], phi=phi, Er=Er, Ez=Ez, eedf=eedf, charge=charge, counters=None)

    def window(self):
        """J and its gradient by autograd through the window's steps."""
        m, K = self.m, self.c["steps"]
        amp = torch.tensor(self.c["amp"], dtype=torch.float64, device=self.dev, requires_grad=True)
        top = torch.zeros(m.nr, dtype=torch.float64, device=self.dev, requires_grad=True)
        w = torch.tensor(_weight(self.cfg).reshape(-1), device=self.dev)
        p = [next(self.chunks(s)) for s in (0, 1)]
        N, J = self.deposits([[x] for x in p]), 0.0
        for k in range(K):
            Ez, Er = m.field(self.potential(N, self.step + k, amp, top))
            N = []
            for s in (0, 1):
                for push in (lambda q: self.final_push(s, q, Ez, Er), self.first_push):
                    q = push(p[s])
                    alive = m.wall(q["zc"].detach(), q["rc"].detach()) < 0
                    p[s] = {f: v[alive] for f, v in q.items()}
                N.append(m.deposit(torch.zeros_like(w), p[s]["zc"], p[s]["rc"], p[s]["w"]))
            J = J + (w * N[1]).sum() / K
        gA, gP = torch.autograd.grad(J, (amp, top))
        return dict(J=J.detach(), dJ_damp=gA, dJ_dphi=gP)


def exact(case, seed):
    c, dev = case, "cuda" if torch.cuda.is_available() else "cpu"
    if c["kind"] == "solve":
        rho, chi, V = _charge_and_chi(c, seed)
        one = torch.ones(c["nr"], dtype=torch.float64, device=rho.device)
        return _Mesh(config(c, seed), rho.device).solve(rho, chi, V * one, 0.0 * one)
    if c["kind"] == "batch":
        return [_Exact(x, config(x, seed * 100 + k), seed * 100 + k, dev).averages()
                for k, x in enumerate(_sweep(c))]
    if c["kind"] == "window":
        return _Exact(c, config(c, seed, collisions=False), seed, dev).window()
    if c["steps"] > 1 or c.get("circuit") or c["n"] > 30_000_000:
        return None  # the steps after the first, and the largest load, take more than some seconds here
    cfg = config(c, seed)
    stored = [_stored_particles(c, cfg, s, seed) for s in (0, 1)] if c.get("restart") else None
    return _Exact(c, cfg, seed, dev, stored).averages()
