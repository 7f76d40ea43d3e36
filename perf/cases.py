"""Performance cases of the nanodisk library: what its users run, through the package's public calls.

Every case is a dict of plain values:
  kind       field | energy | observe | rk4 | heun | relax | graph
  R, L       disk radius and thickness in nm (cell edge a = 2 nm, so D = round(R) cells a side);
             kinds relax and graph with "disks" > 0 hold that many disks of different sizes instead
  replicas   states per disk in the handle
  fp64       handle precision
  steps      time steps of one call (rk4, heun, graph)
  T          temperature in kelvin (heun)
  alpha, hy  damping, external field along y in A/m
  plan       stepping plan (-1: the handle's default; 200 / 201: the 8- and 16-CTA cluster plans that
             the autotuner picks for single disks)
  grid3x     allow the padded sizes 192 and 200
  tol        relaxation tolerance
"""
import math

import numpy as np
import torch

import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import autograd as nd_autograd

# Permalloy-like material of the paper's simulations
A_EX, MS, GAMMA, A_CELL = 1.3e-11, 8.6e5, 1.76e11, 2.0e-9
MU0, KB = 4.0e-7 * math.pi, 1.380649e-23
LAMBDA = math.sqrt(2.0 * A_EX / (MU0 * MS * MS))
CFAC = (A_CELL / LAMBDA) ** 2
B0 = 2.0 * A_EX / (A_CELL ** 2 * MS)
DT_HEUN, DT_RK4 = 1e-14, 5e-15

DEFAULTS = dict(kind="heun", R=50.0, L=10.0, replicas=1, fp64=False, steps=50, T=300.0, alpha=0.01, hy=0.0, plan=-1,
                grid3x=False, tol=1e-5, disks=0)


def _case(name=None, **kw):
    c = dict(DEFAULTS, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one effective field of the paper's smallest disk: the latency of the smallest call (the
        # backward of the energy, field maps, the smoke test)
        _case("field_r30", kind="field", L=5.0, R=30.0, hy=1e4),
        # energy with autograd: FP64 energies, the gradient for the state and for the thickness, at the
        # sixteen core positions of a k_F map
        _case("energy_grad_r60_x16", kind="energy", R=60.0, L=10.0, replicas=16),
        # what is read off a thermal ensemble every sampling interval: core positions and <m>
        _case("observe_r50_x256", kind="observe", replicas=256),
        # the energy-conservation run: one disk in FP64, undamped RK4, dt = 5 fs
        _case("rk4_r30_fp64", kind="rk4", R=30.0, L=5.0, fp64=True, alpha=0.0, plan=200),
        # gyrotropic dynamics released from the sixteen relaxed core positions, RK4 with damping
        _case("rk4_r60_x16", kind="rk4", R=60.0, L=10.0, replicas=16),
        # a single thermal disk, on the plan the autotuner picks for it
        _case("heun_r50_x1", plan=201),
        # the batched Langevin ensemble: 256 thermal replicas of one disk
        _case("heun_r50_x256", replicas=256),
        # an odd grid of medium size: D = 121 on the 256 grid, a few dozen replicas
        _case("heun_r121_x24", R=121.0, L=20.0, replicas=24, steps=20),
        # the large-disk throughput run: D = 500 on the 1024 grid
        _case("heun_r500_x8", R=500.0, L=20.0, replicas=8, steps=20),
        # the uneven batch: 64 disks of R = 20..100 nm, RK4 at T = 0 and Heun otherwise, one joined graph
        _case("graph_uneven64", kind="graph", disks=64),
        # the k_F map: constrained relaxations at sixteen core positions of one disk
        _case("relax_r60_x16", kind="relax", R=60.0, L=10.0, replicas=16),
        # a geometry sweep in FP64, whose k_F is a difference of energies: two core positions per disk, one disk
        # of each size class
        _case("relax_sweep3_fp64", kind="relax", disks=3, replicas=2, fp64=True, tol=3e-5),
    ]


def draw(rng):
    def logu(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["field", "energy", "observe", "rk4", "heun", "heun", "heun", "relax", "graph"])
    if kind == "graph":
        return _case(kind=kind, disks=rng.randint(8, 64), steps=rng.randint(5, 50))
    fp64 = kind in ("field", "rk4", "heun", "relax") and rng.random() < 0.2
    dmax = (60 if fp64 else 80) if kind == "relax" else 200 if fp64 or kind == "energy" else 500
    R = round(logu(13.0, dmax), 1)
    C = math.pi * (R / 2) ** 2
    most = 16 if kind == "relax" or fp64 else 256
    reps = max(1, int(logu(1.0, max(1.0, min(most, 8 * 196364 / C)))))
    c = _case(kind=kind, R=R, L=round(R * rng.uniform(0.05, 0.3), 1), replicas=reps, fp64=fp64,
              T=round(rng.uniform(0.0, 400.0), 1), alpha=round(rng.uniform(0.0, 0.1), 3),
              hy=rng.choice([0.0, 1e4]), grid3x=rng.random() < 0.3)
    if kind in ("rk4", "heun"):
        c["steps"] = int(logu(2.0, 50.5))
        P = _padded(_grid(R))
        if reps <= 4 and 32 <= P <= 128 and rng.random() < 0.5:
            c["plan"] = rng.choice([200, 201])
        # no dearer than the large-disk run (FP64 arithmetic is far slower here)
        top = 5e11
        while c["steps"] > 1 and work(c)["flops"] * (30 if fp64 else 4 if P > 128 else 1) > top:
            c["steps"] //= 2
    return c


# ------------------------------------------------------------------ inputs

def _grid(R):
    return int(math.floor(2.0 * R * 1e-9 / A_CELL + 0.5))


def _padded(D):
    P = 16
    while P < 2 * D - 1:
        P *= 2
    return P


def _disks(case, seed):
    """[(R, L, T, replicas)] in SI units, in two groups for a graph: T = 0 first."""
    if not case["disks"]:
        return [(case["R"] * 1e-9, case["L"] * 1e-9, case["T"], case["replicas"])]
    n = case["disks"]
    if case["kind"] == "relax":
        R = np.linspace(30.0, 100.0, n)
        return [(r * 1e-9, max(5.0, 0.1 * r) * 1e-9, 0.0, case["replicas"]) for r in R]
    # the sizes are the case's own, drawn once; the states and the noise come from the seed
    rng = np.random.default_rng(0)
    R = rng.uniform(20e-9, 100e-9, n)
    L = R * rng.uniform(0.05, 0.2, n)
    T = rng.uniform(1.0, 400.0, n)
    T[:max(1, n // 8)] = 0.0
    return [(float(R[k]), float(L[k]), float(T[k]), 1) for k in range(n)]


def _mask(D, R):
    i = torch.arange(D, dtype=torch.float64, device="cuda") - 0.5 * (D - 1)
    return i[None, :] ** 2 + i[:, None] ** 2 <= (R / A_CELL) ** 2


def _cores(case, seed, n, R):
    """Core positions of n replicas in metres: a k_F map along x (relax), else scattered near the centre."""
    rng = np.random.default_rng([seed, n, int(R * 1e12)])
    if case["kind"] == "relax":
        x = np.arange(n) * (0.5 * R / 16) + rng.uniform(0.0, 1e-9, n)
        return np.stack([x, np.zeros(n)], 1)
    return rng.uniform(-0.1 * R, 0.1 * R, (n, 2))


def _states(case, seed, n, R, L, T):
    """[n, 3, D, D] FP64 on the GPU: the vortex profile with, in a dynamic run, thermal tilts of its cells."""
    D = int(math.floor(2.0 * R / A_CELL + 0.5))
    X = torch.from_numpy(_cores(case, seed, n, R)).cuda() / A_CELL
    i = torch.arange(D, dtype=torch.float64, device="cuda") - 0.5 * (D - 1)
    dx, dy = i[None, None, :] - X[:, 0, None, None], i[None, :, None] - X[:, 1, None, None]
    mz = torch.exp(-(dx * dx + dy * dy) * (A_CELL / LAMBDA) ** 2).expand(n, D, D)
    phi = torch.atan2(dy, dx).expand(n, D, D) + 0.5 * math.pi
    sp = torch.sqrt(1.0 - mz * mz)
    m = torch.stack([sp * torch.cos(phi), sp * torch.sin(phi), mz], 1)
    if case["kind"] != "relax":
        g = torch.Generator(device="cuda").manual_seed(seed * 1009 + D)
        tilt = 0.02 + math.sqrt(0.5 * KB * T / (2.0 * A_EX * L))
        m = m + tilt * torch.randn(m.shape, generator=g, dtype=torch.float64, device="cuda")
        m = m / m.norm(dim=1, keepdim=True)
    return m * _mask(D, R)


def _noise_seeds(seed, n):
    return (np.arange(n, dtype=np.uint64) + np.uint64(1000003 * (seed % 100000))).astype(np.uint64)


class _Graph:
    """One joined graph and what it replays."""

    def __init__(self, parts, handles):
        self.parts, self.handles = parts, handles
        self.g = nd.nd_graph_join(parts)

    def __del__(self):
        try:
            nd.nd_graph_destroy(self.g)
            for p in self.parts:
                nd.nd_graph_destroy(p)
        except Exception:
            pass


def _handle(case, disks, seed):
    """A handle over the disks, its packed initial state and the cores of its replicas."""
    h = nd.Nanodisk([nd.Disk(R, L, alpha=case["alpha"], hext=(0.0, case["hy"], 0.0)) for R, L, _, _ in disks],
                    [d[3] for d in disks], nd.ND_FP64 if case["fp64"] else nd.ND_FP32, grid3x=case["grid3x"])
    m0 = h.empty_device()
    r, X = 0, []
    for k, (R, L, T, n) in enumerate(disks):
        lay = h.layout[r]
        D, Dp, off = lay["D"], lay["Dpad"], lay["offset"]
        m0[off:off + n * 3 * D * Dp].view(n, 3, D, Dp)[..., :D] = _states(case, seed + k, n, R, L, T).to(m0.dtype)
        X.append(_cores(case, seed + k, n, R))
        r += n
    return h, m0, np.concatenate(X)


def prepare(case, seed):
    case = dict(DEFAULTS, **case)
    disks = _disks(case, seed)
    if case["kind"] == "graph":
        st = {"case": case, "parts": []}
        graphs = []
        for cold in (True, False):
            grp = [d for d in disks if (d[2] == 0.0) == cold]
            h, m0, _ = _handle(case, grp, seed + (0 if cold else 500))
            m = m0.clone()
            meth = nd.ND_METHOD_RK4 if cold else nd.ND_METHOD_HEUN
            T = np.array([d[2] for d in grp])
            graphs.append(nd.nd_graph_create(h.h, m, meth, case["steps"], DT_HEUN, T, _noise_seeds(seed, h.B)))
            st["parts"].append((h, m0, m))
        st["graph"] = _Graph(graphs, [p[0] for p in st["parts"]])
        return st
    h, m0, X = _handle(case, disks, seed)
    st = {"case": case, "h": h, "m0": m0, "X": X}
    if case["kind"] in ("rk4", "heun") and case["plan"] >= 0:
        nd.nd_set_plan(h.h, 0, nd.ND_METHOD_RK4 if case["kind"] == "rk4" else nd.ND_METHOD_HEUN, case["plan"])
    st["T"] = np.full(h.B, case["T"])
    st["seeds"] = _noise_seeds(seed, h.B)
    if case["kind"] == "field":
        st["b"] = h.empty_device()
    if case["kind"] == "energy":
        st["Lt"] = torch.tensor(h.disks[0].L, dtype=torch.float64)
    return st


def run(state):
    """One pass.  Steppers and relaxations work in place, so each pass starts from a copy of the prepared
    state, as the members of an ensemble start from one relaxed state."""
    case = state["case"]
    kind = case["kind"]
    if kind == "graph":
        for _, m0, m in state["parts"]:
            m.copy_(m0)
        nd.nd_graph_launch(state["graph"].g)
        return [m for _, _, m in state["parts"]]
    h, m0 = state["h"], state["m0"]
    if kind == "field":
        return h.field(m0, state["b"])
    if kind == "energy":
        m = m0.detach().requires_grad_(True)
        L = state["Lt"].detach().requires_grad_(True)
        E = nd_autograd.energy(m, L, h)
        gm, gL = torch.autograd.grad(E.sum(), (m, L))
        return {"E": E, "gm": gm, "gL": gL}
    if kind == "observe":
        Xc, _ = h.vortex_core(m0)
        return {"core": Xc, "mean": h.mean_m(m0)}
    m = m0.clone()
    if kind == "rk4":
        h.rk4(m, case["steps"], DT_RK4)
        return m
    if kind == "heun":
        h.heun(m, case["steps"], DT_HEUN, state["T"], state["seeds"])
        return m
    # relax: the state and its energies, these in the precision of the state they belong to; the multipliers,
    # which a single-precision relaxation stopped at its tolerance does not pin down, in FP64 only
    _, U, lam, _ = h.relax(m, state["X"], tol=case["tol"])
    out = {"m": m, "U": torch.from_numpy(U).to(m.dtype)}
    if case["fp64"]:
        out["lam"] = torch.from_numpy(lam)
    return out


# -------------------------------------------------------------------- work

RELAX_SWEEPS = 5000   # order of magnitude of the sweeps of one relaxation at these tolerances


def work(case):
    """Bytes: states in and out, and the spectral kernel's four real entries once per disk.  Operations: the
    pruned transforms (D of the P rows hold data), the spectral multiply and 60 per cell, per evaluation."""
    case = dict(DEFAULTS, **case)
    kind, elt = case["kind"], 8 if case["fp64"] else 4
    nbytes = flops = 0.0
    for R, L, T, n in _disks(case, 0):
        D = int(math.floor(2.0 * R / A_CELL + 0.5))
        P, C = _padded(D), math.pi * (R / A_CELL) ** 2
        lg, kh = math.log2(P), P // 2 + 1
        ev = 2 * 3 * D * 2.5 * P * lg + 2 * 3 * kh * 5.0 * P * lg + 14.0 * P * kh + 60.0 * C
        state, table = 3.0 * C * elt, 4.0 * kh * kh * elt
        if kind == "observe":
            nbytes += n * state
            flops += n * 30.0 * C
            continue
        if kind == "graph":
            evals = case["steps"] * (4 if T == 0.0 else 2)
        else:
            evals = {"field": 1, "energy": 3, "rk4": 4 * case["steps"], "heun": 2 * case["steps"],
                     "relax": RELAX_SWEEPS}[kind]
        nbytes += 2 * n * state + table
        flops += n * ev * evals
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------- the same in 64 bits

class _Model:
    """The paper's equations for n states of one disk in FP64: Sec. II.B's thin-film tensor as an FFT
    convolution, the exchange with neighbours inside the disk, Eqs. Bi, Hmm, LV and the constrained
    relaxation of Sec. IV as include/nanodisk.h states it."""

    def __init__(self, R, L, alpha, hy):
        self.R, self.L, self.alpha = R, L, alpha
        self.D = D = int(math.floor(2.0 * R / A_CELL + 0.5))
        self.P = _padded(D)
        self.mask = _mask(D, R)
        self.J = 2.0 * A_EX * L
        self.h = torch.tensor([0.0, hy / MS, 0.0], dtype=torch.float64, device="cuda")
        self.Ghat = self.tensor(torch.tensor(L / A_CELL, dtype=torch.float64, device="cuda"))

    def tensor(self, l):
        """Spectra of a^2 G (xx, yy, xy, zz) on the padded grid; l = L/a may require grad."""
        P = self.P
        d = torch.arange(P, dtype=torch.float64, device="cuda")
        d = torch.where(d > P / 2, d - P, d)
        x, y = torch.broadcast_tensors(d[None, :], d[:, None])
        self0 = (x == 0) & (y == 0)
        x, y = torch.where(self0, torch.ones_like(x), x), torch.where(self0, torch.ones_like(y), y)
        r2 = x * x + y * y
        r, s = r2.sqrt(), (r2 + l * l).sqrt()
        pre = l / (2.0 * math.pi * r2 * r2)
        ro = 1.0 / math.sqrt(math.pi)
        q = (l * l + ro * ro).sqrt()
        nz, nx = (l + ro - q) / l, (q - ro) / (2.0 * l)
        xx = torch.where(self0, -nx, pre * (x * x / s - y * y / (s + r)))
        yy = torch.where(self0, -nx, pre * (y * y / s - x * x / (s + r)))
        xy = torch.where(self0, torch.zeros_like(x), pre * ((2.0 * s + r) / (s + r)) * (x * y / s))
        zz = torch.where(self0, -nz, -l / (2.0 * math.pi * r * s * (s + r)))
        # displacements beyond D - 1 never meet a cell pair
        far = (d.abs() > self.D - 1)
        keep = ~(far[None, :] | far[:, None])
        return [torch.fft.rfft2(torch.where(keep, g, torch.zeros_like(g))) for g in (xx, yy, xy, zz)]

    def demag(self, m, G=None):
        D, P = self.D, self.P
        gxx, gyy, gxy, gzz = G or self.Ghat
        f = torch.fft.rfft2(m, s=(P, P))
        h = torch.stack([gxx * f[:, 0] + gxy * f[:, 1], gxy * f[:, 0] + gyy * f[:, 1], gzz * f[:, 2]], 1)
        return torch.fft.irfft2(h, s=(P, P))[..., :D, :D]

    def exchange(self, m):
        e = torch.zeros_like(m)
        e[..., 1:, :] += m[..., :-1, :]
        e[..., :-1, :] += m[..., 1:, :]
        e[..., :, 1:] += m[..., :, :-1]
        e[..., :, :-1] += m[..., :, 1:]
        return e

    def field(self, m):
        b = self.exchange(m) + CFAC * (self.h[None, :, None, None] + self.demag(m))
        return b * self.mask

    def energy(self, m, G=None):
        """E/J of Eq. Hmm."""
        e = 0.5 * self.exchange(m) + CFAC * (self.h[None, :, None, None] + 0.5 * self.demag(m, G))
        return -(e * m).sum((1, 2, 3))


def _cross(a, b):
    return torch.stack([a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1], a[:, 2] * b[:, 0] - a[:, 0] * b[:, 2],
                        a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]], 1)


def _unit(v):
    return v / torch.where(v.norm(dim=1, keepdim=True) > 0, v.norm(dim=1, keepdim=True), torch.ones(1, 1, 1, 1, dtype=v.dtype, device=v.device))


def _rk4(mod, m, steps, dtau):
    def f(u):
        p = _cross(u, mod.field(u))
        return p - mod.alpha * _cross(u, p)

    for _ in range(steps):
        k1 = f(m)
        k2 = f(m + 0.5 * dtau * k1)
        k3 = f(m + 0.5 * dtau * k2)
        k4 = f(m + dtau * k3)
        m = _unit(m + dtau / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4))
    return m


def _philox(cells, step, seeds):
    """Philox4x32-10 words [4][n][cells] for counter (cell, step, 0, 0) and key = seed."""
    M = 0xFFFFFFFF
    c = [cells[None, :].expand(len(seeds), -1), torch.full_like(cells, step)[None, :], torch.zeros_like(cells)[None, :],
         torch.zeros_like(cells)[None, :]]
    k0, k1 = (seeds & M)[:, None], ((seeds >> 32) & M)[:, None]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & M) ^ c[1] ^ k0, p1 & M, ((p0 >> 32) & M) ^ c[3] ^ k1, p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c


def _heun(mod, m, steps, dtau, T, seeds):
    D = mod.D
    sigma = math.sqrt(2.0 * mod.alpha * (KB * T / mod.J) * dtau)
    cells = torch.arange(D * D, device="cuda")
    keys = torch.from_numpy(seeds.astype(np.int64)).cuda()

    def dm(u, w):
        g = mod.field(u) * dtau + sigma * w
        return _cross(u, g - mod.alpha * _cross(u, g))

    for n in range(steps):
        w = torch.zeros_like(m)
        if sigma > 0:
            r = [v.double() for v in _philox(cells, n, keys)]
            ra, rb = torch.sqrt(-2.0 * torch.log((r[0] + 1) / 2 ** 32)), torch.sqrt(-2.0 * torch.log((r[2] + 1) / 2 ** 32))
            a1, a3 = 2.0 * math.pi * r[1] / 2 ** 32, 2.0 * math.pi * r[3] / 2 ** 32
            w = torch.stack([ra * torch.cos(a1), ra * torch.sin(a1), rb * torch.cos(a3)], 1).view_as(m) * mod.mask
        d1 = dm(m, w)
        d2 = dm(_unit(m + d1), w)
        m = _unit(m + 0.5 * (d1 + d2))
    return m


def _relax(mod, m, X, tol, max_iter=20000, eta=0.5):
    n, D = m.shape[0], mod.D
    i = torch.arange(D, dtype=torch.float64, device="cuda") - 0.5 * (D - 1)
    Xc = torch.from_numpy(X).cuda() / A_CELL
    dx, dy = torch.broadcast_tensors(i[None, None, :] - Xc[:, 0, None, None], i[None, :, None] - Xc[:, 1, None, None])
    win = ((dx * dx + dy * dy) < (4.0 * LAMBDA / A_CELL) ** 2) & mod.mask
    wx, wy = dx * win, dy * win
    lam = torch.zeros(n, 2, dtype=torch.float64, device="cuda")
    one = torch.ones((), dtype=torch.float64, device="cuda")

    def align(lam):
        e = b.clone()
        e[:, 2] += 2.0 * m[:, 2] * (lam[:, 0, None, None] * wx + lam[:, 1, None, None] * wy)
        en = torch.where(mod.mask, e.norm(dim=1), one)
        u = e / en[:, None]
        v = (1.0 - eta) * m + eta * u
        vn = torch.where(mod.mask, v.norm(dim=1), one)
        return u, en, v / vn[:, None], vn

    run_ = torch.ones(n, dtype=torch.bool, device="cuda")
    for it in range(max_iter):
        b = mod.field(m)
        u, en, mp, vn = align(lam)
        res = (_cross(m, u).norm(dim=1) * mod.mask).amax((1, 2))
        run_ = run_ & ~(res < tol)
        if it % 8 == 0 and not bool(run_.any()):
            break
        q = torch.stack([-u[:, 0] * u[:, 2], -u[:, 1] * u[:, 2], 1.0 - u[:, 2] ** 2], 1) / en[:, None]
        kap = eta * (q[:, 2] - mp[:, 2] * (mp * q).sum(1)) / vn
        w = 4.0 * mp[:, 2] * m[:, 2] * kap
        z2 = mp[:, 2] ** 2
        c0, c1 = (z2 * wx).sum((1, 2)), (z2 * wy).sum((1, 2))
        j00, j01, j11 = (w * wx * wx).sum((1, 2)), (w * wx * wy).sum((1, 2)), (w * wy * wy).sum((1, 2))
        det = j00 * j11 - j01 * j01
        step = torch.stack([-(j11 * c0 - j01 * c1) / det, -(j00 * c1 - j01 * c0) / det], 1)
        lam = torch.where(run_[:, None], lam + step, lam)
        m = torch.where(run_[:, None, None, None], align(lam)[2] * mod.mask, m)
    return m, lam


def _core(mod, m):
    """Core centroid of Sec. IV: m_z^2-weighted over the disk cells within 4 lambda of the winding +1 plaquette."""
    D = mod.D
    phi = torch.atan2(m[:, 1], m[:, 0])
    ring = [phi[:, :-1, :-1], phi[:, :-1, 1:], phi[:, 1:, 1:], phi[:, 1:, :-1]]
    wind = sum(torch.remainder(ring[(k + 1) % 4] - ring[k] + math.pi, 2.0 * math.pi) - math.pi for k in range(4))
    mk = mod.mask
    ok = (wind / (2.0 * math.pi)).round() == 1
    ok &= mk[:-1, :-1] & mk[:-1, 1:] & mk[1:, 1:] & mk[1:, :-1]
    z2 = m[:, 2] ** 2
    score = torch.where(ok, z2[:, :-1, :-1] + z2[:, :-1, 1:] + z2[:, 1:, :-1] + z2[:, 1:, 1:], torch.full((), -1.0, dtype=m.dtype, device=m.device))
    best = score.flatten(1).argmax(1)
    i = torch.arange(D, dtype=torch.float64, device="cuda") - 0.5 * (D - 1)
    cx, cy = i[best % (D - 1)] + 0.5, i[best // (D - 1)] + 0.5
    near = ((i[None, None, :] - cx[:, None, None]) ** 2 + (i[None, :, None] - cy[:, None, None]) ** 2) < (4.0 * LAMBDA / A_CELL) ** 2
    w = z2 * (near & mk)
    tot = w.sum((1, 2))
    return torch.stack([(w * i[None, None, :]).sum((1, 2)) / tot, (w * i[None, :, None]).sum((1, 2)) / tot], 1) * A_CELL


def _packed(grids):
    """[n, 3, D, D] per disk -> one flat buffer with rows padded to multiples of four."""
    out = []
    for g in grids:
        D = g.shape[-1]
        out.append(torch.nn.functional.pad(g, (0, (D + 3) // 4 * 4 - D)).reshape(-1))
    return torch.cat(out)


def exact(case, seed):
    case = dict(DEFAULTS, **case)
    kind = case["kind"]
    dt = torch.float64 if case["fp64"] else torch.float32
    dtau = GAMMA * B0 * (DT_RK4 if kind == "rk4" else DT_HEUN)
    disks = _disks(case, seed)
    if kind == "graph":
        outs = []
        for cold in (True, False):
            grp, res = [d for d in disks if (d[2] == 0.0) == cold], []
            keys = _noise_seeds(seed, len(grp))
            for k, (R, L, T, n) in enumerate(grp):
                mod = _Model(R, L, case["alpha"], case["hy"])
                m = _states(case, seed + (0 if cold else 500) + k, n, R, L, T).to(dt).double()
                res.append(_rk4(mod, m, case["steps"], dtau) if cold else _heun(mod, m, case["steps"], dtau, T, keys[k:k + 1]))
            outs.append(_packed(res))
        return outs
    ms, Us, lams = [], [], []
    for k, (R, L, T, n) in enumerate(disks):
        mod = _Model(R, L, case["alpha"], case["hy"])
        m = _states(case, seed + k, n, R, L, T).to(dt).double()
        if kind == "field":
            return _packed([mod.field(m)])
        if kind == "energy":
            l = torch.tensor(L / A_CELL, dtype=torch.float64, device="cuda", requires_grad=True)
            E = 2.0 * A_EX * A_CELL * l * mod.energy(m, mod.tensor(l))
            (gl,) = torch.autograd.grad(E.sum(), l)
            return {"E": E.detach(), "gm": _packed([-mod.J * mod.field(m)]), "gL": gl / A_CELL}
        if kind == "observe":
            return {"core": _core(mod, m), "mean": (m * mod.mask).sum((2, 3)) / mod.mask.sum()}
        if kind == "rk4":
            return _packed([_rk4(mod, m, case["steps"], dtau)])
        if kind == "heun":
            return _packed([_heun(mod, m, case["steps"], dtau, T, _noise_seeds(seed, n))])
        m, lam = _relax(mod, m, _cores(case, seed + k, n, R), case["tol"])
        ms.append(m)
        lams.append(lam)
        Us.append(mod.energy(m))
    out = {"m": _packed(ms), "U": torch.cat(Us)}
    if case["fp64"]:
        out["lam"] = torch.cat(lams)
    return out
