"""The calls that a user of the SCF gravity library makes, at the sizes that they make them.

A case is one call of the public API (``paper_2602_13385_gb300.SCF`` or
``adjoint.run``) on a cluster sample: leapfrog steps on device or host memory,
the boundedness sums of a refresh, an evolution with refreshes, the
coefficients or the field alone, and a differentiable run.  Samples are
Plummer or King (1966) spheres in Henon units (G = M = 1) drawn on the GPU
from the seed, the hosts those of App. A; the sizes are those of the
workloads in ``workloads/`` and of ``tests/``.

``exact`` is the textbook form of the same quantities in 64 bits: the radial
basis by the unscaled Gegenbauer recurrence, the field as the gradient of the
potential by automatic differentiation.
"""
from __future__ import annotations

import contextlib
import math

import numpy as np
import torch

from paper_2602_13385_gb300 import SCF, Config, adjoint

DEV = "cuda"
RV_PC = 4.0                # length unit of the clusters (pc) for the host in cluster units
M_MSUN = 1.0e5             # mass unit
HERNQUIST, NFW, MN, POWCUT = 1, 2, 3, 4

# (kind, mass in Msun, scale length in pc, second parameter: pc, or the index of the cut-off bulge)
HOSTS = {
    "none": [],
    # NFW halo, Miyamoto-Nagai disk, Hernquist bulge
    "galaxy": [(NFW, 6.6e11, 20.0e3, 0.0), (MN, 6.8e10, 3.0e3, 280.0), (HERNQUIST, 5.0e9, 500.0, 0.0)],
    # two Hernquist bulges, a disk of three Miyamoto-Nagai parts, NFW halo
    "mw2022": [(HERNQUIST, 1.8142e9, 68.8867, 0.0), (HERNQUIST, 5.0e9, 1.0e3, 0.0),
               (MN, 7.8723e9, 1525.9, 206.637), (MN, -2.75625e11, 6782.8, 206.637), (MN, 3.206184e11, 5894.8, 206.637),
               (NFW, 5.5427e11, 15626.0, 0.0)],
}


def listed():
    big = {"nmax": 20, "lmax": 10, "alpha": 1.0}
    stream = {"nmax": 10, "lmax": 5, "alpha": 1.0}
    return [
        # the isolated validation cluster: the smallest step, launches and latency
        {"name": "step_4096_fp64", "do": "step", "n": 4096, "n_prog": 1, "nmax": 10, "lmax": 6, "alpha": 1.0,
         "precision": "fp64", "model": "plummer", "host": "none", "tail": 0.0},
        # a typical production cluster in the paper's precision
        {"name": "step_100000_fp64", "do": "step", "n": 100_000, "n_prog": 1, "nmax": 20, "lmax": 8, "alpha": 1.0,
         "precision": "fp64", "model": "king", "host": "galaxy", "tail": 0.0},
        # the largest cluster, both precisions
        {"name": "step_1000000_fp64", "do": "step", "n": 1_000_000, "n_prog": 1, **big, "precision": "fp64",
         "model": "plummer", "host": "galaxy", "tail": 0.0},
        {"name": "step_1000000_mixed", "do": "step", "n": 1_000_000, "n_prog": 1, **big, "precision": "mixed",
         "model": "plummer", "host": "galaxy", "tail": 0.0},
        # ten clusters of uneven sizes in one batch
        {"name": "step_batch10_mixed", "do": "step", "n": 1_909_153, "n_prog": 10, **big, "precision": "mixed",
         "model": "king", "host": "galaxy", "tail": 0.0},
        # the paper's stream progenitors on its ten orbits, already losing stars
        {"name": "step_orbits10_mixed", "do": "step", "n": 2_000_000, "n_prog": 10, **stream, "precision": "mixed",
         "model": "king", "host": "mw2022", "tail": 0.03},
        # a ragged cluster in the Clutton-Brock member of the radial family
        {"name": "step_314159_cb_mixed", "do": "step", "n": 314_159, "n_prog": 1, "nmax": 20, "lmax": 10, "alpha": 0.5,
         "precision": "mixed", "model": "plummer", "host": "galaxy", "tail": 0.0},
        # the state kept in host memory between steps
        {"name": "hoststep_1000000_mixed", "do": "hoststep", "n": 1_000_000, "n_prog": 1, **big, "precision": "mixed",
         "model": "plummer", "host": "galaxy", "tail": 0.0},
        # the direct sums of a refresh, in both precisions
        {"name": "bound_100000_fp64", "do": "bound", "n": 100_000, "n_prog": 1, **stream, "precision": "fp64",
         "model": "king", "host": "galaxy", "tail": 0.03},
        {"name": "bound_batch10_mixed", "do": "bound", "n": 1_000_003, "n_prog": 10, **stream, "precision": "mixed",
         "model": "king", "host": "galaxy", "tail": 0.03},
        # a stream-forming cluster run through its refreshes
        {"name": "evolve_100000_mixed", "do": "evolve", "n": 100_000, "n_prog": 1, **stream, "precision": "mixed",
         "model": "plummer", "host": "galaxy", "tail": 0.03, "nsteps": 100},
        # a differentiable run: forward, recomputation and adjoint sweep
        {"name": "adjoint_20000_fp64", "do": "adjoint", "n": 20_000, "n_prog": 1, "nmax": 20, "lmax": 8, "alpha": 1.0,
         "precision": "fp64", "model": "king", "host": "galaxy", "tail": 0.0, "nsteps": 4},
    ]


def draw(rng):
    do = rng.choice(["step", "step", "step", "step", "hoststep", "coeffs", "forces", "bound", "evolve", "adjoint"])
    nmax, lmax = rng.choice([(10, 5), (10, 6), (20, 8), (20, 10)])
    top = {"bound": 2e5, "evolve": 2e5, "adjoint": 3e4}.get(do, 1e6)
    n = int(round(math.exp(rng.uniform(math.log(3e3), math.log(top)))))
    case = {"do": do, "n": n + rng.randrange(2), "n_prog": 1, "nmax": nmax, "lmax": lmax, "alpha": 1.0,
            "precision": rng.choice(["fp64", "mixed"]), "model": rng.choice(["plummer", "king"]),
            "host": rng.choice(["galaxy", "galaxy", "mw2022", "none"]), "tail": rng.choice([0.0, 0.03])}
    if do not in ("adjoint",) and rng.random() < 0.4:
        case["n_prog"] = rng.randrange(2, 11)
        case["n"] += 2000 * case["n_prog"]
    if do in ("step", "coeffs", "forces") and rng.random() < 0.25:
        case["alpha"] = 0.5
    if do in ("evolve", "adjoint"):
        case["nsteps"] = rng.randrange(20, 101) if do == "evolve" else rng.randrange(2, 6)
    if do == "adjoint":
        case["precision"], case["host"] = "fp64", "galaxy"
    return case


# --------------------------------------------------------------------------
# samples
# --------------------------------------------------------------------------
def offsets_of(case):
    """Progenitor boundaries: sizes spread by a factor of 25 in a batch (equal for the ten-orbit stream model)."""
    k, n = case["n_prog"], case["n"]
    if k == 1:
        return [0, n]
    ratio = 25.0 if (case["nmax"], case["lmax"]) != (10, 5) else 1.0
    w = np.array([ratio ** (((7 * i) % k) / (k - 1)) for i in range(k)])
    return [int(x) for x in np.round(np.concatenate([[0.0], np.cumsum(w)]) / w.sum() * n)]


def isotropic(n, g):
    u = 2.0 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64) - 1.0
    ph = 2.0 * math.pi * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    s = torch.sqrt(1.0 - u * u)
    return torch.stack([s * torch.cos(ph), s * torch.sin(ph), u], dim=1)


def reject(n, g, top, pdf):
    """Samples x in [0, top_i] of the unnormalised densities pdf(x, i) <= 1."""
    x = torch.empty(n, device=DEV, dtype=torch.float64)
    todo = torch.arange(n, device=DEV)
    while todo.numel():
        y = torch.rand(todo.numel(), generator=g, device=DEV, dtype=torch.float64) * top[todo]
        ok = torch.rand(todo.numel(), generator=g, device=DEV, dtype=torch.float64) < pdf(y, todo)
        x[todo[ok]] = y[ok]
        todo = todo[~ok]
    return x


def plummer(n, g):
    """Plummer sphere of scale 3 pi / 16, cut at 22.8 scales; speeds q = v / v_esc from q^2 (1 - q^2)^(7/2)."""
    a = 3.0 * math.pi / 16.0
    cut = (1.0 + 22.8 ** -2) ** -1.5
    x = cut * torch.rand(n, generator=g, device=DEV, dtype=torch.float64).clamp_min(1e-12)
    r = 1.0 / torch.sqrt(x ** (-2.0 / 3.0) - 1.0)
    one = torch.ones(n, device=DEV, dtype=torch.float64)
    q = reject(n, g, one, lambda y, i: y * y * (1.0 - y * y) ** 3.5 / 0.1)
    v = q * math.sqrt(2.0 / a) * (1.0 + r * r) ** -0.25
    return a * r, v


_KING = {}


def king_table(W0):
    """King (1966) model: r, W, enclosed mass (r0 = sigma = G = 1), by fourth-order Runge-Kutta on W'' + 2 W'/r = -9 rho/rho0."""
    if W0 in _KING:
        return _KING[W0]

    def rho(W):
        W = max(W, 0.0)
        return math.exp(W) * math.erf(math.sqrt(W)) - math.sqrt(4.0 * W / math.pi) * (1.0 + 2.0 * W / 3.0)

    rho0 = rho(W0)

    def slope(r, W, d):
        return d, -9.0 * rho(W) / rho0 - 2.0 * d / r

    r, W, d = 1e-4, W0 - 1.5e-8, -3e-4
    rs, Ws, Ms = [0.0, r], [W0, W], [0.0, 3e-12]
    while W > 0.0:
        h = 0.01 * (0.1 + r)
        k1 = slope(r, W, d)
        k2 = slope(r + h / 2, W + h / 2 * k1[0], d + h / 2 * k1[1])
        k3 = slope(r + h / 2, W + h / 2 * k2[0], d + h / 2 * k2[1])
        k4 = slope(r + h, W + h * k3[0], d + h * k3[1])
        r, W, d = r + h, W + h / 6 * (k1[0] + 2 * k2[0] + 2 * k3[0] + k4[0]), d + h / 6 * (k1[1] + 2 * k2[1] + 2 * k3[1] + k4[1])
        rs.append(r)
        Ws.append(max(W, 0.0))
        Ms.append(max(-r * r * d, Ms[-1]))
    _KING[W0] = tuple(np.array(t) for t in (rs, Ws, Ms))
    return _KING[W0]


def interp(x, xp, fp):
    i = torch.searchsorted(xp, x).clamp(1, xp.numel() - 1)
    t = (x - xp[i - 1]) / (xp[i] - xp[i - 1]).clamp_min(1e-300)
    return fp[i - 1] + t * (fp[i] - fp[i - 1])


def king(n, W0, g):
    rs, Ws, Ms = king_table(W0)
    M = Ms[-1]
    U = -np.sum(0.5 * (Ms[1:] + Ms[:-1]) * np.diff(Ms) / np.maximum(0.5 * (rs[1:] + rs[:-1]), 1e-30))
    L = M * M / (2.0 * abs(U))           # model length of a Henon unit: U = -M^2 / (2 L)
    tr, tW, tM = (torch.tensor(t, device=DEV, dtype=torch.float64) for t in (rs, Ws, Ms))
    r = interp(torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * M, tM, tr)
    W = interp(r, tr, tW)
    top = torch.sqrt(2.0 * W)
    env = torch.minimum(top * top, torch.full_like(top, 2.0 / math.e)) * torch.exp(W)

    def pdf(y, i):
        return y * y * (torch.exp(W[i] - 0.5 * y * y) - 1.0) / env[i].clamp_min(1e-300)
    v = reject(n, g, top, pdf) if n else top
    return r / L, v * math.sqrt(L / M)


def sample(case, seed):
    """(pos, vel) float64 (n, 4) on the GPU, and the half-mass radius of each progenitor."""
    off = offsets_of(case)
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * (seed % 1_000_003) + 17)
    P, V, rh = [], [], []
    for p in range(case["n_prog"]):
        n = off[p + 1] - off[p]
        r, v = plummer(n, g) if case["model"] == "plummer" else king(n, 4.0 + 4.0 * ((3 * p + 5) % 10) / 10.0, g)
        rh.append(float(r.median()))
        x, w = r[:, None] * isotropic(n, g), v[:, None] * isotropic(n, g)
        k = int(case["tail"] * n)
        if k:  # stars already stripped: two tails out to 60 half-mass radii, moving away faster than escape
            t = 3.0 * 20.0 ** torch.rand(k, generator=g, device=DEV, dtype=torch.float64)
            side = torch.where(torch.arange(k, device=DEV) % 2 == 0, 1.0, -1.0)[:, None]
            y = side * t[:, None] * torch.tensor([0.1, 1.0, 0.05], device=DEV, dtype=torch.float64)
            y = y + 0.2 * t[:, None] * isotropic(k, g)
            x[:k] = y
            w[:k] = 2.0 * y / y.norm(dim=1, keepdim=True) * torch.sqrt(1.0 / t)[:, None]
            turn = torch.randperm(n, generator=g, device=DEV)      # escapers lie anywhere in the arrays
            x, w = x[turn], w[turn]
        x = torch.cat([x - x.mean(0), torch.full((n, 1), 1.0 / max(n, 1), device=DEV, dtype=torch.float64)], 1)
        P.append(x)
        V.append(torch.cat([w - w.mean(0), torch.zeros((n, 1), device=DEV, dtype=torch.float64)], 1))
    return torch.cat(P).contiguous(), torch.cat(V).contiguous(), rh


def host_of(case):
    """Host components in the clusters' units (length RV_PC, mass M_MSUN)."""
    return [(k, M / M_MSUN, a / RV_PC, b / RV_PC) for k, M, a, b in HOSTS[case["host"]]]


def host_accel(host, x):
    """App. A accelerations (G = 1) at x (..., 3); host: (kind, M, a, b) with M, a numbers or tensors."""
    acc = torch.zeros_like(x)
    r2 = (x * x).sum(-1, keepdim=True)
    r = torch.sqrt(r2)
    for k, M, a, b in host:
        if k == HERNQUIST:
            acc = acc - M * x / (r * (r + a) ** 2)
        elif k == NFW:
            u = r / a
            acc = acc - M * x * (torch.log1p(u) - u / (1.0 + u)) / (r2 * r)
        else:
            zb = torch.sqrt(x[..., 2:] ** 2 + b * b)
            D2 = x[..., 0:1] ** 2 + x[..., 1:2] ** 2 + (zb + a) ** 2
            f = torch.cat([x[..., :2], x[..., 2:] * (1.0 + a / zb)], -1)
            acc = acc - M * f / (D2 * torch.sqrt(D2))
    return acc


def centres(case, seed):
    """(n_prog, 6) float64: centres between 8 and 20 kpc moving across the host at 0.45 to 1 of the circular speed."""
    host = host_of(case)
    if not host:
        return None
    g = np.random.default_rng(seed % (1 << 30))
    out = []
    for p in range(case["n_prog"]):
        n = g.normal(size=3)
        n /= np.linalg.norm(n)
        R = n * (8.0e3 + 12.0e3 * g.random()) / RV_PC
        t = np.cross(n, g.normal(size=3))
        t /= np.linalg.norm(t)
        aR = host_accel(host, torch.tensor(R))
        out.append(np.concatenate([R, t * (0.45 + 0.55 * g.random()) * math.sqrt(float(aR.norm()) * np.linalg.norm(R))]))
    return torch.tensor(np.array(out), device=DEV)


def scales(case, rh):
    """Basis scale of each progenitor: the lowest-order density of Eq. 4 has the sample's half-mass radius."""
    al = case["alpha"]
    return [r * (2.0 ** (1.0 / (al + 1.0)) - 1.0) ** al for r in rh]


def mask_of(case, pos):
    r2 = (pos[:, :3].double() ** 2).sum(1)
    return (r2 < 6.0 ** 2).to(torch.uint8)


# --------------------------------------------------------------------------
# the measured calls
# --------------------------------------------------------------------------
_STREAM = []


def stream():
    """The program's own stream (a captured step needs one other than the default)."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def on(case):
    return contextlib.nullcontext() if case["do"] == "adjoint" else torch.cuda.stream(stream())


def prepare(case, seed):
    pos, vel, rh = sample(case, seed)
    com = centres(case, seed)
    b = scales(case, rh)
    cfg = Config(nmax=case["nmax"], lmax=case["lmax"], b=b[0], dt=0.01, precision=case["precision"],
                 host=host_of(case), alpha=case["alpha"])
    pos, vel = pos.to(cfg.dtype).contiguous(), vel.to(cfg.dtype).contiguous()
    st = {"case": case, "pos": pos, "vel": vel, "com": com}
    torch.cuda.synchronize()
    if case["do"] == "adjoint":
        spec = adjoint.RunSpec(config=cfg, nsteps=case["nsteps"], checkpoint_every=2)
        hp = adjoint.host_params_of(cfg, device=DEV)
        st.update(spec=spec, leaves=[t.clone().requires_grad_(True) for t in (pos, vel, com[0], hp)],
                  idx=torch.arange(0, case["n"], 97, device=DEV), track=track(com[0], len(range(0, case["n"], 97))))
        return st
    with on(case):
        sim = SCF(cfg, offsets=offsets_of(case), b_per_prog=b)
        A = sim.coeffs(pos)
        acc = sim.forces(pos, A, com)
        st.update(sim=sim, acc=acc, A=A)
        if case["do"] == "coeffs":
            st["mask"] = mask_of(case, pos)
        if case["do"] == "hoststep":
            for k in ("pos", "vel", "acc", "com"):
                st["host_" + k] = None if st[k] is None else st[k].cpu().pin_memory()
    torch.cuda.synchronize()
    return st


def track(com, k):
    """The loss's target points: along the centre's motion, one for each selected star."""
    s = torch.linspace(-50.0, 50.0, k, device=DEV, dtype=torch.float64)
    t = com[3:] / com[3:].norm()
    return com[:3] + s[:, None] * t


def loss_of(pos, com, idx, target):
    P = com[:3] + pos[idx, :3]
    return ((P - target) ** 2).sum(1).mean()


def run(st):
    case, do = st["case"], st["case"]["do"]
    if do == "adjoint":
        for t in st["leaves"]:
            t.grad = None
        pos, vel, com = adjoint.run(*st["leaves"], st["spec"])
        loss_of(pos, com, st["idx"], st["track"]).backward()
        return {"pos": pos.detach(), "vel": vel.detach(), "com": com.detach(),
                **{"d_" + k: t.grad for k, t in zip(("pos", "vel", "com", "host"), st["leaves"])}}
    sim = st["sim"]
    with on(case):
        if do == "step":
            sim.step(st["pos"], st["vel"], st["acc"], st["com"])
            out = {k: st[k] for k in ("pos", "vel", "acc")}
            if case["precision"] == "fp64":
                out["A"] = sim.last_coeffs(st["A"])
        elif do == "hoststep":
            sim.step_host(st["pos"], st["vel"], st["acc"], st["host_pos"], st["host_vel"], st["host_acc"], st["com"],
                          st["host_com"])
            out = {k: st["host_" + k] for k in ("pos", "vel", "acc")}
            return out if st["host_com"] is None else dict(out, com=st["host_com"])
        elif do == "coeffs":
            # in mixed precision the sums of single-precision terms: returned as such
            A = sim.coeffs(st["pos"], mask=st["mask"], out=st["A"])
            return A if case["precision"] == "fp64" else A.float()
        elif do == "forces":
            return sim.forces(st["pos"], st["A"], st["com"], out=st["acc"])
        elif do == "bound":
            b, m, stats, E = sim.bound(st["pos"], st["vel"], energies=True)
            # in mixed precision the energies are sums of single-precision terms: returned as such
            return {"bound": b, "mask": m, "stats": stats, "E": E if case["precision"] == "fp64" else E.float()}
        else:
            b, m, stats, n_int = sim.evolve(st["pos"], st["vel"], st["acc"], st["com"], nsteps=case["nsteps"],
                                            retune_every=5, retune_rule="a000")
            out = {"pos": st["pos"], "vel": st["vel"], "acc": st["acc"], "bound": b, "mask": m, "n_int": n_int}
    return out if st["com"] is None else dict(out, com=st["com"])


def work(case):
    """Bytes: the state read once and written once.  Flops: the sums of Eqs. 1a and 3b over n, l, m (and the pair sums)."""
    off = offsets_of(case)
    rec = 32 if case["precision"] == "fp64" else 16
    n, nc = case["n"], (case["nmax"] + 1) * (case["lmax"] + 1) * (case["lmax"] + 2) // 2
    one = 12 * nc * n                        # coefficients and field: 4 and 8 flops per (n, l, m)
    if case["do"] in ("step", "hoststep"):
        return {"bytes": 6 * rec * n, "flops": one}
    if case["do"] == "coeffs":
        return {"bytes": (rec + 1) * n + 16 * nc * case["n_prog"], "flops": 4 * nc * n}
    if case["do"] == "forces":
        return {"bytes": 2 * rec * n + 16 * nc * case["n_prog"], "flops": 8 * nc * n}
    pairs = sum((off[p + 1] - off[p]) ** 2 for p in range(case["n_prog"]))
    if case["do"] == "bound":                # half of the ordered pairs: a distance, 1/r and two products each
        return {"bytes": (2 * rec + 10) * n, "flops": 6 * pairs}
    if case["do"] == "evolve":
        return {"bytes": 6 * rec * n, "flops": 6 * pairs + case["nsteps"] * one}
    return {"bytes": 10 * rec * n, "flops": 4 * case["nsteps"] * one}


# --------------------------------------------------------------------------
# the same quantities in 64 bits, from the textbook formulas
# --------------------------------------------------------------------------
def basis(x, b, case):
    """Per degree l: radial rows s^l (1+t)^(-a_l) C_n (nmax+1, N), and per m the angular rows Pb_lm cos, Pb_lm sin."""
    al, nmax, lmax = case["alpha"], case["nmax"], case["lmax"]
    r = torch.sqrt((x * x).sum(1))
    u = x / r[:, None]
    c = u[:, 2]
    s = r / b
    t = s if al == 1.0 else s ** (1.0 / al)
    xi = (t - 1.0) / (t + 1.0)
    Wc, Ws = [torch.ones_like(c)], [torch.zeros_like(c)]
    for m in range(1, lmax + 1):
        Wc.append(Wc[-1] * u[:, 0] - Ws[-1] * u[:, 1])
        Ws.append(Wc[-2] * u[:, 1] + Ws[-1] * u[:, 0])
    P = {}
    for l in range(lmax + 1):
        for m in range(l + 1):
            if l == m:
                P[l, m] = torch.full_like(c, 1.0 / math.sqrt(4.0 * math.pi)) if l == 0 else -math.sqrt((2 * l + 1) / (2 * l)) * P[l - 1, l - 1]
            elif m == l - 1:
                P[l, m] = math.sqrt(2 * l + 1) * c * P[l - 1, m]
            else:
                f = math.sqrt((4.0 * l * l - 1) / (l * l - m * m))
                h = math.sqrt(((l - 1.0) ** 2 - m * m) * (2 * l + 1) / ((2 * l - 3.0) * (l * l - m * m)))
                P[l, m] = f * c * P[l - 1, m] - h * P[l - 2, m]
        lam = (2 * l + 1) * al + 0.5
        C = [torch.ones_like(c), 2.0 * lam * xi]
        for n in range(2, nmax + 1):
            C.append((2.0 * (n + lam - 1.0) * xi * C[-1] - (n + 2.0 * lam - 2.0) * C[-2]) / n)
        rad = s ** l * (1.0 + t) ** (-(2 * l + 1) * al) * torch.stack(C[:nmax + 1])
        yield l, rad, [P[l, m] * Wc[m] for m in range(l + 1)], [P[l, m] * Ws[m] for m in range(l + 1)]


def norms(case, l):
    """(N_lm (l+1,), I_nl(b = 1) (nmax+1,))."""
    al = case["alpha"]
    N = [math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m)) for m in range(l + 1)]
    a, lam = (2 * l + 1) * al, (2 * l + 1) * al + 0.5
    I = [-(n + a) * (n + a + 1) / al * math.exp(math.lgamma(n + 2 * lam) - (4 * a + 3) * math.log(2.0) - math.lgamma(n + 1.0)
                                                 - math.log(n + lam) - 2 * math.lgamma(lam)) for n in range(case["nmax"] + 1)]
    f64 = {"device": DEV, "dtype": torch.float64}
    return torch.tensor(N, **f64), torch.tensor(I, **f64)


CHUNK = 1 << 17


def exact_coeffs(x, m, b, case):
    """[S, T], each {l: (nmax+1, l+1)}; differentiable in x."""
    out = {}
    for k in range(0, len(x), CHUNK):
        for l, rad, yc, ys in basis(x[k:k + CHUNK], b, case):
            N, I = norms(case, l)
            f = -N / I[:, None] * torch.tensor([1.0] + [2.0] * l, device=DEV, dtype=torch.float64)
            w = rad * m[k:k + CHUNK]
            part = (f * (w @ torch.stack(yc).T), f * (w @ torch.stack(ys).T))
            out[l] = part if l not in out else (out[l][0] + part[0], out[l][1] + part[1])
    return out


def exact_accel(x, A, b, case, graph=False):
    """(acceleration, potential) of the expansion: minus the gradient of Eq. 1a at fixed coefficients."""
    acc, pot = [], []
    for k in range(0, len(x), CHUNK):
        y = x[k:k + CHUNK] * 1.0 if graph else x[k:k + CHUNK].detach().requires_grad_(True)
        psi = 0.0
        for l, rad, yc, ys in basis(y, b, case):
            N, _ = norms(case, l)
            S, T = (t / N for t in A[l])
            psi = psi - ((S.T @ rad) * torch.stack(yc) + (T.T @ rad) * torch.stack(ys)).sum(0) / b
        g, = torch.autograd.grad(psi.sum(), y, create_graph=graph)
        acc.append(-g)
        pot.append(psi if graph else psi.detach())
    return torch.cat(acc), torch.cat(pot)


def flat(A, case):
    """The library's [S | T] row: n-major, then l(l+1)/2 + m; T at m = 0 is 0."""
    S = torch.cat([A[l][0] for l in range(case["lmax"] + 1)], 1).reshape(-1)
    T = torch.cat([A[l][1] for l in range(case["lmax"] + 1)], 1).reshape(-1)
    return torch.cat([S, T])


def field(x, m, com, b, host, case, graph=False, A=None):
    """Coefficients of one cluster and the acceleration, tide included, at its particles."""
    A = exact_coeffs(x, m, b, case) if A is None else A
    a, psi = exact_accel(x, A, b, case, graph)
    if host:
        a = a + host_accel(host, com[:3] + x) - host_accel(host, com[:3])
    return A, a, psi


def exact_step(x, v, a, com, m, b, host, case, graph=False):
    h, dt = 0.005, 0.01
    v = v + h * a
    x = x + dt * v
    if host:
        V = com[3:] + h * host_accel(host, com[:3])
        R = com[:3] + dt * V
        com = torch.cat([R, V + h * host_accel(host, R)])
    A, a, psi = field(x, m, com, b, host, case, graph)
    return x, v + h * a, a, com, A, psi


def exact_energy(x, v, m):
    """0.5 v^2 - sum_j m_j / r_ij."""
    E = 0.5 * (v * v).sum(1)
    for k in range(0, len(x), 2048):
        d2 = torch.zeros((len(x[k:k + 2048]), len(x)), device=DEV, dtype=torch.float64)
        for i in range(3):
            d2 += (x[k:k + 2048, i:i + 1] - x[None, :, i]) ** 2
        inv = torch.rsqrt(d2)
        inv[d2 == 0] = 0.0
        E[k:k + 2048] -= inv @ m
    return E


def exact(case, seed):
    do = case["do"]
    if do == "evolve":
        return None
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    pos, vel, rh = sample(case, seed)
    pos, vel = pos.to(dtype).double(), vel.to(dtype).double()
    coms, host, b, off = centres(case, seed), host_of(case), scales(case, rh), offsets_of(case)
    rows = []
    if do == "adjoint":
        return exact_adjoint(case, pos, vel, coms[0], host, b[0])
    for p in range(case["n_prog"]):
        s = slice(off[p], off[p + 1])
        x, v, m = pos[s, :3].contiguous(), vel[s, :3].contiguous(), pos[s, 3]
        com = None if coms is None else coms[p]
        if do == "bound":
            E = exact_energy(x, v, m)
            r2 = (x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1]) + x[:, 2] * x[:, 2]
            bnd = E < 0
            k = math.ceil(0.999 * int(bnd.sum()))
            cut = torch.sort(r2[bnd]).values[k - 1]
            st = [float(bnd.sum()), float(m[bnd].sum()), math.sqrt(float(cut)), float((r2 <= cut).sum())]
            rows.append((bnd.to(torch.uint8), (r2 <= cut).to(torch.uint8), torch.tensor(st, device=DEV, dtype=torch.float64), E))
        elif do == "coeffs":
            rows.append(flat(exact_coeffs(x, m * mask_of(case, x), b[p], case), case))
        else:
            A, a, psi = field(x, m, com, b[p], host, case)
            if do == "forces":
                rows.append(torch.cat([a, psi[:, None]], 1))
                continue
            x, v, a, com, A, psi = exact_step(x, v, a, com, m, b[p], host, case)
            zero = torch.zeros_like(m)[:, None]
            rows.append((torch.cat([x, m[:, None]], 1), torch.cat([v, zero], 1), torch.cat([a, psi[:, None]], 1), flat(A, case), com))
    if do == "coeffs":
        return torch.stack(rows)
    if do == "forces":
        return torch.cat(rows)
    if do == "bound":
        return {"bound": torch.cat([r[0] for r in rows]), "mask": torch.cat([r[1] for r in rows]),
                "stats": torch.stack([r[2] for r in rows]), "E": torch.cat([r[3] for r in rows])}
    out = {"pos": torch.cat([r[0] for r in rows]), "vel": torch.cat([r[1] for r in rows]), "acc": torch.cat([r[2] for r in rows])}
    if do == "step" and case["precision"] == "fp64":
        out["A"] = torch.stack([r[3] for r in rows])
    return out if coms is None else dict(out, com=torch.stack([r[4] for r in rows]))


def exact_adjoint(case, pos, vel, com, host, b):
    m = pos[:, 3]
    hp = torch.tensor([[M, a] for _, M, a, _ in host], device=DEV, dtype=torch.float64, requires_grad=True)
    lp, lv, lc = (t.clone().requires_grad_(True) for t in (pos, vel, com))
    hosts = [(k, hp[i, 0], hp[i, 1], bb) for i, (k, _, _, bb) in enumerate(host)]
    x, v, c = lp[:, :3], lv[:, :3], lc
    _, a, _ = field(x, m, c, b, hosts, case, graph=True)
    for _ in range(case["nsteps"]):
        x, v, a, c, _, _ = exact_step(x, v, a, c, m, b, hosts, case, graph=True)
    idx = torch.arange(0, case["n"], 97, device=DEV)
    loss_of(x, c, idx, track(com, len(idx))).backward()
    gp, gv = lp.grad.clone(), lv.grad.clone()
    gp[:, 3] = 0.0
    gv[:, 3] = 0.0
    return {"pos": torch.cat([x, m[:, None]], 1).detach(), "vel": torch.cat([v, torch.zeros_like(m)[:, None]], 1).detach(),
            "com": c.detach(), "d_pos": gp, "d_vel": gv, "d_com": lc.grad, "d_host": hp.grad}
