"""Radial bins against the direct kernels of the same handle options (SCF_OPT_RADIAL_BINS 2
and 0), where a mistake cannot be in both: steps with their kicks and drifts, masks and
progenitors, every exponent, an adjoint level, and a handle moved between exponents.

Tolerances (derived as in test_gpu_bins.py): a double-precision sum of N terms with
recurrences of tens of steps, 1e-11; single-precision terms with some tens of roundings of
6e-8, 5e-6 of the largest value; a state kept in single precision adds its own rounding of
6e-8 a step to increments.  Single-precision fields and coefficients of every exponent are
compared with double precision on the same positions, where the direct kernels are the measure:
their own error is that of the arithmetic (up to 4e-4 of the acceleration of a particle whose
terms cancel, and 8e-5 of the largest coefficient at alpha = 4, where factors leave the normal
float range), and the binned passes, with as many or fewer roundings, may be off by half as
much again at most (the largest of tens of thousands of errors: by ten times).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from test_gpu_bins import TOL, bi_orthonormal, sample  # noqa: E402



@pytest.fixture(scope="module")
def scf():
    import paper_2602_13385_gb300 as m
    return m


def both(scf, cfg, **kw):
    """(binned, direct) handles."""
    from paper_2602_13385_gb300 import _lib
    sims = [scf.SCF(cfg, **kw) for _ in range(2)]
    for sim, mode in zip(sims, (2, 0)):
        _lib.scf_set_option(sim._h, _lib.SCF_OPT_RADIAL_BINS, mode)
    assert [s.launches_per_call("step") > 4 for s in sims] == [True, False]
    return sims


def errors(got, ref):
    """Each particle's acceleration and potential, on its own scale (a thousandth of the median's at least)."""
    a, b = got.double(), ref.double()
    own = b[:, :3].norm(dim=1)
    return (a - b)[:, :3].norm(dim=1) / (own + 1e-3 * own.median()), (a - b)[:, 3].abs() / b[:, 3].abs()


def no_worse(got, direct, floor=1e-7):
    """Errors of the binned passes against the direct kernels' errors."""
    got, direct = got.sort().values, direct.sort().values
    for q, factor in ((0.5, 1.5), (0.99, 1.5), (0.999, 1.5), (1.0, 10.0)):
        i = int(q * (len(got) - 1))
        assert got[i] <= factor * direct[i] + floor, (q, got[i].item(), direct[i].item())


@pytest.mark.parametrize("nmax,lmax,n", [(20, 8, 12001), (20, 10, 60013)])
@pytest.mark.parametrize("alpha", [0.1, 0.5, 1.0, 2.0, 4.0])
def test_every_exponent_fp64(scf, nmax, lmax, n, alpha):
    cfg = scf.Config(nmax=nmax, lmax=lmax, b=0.7, alpha=alpha)
    pos = sample(n, 3, cfg.dtype)
    pos[n // 2] = pos[n // 2 + 3]            # (the field of alpha > 1 diverges at the centre)
    pos[n // 2, 1] = 0.01
    sims = both(scf, cfg, n=n)
    A = [s.coeffs(pos) for s in sims]
    a, ref = (bi_orthonormal(x, nmax, lmax, alpha) for x in A)
    assert ((a - ref).abs().max() / ref.abs().max()).item() <= TOL["fp64"]
    for e in errors(*[s.forces(pos, A[1]) for s in sims]):
        assert e.max().item() <= TOL["fp64"]
    for s in sims:
        assert s.status() == (0, 0)
        s.close()


@pytest.mark.parametrize("nmax,lmax,n", [(20, 10, 70001), (20, 10, 420007), (10, 5, 300001)])
@pytest.mark.parametrize("alpha", [0.1, 0.5, 1.0, 2.0, 4.0])
def test_every_exponent_mixed(scf, nmax, lmax, n, alpha):
    cfg = scf.Config(nmax=nmax, lmax=lmax, b=0.7, precision="mixed", alpha=alpha)
    pos = sample(n, 3, cfg.dtype)
    pos[n // 2] = pos[n // 2 + 3]
    pos[n // 2, 1] = 0.01
    far = pos[:, :3].norm(dim=1) > 50.0      # (r / b)^10 of alpha = 0.1 stays in the float range
    pos[far, :3] *= 50.0 / pos[far, :3].norm(dim=1, keepdim=True)
    exact = scf.SCF(scf.Config(nmax=nmax, lmax=lmax, b=0.7, alpha=alpha), n=n)
    A = exact.coeffs(pos.double())
    ref, a0 = exact.forces(pos.double(), A), bi_orthonormal(A, nmax, lmax, alpha)
    exact.close()
    coef, field = [], []
    for s in both(scf, cfg, n=n):
        coef.append((bi_orthonormal(s.coeffs(pos), nmax, lmax, alpha) - a0).abs().max() / a0.abs().max())
        field.append(errors(s.forces(pos, A), ref))
        assert s.status() == (0, 0)
        s.close()
    assert coef[0] <= 1.5 * coef[1] + 1e-7
    for got, direct in zip(*field):
        no_worse(got, direct)


@pytest.mark.parametrize("prec,nmax,lmax,offsets", [("fp64", 20, 8, [0, 30001]), ("fp64", 10, 5, [0, 20000, 20000, 20031, 60007]),
                                                    ("mixed", 20, 10, [0, 70001]), ("mixed", 10, 5, [0, 300001]),
                                                    ("mixed", 20, 8, [0, 100000, 100000, 100031, 205000])])
@pytest.mark.parametrize("with_mask", [False, True])
def test_steps(scf, prec, nmax, lmax, offsets, with_mask):
    """Displacements, velocity changes and the last field of three steps from a moving state."""
    n, P, dt = offsets[-1], len(offsets) - 1, 0.05
    cfg = scf.Config(nmax=nmax, lmax=lmax, b=0.7, dt=dt, precision=prec, host=[(2, 6.6e6, 5000.0, 0.0), (3, 6.8e5, 750.0, 70.0)])
    pos = sample(n, 7, cfg.dtype)
    far = pos[:, :3].norm(dim=1) > 20.0
    pos[far, :3] *= 20.0 / pos[far, :3].norm(dim=1, keepdim=True)
    vel = (0.5 * torch.randn(n, 4, device="cuda", dtype=torch.float64,
                             generator=torch.Generator("cuda").manual_seed(2))).to(cfg.dtype)
    com = torch.tensor([[2000.0 + 50 * p, 100.0, -30.0, 0.0, 40.0, 0.0] for p in range(P)], device="cuda", dtype=torch.float64)
    mask = (torch.arange(n, device="cuda") % 3 != 0).to(torch.uint8) if with_mask else None
    out = []
    for sim in both(scf, cfg, offsets=offsets, b_per_prog=[0.7 + 0.1 * p for p in range(P)]):
        sim.set_mask(mask)
        p, v, c = pos.clone(), vel.clone(), com.clone()
        a = sim.forces(p, sim.coeffs(p, mask=mask), com=c)
        sim.step(p, v, a, c, nsteps=3)
        assert sim.status() == (0, 0)
        out.append(((p - pos)[:, :3].double(), (v - vel)[:, :3].double(), a, c, p, v))
        sim.close()
    (dx, dv, a, c, _, _), (dx0, dv0, a0, c0, p0, v0) = out
    assert torch.equal(c, c0)
    eps = 0.0 if prec == "fp64" else 3 * 6e-8
    assert (dx - dx0).abs().max().item() <= TOL[prec] * dx0.abs().max().item() + eps * p0[:, :3].abs().max().item()
    assert (dv - dv0).abs().max().item() <= TOL[prec] * dv0.abs().max().item() + eps * v0[:, :3].abs().max().item()
    assert (a - a0)[:, :3].abs().max().item() <= 2 * TOL[prec] * a0[:, :3].abs().max().item()


@pytest.mark.parametrize("nmax,lmax,offsets", [(20, 10, [0, 9001]), (10, 5, [0, 16385]), (20, 8, [0, 60013]),
                                               (20, 10, [0, 20001, 20001, 20050, 43210])])
def test_adjoint_level(scf, nmax, lmax, offsets):
    from paper_2602_13385_gb300 import _lib
    n, P = offsets[-1], len(offsets) - 1
    g = np.random.default_rng(n + lmax)
    x = g.normal(size=(n, 3))
    x *= (np.exp(g.normal(-0.3, 0.9, n)) / np.linalg.norm(x, axis=1))[:, None]

    def dev(a):
        return torch.tensor(a, dtype=torch.float64, device="cuda")
    pos = dev(np.concatenate([x, g.uniform(0.5, 1.5, (n, 1)) / n], 1))
    com = dev(np.concatenate([g.normal(size=(P, 3)) * 3000.0, g.normal(size=(P, 3))], 1))
    start = [dev(g.normal(size=(n, 4))), dev(g.normal(size=(n, 4))), dev(g.normal(size=(P, 6))), dev(np.zeros((P, 4)))]
    cfg = scf.Config(nmax=nmax, lmax=lmax, b=0.7, host=[(2, 6.6e6, 5000.0, 0.0), (3, 6.8e5, 750.0, 70.0)])
    out = []
    for sim in both(scf, cfg, offsets=offsets):
        t = [s.clone() for s in start]
        _lib.scf_adjoint_level(sim._h, pos, com, 0.01, True, *t)
        assert sim.status() == (0, 0)
        out.append([a - b for a, b in zip(t, start)])
        sim.close()
    for got, ref in zip(*out):
        assert (got - ref).abs().max().item() <= 1e-11 * ref.abs().max().item() + 1e-15


@pytest.mark.parametrize("prec,n", [("fp64", 12001), ("fp64", 60013), ("mixed", 90001)])
def test_a_handle_moved_between_exponents(scf, prec, n):
    """scf_retune_alpha over narrow ranges: other bins, past the allocation (direct), and back.
    Each time the handle is one that was made for the exponent."""
    nmax, lmax = 20, 8
    cfg = scf.Config(nmax=nmax, lmax=lmax, b=0.7, precision=prec)
    pos = sample(n, 9, cfg.dtype)
    pos[n // 2] = pos[n // 2 + 3]
    pos[n // 2, 1] = 0.01
    sim = scf.SCF(cfg, n=n)
    for lo, hi, binned in ((0.5, 0.51, True), (1.9, 1.95, True), (3.4, 3.5, False), (0.3, 0.31, True), (3.9, 3.95, False),
                           (1.2, 1.21, True)):
        al = sim.retune_alpha(pos, alpha_lo=lo, alpha_hi=hi)
        assert lo * (1 - 1e-12) <= al <= hi * (1 + 1e-12)
        assert (sim.launches_per_call("step") > 4) == binned, al
        fresh = scf.SCF(scf.Config(nmax=nmax, lmax=lmax, b=0.7, precision=prec, alpha=al), n=n, b_per_prog=sim.scales().tolist())
        A, ref = sim.coeffs(pos), fresh.coeffs(pos)
        acc, acc0 = sim.forces(pos, ref), fresh.forces(pos, ref)
        if binned:                           # the same bins: the same bits
            assert torch.equal(A, ref) and torch.equal(acc, acc0)
        else:
            a, r = bi_orthonormal(A, nmax, lmax, al), bi_orthonormal(ref, nmax, lmax, al)
            assert ((a - r).abs().max() / r.abs().max()).item() <= (TOL["fp64"] if prec == "fp64" else 1e-4)
            for e in errors(acc, acc0):
                assert e.quantile(0.999).item() <= (TOL["fp64"] if prec == "fp64" else 1e-4)
        assert sim.status() == (0, 0)
        fresh.close()
    sim.close()


def test_evolution_with_retuned_exponents(scf):
    """scf_evolve with complete refreshes of alpha and b: the step's graph, the tables and the bins of every
    new exponent.  Fields agree to 1e-11 and thirty short steps amplify little; the exponent is the root of a
    sum over the particles, found to 1e-8."""
    nmax, lmax, n = 10, 6, 20011
    pos0 = sample(n, 5, torch.float64)
    far = pos0[:, :3].norm(dim=1) > 20.0
    pos0[far, :3] *= 20.0 / pos0[far, :3].norm(dim=1, keepdim=True)
    com = torch.tensor([[2000.0, 100.0, -30.0, 0.0, 40.0, 0.0]], device="cuda", dtype=torch.float64)
    cfg = dict(nmax=nmax, lmax=lmax, b=0.7, dt=0.01, host=[(2, 6.6e6, 5000.0, 0.0), (3, 6.8e5, 750.0, 70.0)])
    out = []
    for sim in both(scf, scf.Config(**cfg), n=n):
        sim.config = scf.Config(**cfg)       # (evolve writes the exponent into it)
        p, v, c = pos0.clone(), torch.zeros_like(pos0), com.clone()
        a = sim.forces(p, sim.coeffs(p), com=c)
        alphas = []
        for _ in range(3):
            sim.evolve(p, v, a, c, nsteps=10, max_steps=5, retune_every=1, retune_rule="alpha_a000", alpha_range=(0.5, 1.8))
            alphas.append(sim.config.alpha)
        assert sim.status() == (0, 0)
        out.append((alphas, sim.scales(), (p - pos0)[:, :3], v[:, :3], a[:, :3], c))
        sim.close()
    (al, *got), (al0, *ref) = out
    assert al[0] != 1.0 and np.allclose(al, al0, rtol=1e-8, atol=0)
    for x, y in zip(got, ref):
        assert (x - y).abs().max().item() <= 1e-8 * y.abs().max().item()
