"""The coefficient and field passes over radial bins against the direct kernels.

Handles above the size rule sort the particles by radius and replace the
radial polynomials by their interpolants; small handles run the direct kernels.
So the same sample cut into small handles is the comparison: coefficients add
up (Eq. 3b is a sum over particles), and the field at fixed coefficients is one
value a particle.  Tolerances: a double-precision sum of N terms of relative
error 1e-14 (recurrences of tens of steps) stays within 1e-11 of the largest
coefficient and acceleration; single-precision terms carry some tens of
roundings of 6e-8, so 5e-6.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-11, "mixed": 5e-6}
CUT = 1999        # particles of a comparison handle: below the size rule everywhere


@pytest.fixture(scope="module")
def scf():
    import paper_2602_13385_gb300 as m
    return m


def every_pass(sim):
    """Radial bins in every pass, also where the direct kernels are the faster ones."""
    from paper_2602_13385_gb300 import _lib
    _lib.scf_set_option(sim._h, _lib.SCF_OPT_RADIAL_BINS, 2)
    return sim


def sample(n, seed, dtype):
    """A wide sample: core, halo far beyond the basis scale, and the special places."""
    g = np.random.default_rng(seed)
    r = np.exp(g.normal(-0.3, 0.9, n))
    r[: n // 50] *= np.exp(g.uniform(0, 6, n // 50))
    x = g.normal(size=(n, 3))
    x *= (r / np.linalg.norm(x, axis=1))[:, None]
    x[n // 2] = 0.0                       # the centre
    x[n // 2 + 1] = (0.0, 0.0, 1e-9)      # on the axis, next to it
    x[n // 2 + 2] = (3e5, 0.0, -2e5)      # far outside
    x[n // 2 + 3] = (0.4, 0.0, 0.0)
    m = g.uniform(0.5, 1.5, n) / n
    return torch.tensor(np.concatenate([x, m[:, None]], 1), dtype=dtype, device="cuda")


def bi_orthonormal(A, nmax, lmax, alpha):
    """a_nlm of Eq. 3a, S sqrt|I_nl| / ((2 - delta_m0) N_lm): every degree on the scale of its energy."""
    w = np.zeros((nmax + 1, (lmax + 1) * (lmax + 2) // 2))
    for l in range(lmax + 1):
        a, lam = (2 * l + 1) * alpha, (2 * l + 1) * alpha + 0.5
        for n in range(nmax + 1):
            lg = (math.lgamma(n + 2 * lam) - (4 * a + 3) * math.log(2) - math.lgamma(n + 1) - math.log(n + lam)
                  - 2 * math.lgamma(lam))
            I = (n + a) * (n + a + 1) / alpha * math.exp(lg)
            for m in range(l + 1):
                N = math.sqrt((2 * l + 1) / (4 * math.pi) * math.exp(math.lgamma(l - m + 1) - math.lgamma(l + m + 1)))
                w[n, l * (l + 1) // 2 + m] = math.sqrt(I) / ((1 if m == 0 else 2) * N)
    w = torch.tensor(w.reshape(-1), device=A.device)
    return A.reshape(A.shape[0], 2, -1) * w


def pieces(offsets):
    for p in range(len(offsets) - 1):
        for a in range(offsets[p], offsets[p + 1], CUT):
            yield p, a, min(a + CUT, offsets[p + 1])


CASES = [
    # precision, nmax, lmax, alpha, offsets
    ("fp64", 20, 10, 1.0, [0, 9001]),
    ("fp64", 20, 8, 0.5, [0, 60013]),           # the finer bins
    ("fp64", 10, 5, 1.0, [0, 16384]),
    ("fp64", 9, 7, 1.5, [0, 12289]),            # a degree between the compiled ones
    ("fp64", 40, 12, 1.0, [0, 7000]),
    ("fp64", 10, 3, 1.0, [0, 40000]),
    ("fp64", 20, 10, 1.0, [0, 20001, 20001, 20050, 43210]),   # empty and tiny progenitors
    ("mixed", 20, 10, 1.0, [0, 70001]),
    ("mixed", 20, 10, 0.5, [0, 420007]),        # the finer bins
    ("mixed", 10, 5, 1.0, [0, 300001]),
    ("mixed", 11, 6, 1.0, [0, 250000]),
    ("mixed", 40, 12, 1.0, [0, 40961]),
    ("mixed", 20, 8, 1.0, [0, 100000, 100000, 100031, 205000]),
]


@pytest.mark.parametrize("prec,nmax,lmax,alpha,offsets", CASES)
def test_bins_against_direct_kernels(scf, prec, nmax, lmax, alpha, offsets):
    n, P = offsets[-1], len(offsets) - 1
    host = [(2, 6.6e6, 5000.0, 0.0), (3, 6.8e5, 750.0, 70.0)]
    cfg = scf.Config(nmax=nmax, lmax=lmax, b=0.7, precision=prec, host=host, alpha=alpha)
    b = [0.7 + 0.1 * p for p in range(P)]
    com = torch.tensor([[2000.0 + 50 * p, 100.0, -30.0, 0.0, 40.0, 0.0] for p in range(P)], device="cuda",
                       dtype=torch.float64)
    pos = sample(n, 3, cfg.dtype)
    mask = (torch.arange(n, device="cuda") % 7 != 0).to(torch.uint8)
    sim = every_pass(scf.SCF(cfg, offsets=offsets, b_per_prog=b))
    assert sim.launches_per_call("coeffs") > 2, "the sample should be over the size rule"
    A = sim.coeffs(pos, mask=mask)
    assert torch.equal(A, sim.coeffs(pos, mask=mask))                  # fixed order
    ref, small = torch.zeros_like(A), {}
    for p, i, j in pieces(offsets):
        key = (p, j - i)
        if key not in small:
            small[key] = scf.SCF(cfg, n=j - i, b_per_prog=[b[p]])
            assert small[key].launches_per_call("coeffs") == 2
        ref[p] += small[key].coeffs(pos[i:j].contiguous(), mask=mask[i:j].contiguous())[0]
    a, a_ref = bi_orthonormal(A, nmax, lmax, alpha), bi_orthonormal(ref, nmax, lmax, alpha)
    scale = a_ref.abs().amax(dim=(1, 2), keepdim=True).clamp_min(1e-300)
    err = ((a - a_ref).abs() / scale).max().item()
    assert err < TOL[prec], err
    # the field at the same coefficients
    acc = sim.forces(pos, ref, com=com)
    out = torch.empty_like(acc)
    for p, i, j in pieces(offsets):
        out[i:j] = small[(p, j - i)].forces(pos[i:j].contiguous(), ref[p:p + 1].contiguous(), com=com[p:p + 1].contiguous())
    scale = out[:, :3].norm(dim=1).max()
    assert ((acc - out)[:, :3].norm(dim=1).max() / scale).item() < TOL[prec]
    assert ((acc - out)[:, 3].abs().max() / out[:, 3].abs().max()).item() < TOL[prec]
    assert sim.status() == (0, 0)
    sim.close()


@pytest.mark.parametrize("prec,n", [("fp64", 9001), ("mixed", 70001)])
def test_bins_nonfinite_particles_are_left_out_and_flagged(scf, prec, n):
    cfg = scf.Config(nmax=20, lmax=10, b=0.7, precision=prec)
    pos = sample(n, 5, cfg.dtype)
    bad = pos.clone()
    bad[17, 0], bad[n - 1, 2], bad[4000, 3] = float("nan"), float("inf"), float("nan")
    good = pos.clone()
    good[[17, n - 1, 4000], 3] = 0.0
    sim = every_pass(scf.SCF(cfg, n=n))
    A = sim.coeffs(good)
    assert sim.status() == (0, 0)
    B = sim.coeffs(bad)
    assert sim.status()[1] & 1
    assert ((A - B).abs().max() / A.abs().max()).item() < TOL[prec]
    acc = sim.forces(bad, A)
    assert sim.status()[1] & 1
    assert torch.equal(acc[:17], sim.forces(pos, A)[:17])


@pytest.mark.parametrize("prec,n", [("fp64", 9001), ("mixed", 70001)])
def test_bins_step_is_the_same_through_graph_plain_and_host_memory(scf, prec, n):
    host = [(2, 6.6e6, 5000.0, 0.0)]
    cfg = scf.Config(nmax=20, lmax=10, b=0.7, precision=prec, host=host)
    pos0 = sample(n, 6, cfg.dtype)
    pos0[n // 2 + 2, :3] = 1.0
    vel0 = 0.1 * torch.randn(n, 4, device="cuda", generator=torch.Generator("cuda").manual_seed(1)).to(cfg.dtype)
    com0 = torch.tensor([[2000.0, 100.0, -30.0, 0.0, 40.0, 0.0]], device="cuda", dtype=torch.float64)
    got = []
    for form in ("graph", "plain", "mapped", "staged"):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            sim = every_pass(scf.SCF(cfg, n=n))
            p, v, c = pos0.clone(), vel0.clone(), com0.clone()
            a = sim.forces(p, sim.coeffs(p), com=c)
            if form in ("graph", "plain"):
                sim.use_graphs(form == "graph")
                sim.step(p, v, a, c, nsteps=3)
            else:
                h = [t.cpu() for t in (p, v, a, c)]
                if form == "mapped":
                    h = [t.pin_memory() for t in h]
                s.synchronize()
                for _ in range(3):
                    sim.step_host(p, v, a, h[0], h[1], h[2], c, h[3])
                s.synchronize()
                p, v, a, c = h
            s.synchronize()
        got.append([t.cpu() for t in (p, v, a, c)])
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert torch.equal(x, y)


@pytest.mark.parametrize("prec,nmax,lmax,offsets", [("mixed", 10, 5, [0, 300001]), ("mixed", 20, 10, [0, 300001]),
                                                    ("fp64", 10, 5, [0, 20000]), ("fp64", 20, 8, [0, 30001])])
def test_passes_alone_and_host_steps_by_their_own_size_rules(scf, prec, nmax, lmax, offsets):
    """Default handles against bins in every pass and none: the same results whatever each pass runs over."""
    from paper_2602_13385_gb300 import _lib
    cfg = scf.Config(nmax=nmax, lmax=lmax, b=0.7, precision=prec)
    n = offsets[-1]
    pos0 = sample(n, 8, cfg.dtype)
    pos0[n // 2 + 2, :3] = 1.0
    vel0 = torch.zeros_like(pos0)
    got = []
    for mode in (1, 0, 2):
        sim = scf.SCF(cfg, offsets=offsets)
        _lib.scf_set_option(sim._h, _lib.SCF_OPT_RADIAL_BINS, mode)
        assert _lib.scf_get_option(sim._h, _lib.SCF_OPT_RADIAL_BINS) == mode
        A = sim.coeffs(pos0)
        acc = sim.forces(pos0, A)
        h = [t.cpu().pin_memory() for t in (pos0, vel0, acc)]
        d = [t.clone() for t in (pos0, vel0, acc)]
        sim.step_host(*d, *h)
        torch.cuda.synchronize()
        assert sim.status() == (0, 0)
        got.append([bi_orthonormal(A, nmax, lmax, 1.0), acc[:, :3]] + [t[:, :3] for t in h])
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert ((x - y).abs().max() / y.abs().max()).item() < 2 * TOL[prec]
