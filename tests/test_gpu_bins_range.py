"""Radial bins in double precision outside the float range: the units are the
caller's, so a radius may lie anywhere in the double range.

Lengths times a power of two, with G times its cube and velocities times it, are
the same system in other units, and every operation of a double-precision pass
scales exactly: coefficients and adjoints stay the same bit for bit, positions,
velocities and accelerations are times the factor bit for bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def scf():
    import paper_2602_13385_gb300 as m
    return m


def binned(scf, cfg, mode=2, **kw):
    from paper_2602_13385_gb300 import _lib
    sim = scf.SCF(cfg, **kw)
    assert sim.launches_per_call("step") > 4
    _lib.scf_set_option(sim._h, _lib.SCF_OPT_RADIAL_BINS, mode)
    return sim


@pytest.mark.parametrize("alpha", [1.0, 0.5])
@pytest.mark.parametrize("power", [67, -67, 130, -130])
def test_other_units_same_result(scf, alpha, power):
    from paper_2602_13385_gb300 import _lib
    n = 12001
    g = np.random.default_rng(4)
    x = g.normal(size=(n, 3))
    x *= (np.exp(g.normal(-0.3, 0.9, n)) / np.linalg.norm(x, axis=1))[:, None]
    m, v, w = g.uniform(0.5, 1.5, n) / n, 0.3 * g.normal(size=(n, 4)), g.normal(size=(n, 4))
    out = []
    for f in (1.0, 2.0 ** power):
        cfg = scf.Config(nmax=20, lmax=8, b=0.7 * f, G=f ** 3, alpha=alpha)
        sim = binned(scf, cfg, n=n)
        p = torch.tensor(np.concatenate([f * x, m[:, None]], 1), device="cuda")
        vel = torch.tensor(f * v, device="cuda")
        A = sim.coeffs(p)
        acc = sim.forces(p, A)
        got = [A, acc[:, :3] / f]
        if alpha == 1.0:
            xb, vb = torch.tensor(w, device="cuda"), torch.tensor(w[::-1].copy(), device="cuda")
            _lib.scf_adjoint_level(sim._h, p, None, 0.01, True, xb, vb, None, None)
            got += [xb, vb]
        sim.step(p, vel, acc, nsteps=2)
        got += [p[:, :3] / f, vel[:, :3] / f, acc[:, :3] / f]
        assert sim.status() == (0, 0)
        out.append(got)
        sim.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("alpha", [1.0, 4.0])
def test_radii_far_from_the_scale(scf, alpha):
    """r / b from 1e-30 to 1e30 against the direct kernels, each particle on its own
    scale.  1e-11: sums over (20, 8) terms with recurrences of tens of steps in both."""
    n = 12001
    g = np.random.default_rng(5)
    x = g.normal(size=(n, 3))
    r = np.exp(g.normal(-0.3, 0.9, n))
    r[::10] = 10.0 ** g.uniform(-30, 30, r[::10].size)
    x *= (r / np.linalg.norm(x, axis=1))[:, None]
    pos = torch.tensor(np.concatenate([x, g.uniform(0.5, 1.5, (n, 1)) / n], 1), device="cuda")
    cfg = scf.Config(nmax=20, lmax=8, b=0.7, alpha=alpha)
    sims = [binned(scf, cfg, mode, n=n) for mode in (2, 0)]
    A = [s.coeffs(pos) for s in sims]
    assert (A[0] - A[1]).abs().max() <= 1e-11 * A[1].abs().max()
    acc, ref = (s.forces(pos, A[1]) for s in sims)
    for s in sims:
        assert s.status() == (0, 0)
    err = (acc - ref)[:, :3].norm(dim=1) / ref[:, :3].norm(dim=1).clamp_min(1e-300)
    assert err.max().item() <= 1e-11, (err.argmax().item(), err.max().item())
    pot = ((acc - ref)[:, 3] / ref[:, 3]).abs()
    assert pot.max().item() <= 1e-11
