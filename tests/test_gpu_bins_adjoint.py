"""One adjoint level over radial bins against the direct dual-number kernels.

A handle with the float-float field kernel selected keeps the direct adjoint
passes (in native double precision); its default twin runs them over radial
bins.  Both compute the same sums, so positions' and velocities' adjoints and
the centre's and host's agree to the rounding of sums with recurrences of tens
of steps and of second derivatives: 1e-11 of the largest entry.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [
    # nmax, lmax, offsets
    (20, 10, [0, 9001]),
    (10, 5, [0, 16385]),
    (9, 7, [0, 12289]),                             # a degree between the compiled ones
    (40, 12, [0, 7000]),
    (10, 3, [0, 40000]),
    (20, 6, [0, 20001]),
    (20, 8, [0, 60013]),                            # the finer bins
    (20, 10, [0, 20001, 20001, 20050, 43210]),      # empty and tiny progenitors
]


@pytest.mark.parametrize("nmax,lmax,offsets", CASES)
@pytest.mark.parametrize("host", [True, False])
def test_level_against_direct_kernels(nmax, lmax, offsets, host):
    import paper_2602_13385_gb300 as scf
    from paper_2602_13385_gb300 import _lib
    n, P = offsets[-1], len(offsets) - 1
    g = np.random.default_rng(n + lmax)
    x = g.normal(size=(n, 3))
    x *= (np.exp(g.normal(-0.3, 0.9, n)) / np.linalg.norm(x, axis=1))[:, None]
    x[n // 2] = 0.0                     # the centre
    x[n // 2 + 1] = (0.0, 0.0, 0.3)     # on the axis
    x[n // 2 + 2] = (3e4, 0.0, -2e4)    # far outside
    m = g.uniform(0.5, 1.5, n) / n
    comps = [(2, 6.6e6, 5000.0, 0.0), (3, 6.8e5, 750.0, 70.0)] if host else []
    cfg = scf.Config(nmax=nmax, lmax=lmax, b=0.7, host=comps)
    b = [0.7 + 0.1 * p for p in range(P)]

    def dev(a):
        return torch.tensor(a, dtype=torch.float64, device="cuda")
    pos = dev(np.concatenate([x, m[:, None]], 1))
    com = dev(np.concatenate([g.normal(size=(P, 3)) * 3000.0, g.normal(size=(P, 3))], 1))
    start = [dev(g.normal(size=(n, 4))), dev(g.normal(size=(n, 4))), dev(g.normal(size=(P, 6))),
             dev(np.zeros((P, max(2 * len(comps), 1))))]
    out = []
    for direct in (False, True):
        sim = scf.SCF(cfg, offsets=offsets, b_per_prog=b)
        if direct:
            _lib.scf_set_option(sim._h, _lib.SCF_OPT_K3_VARIANT, 1)
        xb, vb, cb, th = (t.clone() for t in start)
        _lib.scf_adjoint_level(sim._h, pos, com if host else None, 0.01, True, xb, vb, cb if host else None,
                               th if host else None)
        assert sim.status() == (0, 0)
        out.append((xb - start[0], vb - start[1], cb - start[2], th))
    for got, ref in zip(*out):
        assert torch.isfinite(got).all()
        top = ref.abs().amax()
        assert float((got - ref).abs().amax()) <= 1e-11 * float(top) + 1e-15
