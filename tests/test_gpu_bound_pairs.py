"""The boundedness sums, which take every unordered pair once, and the selection
at the edges of their chunks: against direct sums in 64 bits with torch.

Tolerances on E relative to the largest |W_i| (or |E_i|, for a particle alone): a double-precision term (float-
float) is good to about 1e-13 and up to 1e4 of them are added, 1e-11; a single-
precision term to a few 6e-8 and its 128-term float sums to a few more, 2e-6.
"""
import math

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def scf():
    import paper_2602_13385_gb300 as m
    return m


def sample(n, dtype, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    x = torch.randn(n, 4, device="cuda", generator=g, dtype=torch.float64)
    x[:, 3] = (0.5 + x[:, 3].abs()) / n
    v = 0.8 * torch.randn(n, 4, device="cuda", generator=g, dtype=torch.float64)
    return x.to(dtype), v.to(dtype)


def direct(pos, vel):
    x, m, v = pos[:, :3].double(), pos[:, 3].double(), vel[:, :3].double()
    inv = 1.0 / (x[:, None] - x[None]).norm(dim=2)
    inv[~torch.isfinite(inv)] = 0.0          # the particle itself, coincident and non-finite pairs
    W = inv @ m
    return 0.5 * (v * v).sum(1) - W, W


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("sizes", [[1], [2], [255], [256], [257], [511], [512], [513], [768], [1025], [2049], [5000],
                                   [300, 0, 1, 1536, 777], [4096, 33]])
def test_pair_sums_and_selection(scf, prec, sizes):
    off = [0]
    for s in sizes:
        off.append(off[-1] + s)
    n = off[-1]
    cfg = scf.Config(nmax=4, lmax=2, b=1.0, precision=prec)
    pos, vel = sample(n, cfg.dtype, n)
    if n > 300:
        pos[n // 3, :3] = pos[n // 2, :3]      # a coincident pair
    sim = scf.SCF(cfg, offsets=off)
    b, mask, stats, E = sim.bound(pos, vel, frac=0.9, energies=True)
    again = sim.bound(pos, vel, frac=0.9, energies=True)
    assert torch.equal(E, again[3]) and torch.equal(stats, again[2])      # fixed order
    tol = 1e-11 if prec == "fp64" else 2e-6
    for p in range(len(sizes)):
        s = slice(off[p], off[p + 1])
        if sizes[p] == 0:
            assert stats[p].tolist() == [0.0, 0.0, 0.0, 0.0]
            continue
        ref, W = direct(pos[s], vel[s])
        assert (E[s] - ref).abs().max().item() <= tol * max(W.max().item(), ref.abs().max().item())
        assert torch.equal(b[s].bool(), E[s] < 0)
        x = pos[s, :3].double()
        r2 = (x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1]) + x[:, 2] * x[:, 2]
        nb = int(b[s].sum())
        cut = torch.sort(r2[b[s].bool()]).values[math.ceil(0.9 * nb) - 1].item() if nb else 0.0
        assert torch.equal(mask[s].bool(), r2 <= cut)
        assert stats[p, 0].item() == nb and stats[p, 2].item() == math.sqrt(cut)
        assert stats[p, 3].item() == int((r2 <= cut).sum())
        assert stats[p, 1].item() == pytest.approx(float(pos[s, 3].double()[b[s].bool()].sum()), rel=1e-12, abs=0)
    sim.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_nonfinite_and_extreme_particles_add_nothing(scf, prec):
    cfg = scf.Config(nmax=4, lmax=2, b=1.0, precision=prec)
    pos, vel = sample(1300, cfg.dtype, 9)
    pos[5, 0], pos[700, 2] = float("nan"), float("inf")
    pos[900, :3] = pos[40, :3] + torch.tensor([1e-25, 0.0, 0.0], device="cuda", dtype=cfg.dtype)   # r^2 below the range
    pos[1299, 1] = 3e25                                                                            # and above it
    sim = scf.SCF(cfg, n=1300)
    b, _, _, E = sim.bound(pos, vel, energies=True)
    ok = torch.ones(1300, dtype=torch.bool, device="cuda")
    ok[[5, 700]] = False
    x, m = pos[:, :3].double(), pos[:, 3].double()
    r2 = ((x[:, None] - x[None]) ** 2).sum(2)
    inv = torch.where((r2 >= 1.17549435e-38) & (r2 <= 3.40282347e38), r2.rsqrt(), torch.zeros_like(r2))
    W = inv @ m
    ref = 0.5 * (vel[:, :3].double() ** 2).sum(1) - W
    tol = 1e-11 if prec == "fp64" else 2e-6
    assert (E - ref)[ok].abs().max().item() <= tol * W[ok].max().item()
    assert not b[5] and not b[700]
