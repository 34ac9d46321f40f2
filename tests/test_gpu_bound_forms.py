"""The forms of the boundedness kernels that the sizes choose between, at the
sizes where they change (tolerances and the direct sums of test_gpu_bound_pairs)."""
import math

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from test_gpu_bound_pairs import direct, sample  # noqa: E402


@pytest.fixture(scope="module")
def scf():
    import paper_2602_13385_gb300 as m
    return m


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("sizes", [[1024], [1025], [13927], [13930], [14001, 0, 7, 300], [64] * 400, [1100] * 40,
                                   [4600], [4900], [11100], [11400],      # ordered pairs below, rounds of chunks above
                                   [14001, 0, 1, 255, 256, 257, 511, 512, 513, 768, 1025, 2049]])
def test_sums_and_selection(scf, prec, sizes):
    off = [0]
    for s in sizes:
        off.append(off[-1] + s)
    cfg = scf.Config(nmax=4, lmax=2, b=1.0, precision=prec)
    pos, vel = sample(off[-1], cfg.dtype, off[-1])
    sim = scf.SCF(cfg, offsets=off)
    b, mask, stats, E = sim.bound(pos, vel, frac=0.9, energies=True)
    assert torch.equal(E, sim.bound(pos, vel, frac=0.9, energies=True)[3])
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
