"""The FP64 pair kernels (pair_fp64.cuh) against the image sums in extended precision: the
symmetric kernel at sizes around its blocks of 32, and the subset's row kernel, for windows
below, at and above the one the closed form is taken from, with softenings from a hundredth
to many periods, separations beyond the closed form's range, equal z and z half a period apart.

The bound is on the error against the sum of the terms' absolute values: 32 roundings for a
pair's own sum (four per image or end, the polynomials, the FP32 terms' 4e-16) and one for each
of its n pairs."""
import numpy as np
import pytest

from paper_2602_20787_gb300 import ics

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_20787_gb300 import steps_cyl
    steps_cyl.load()
    return steps_cyl


def image_sums(pos, m, h, n_cut, r3=False):
    """Pair field and the sum of its terms' absolute values, in extended precision."""
    ld = np.longdouble
    p, m, h = pos.astype(ld), m.astype(ld), h.astype(ld)
    n = len(m)
    acc, mag = np.zeros((n, 3), ld), np.zeros((n, 3), ld)
    for i in range(n):
        d = np.delete(p[i] - p, i, 0)
        mj, hh = np.delete(m, i), np.delete(h[i] + h, i)
        dz = d[:, 2] if r3 else d[:, 2] - np.rint(d[:, 2])
        k = np.zeros(1) if r3 else np.arange(-n_cut, n_cut + 1)
        o = dz[:, None] + k
        r = np.sqrt(o * o + (d[:, 0] ** 2 + d[:, 1] ** 2)[:, None])
        u = r / hh[:, None]
        uo = np.maximum(u, ld(0.25))
        inner = (ld(32) / 3 + u * u * (32 * u - ld(192) / 5)) / hh[:, None] ** 3
        outer = (ld(64) / 3 - 48 * uo + ld(192) / 5 * uo ** 2 - ld(32) / 3 * uo ** 3 - 1 / (15 * uo ** 3)) / hh[:, None] ** 3
        f = np.where(u < 0.5, inner, np.where(u < 1, outer, 1 / np.maximum(r, ld(1e-300)) ** 3))
        f = f if r3 else f * (abs(o) < n_cut)
        sr = f.sum(1)
        for a, v, w in ((0, d[:, 0] * sr, abs(d[:, 0]) * sr), (1, d[:, 1] * sr, abs(d[:, 1]) * sr),
                        (2, (o * f).sum(1), (abs(o) * f).sum(1))):
            acc[i, a] = -(mj * v).sum()
            mag[i, a] = (mj * w).sum()
    return acc, mag


def load(n, soft, seed):
    d = ics.particle_load(n, seed, 1.0)
    pos = d["pos"].copy()
    if n >= 40:
        pos[1:4, 2] = pos[0, 2]                          # equal z
        pos[4, 2], pos[5, 2] = 0.125, 0.625              # half a period
        pos[6, :2] = [40.0, 3.0]                         # beyond the closed form's dR
        pos[7, :2] = [16.0 + pos[8, 0], pos[8, 1]]
        pos[9, :2] = pos[10, :2] + 1e-9                  # close, on one line of images
    return pos, d["m"], np.random.default_rng(seed).uniform(0.3, 1.0, n) * soft


@pytest.mark.parametrize("n", [2, 31, 33, 65, 97])
@pytest.mark.parametrize("n_cut,soft", [(1, 0.3), (2, 0.01), (13, 0.3), (14, 0.01), (14, 9.0), (15, 0.3), (24, 4.0),
                                        (24, 20.0)])
def test_cylinder(sc, n, n_cut, soft):
    pos, m, h = load(n, soft, n)
    ref, mag = image_sums(pos, m, h, n_cut)
    sim = sc.Simulation(sc.Config(n_cut=n_cut, background=sc.STEPS_BG_OFF, precision=sc.STEPS_FP64), pos,
                        np.zeros_like(pos), m, h)
    idx = np.arange(0, n, 2)
    a, s = sim.forces(), sim.forces_subset(idx)
    sim.close()
    assert np.all(abs(a - ref) <= (32 + n) * EPS * mag), float((abs(a - ref) / mag).max() / EPS)
    assert np.all(abs(s - ref[idx]) <= (32 + n) * EPS * mag[idx])


@pytest.mark.parametrize("n,soft", [(2, 0.1), (33, 0.01), (97, 0.3), (97, 9.0)])
def test_r3(sc, n, soft):
    pos, m, h = load(n, soft, n)
    ref, mag = image_sums(pos, m, h, 1, r3=True)
    sim = sc.Simulation(sc.Config(topology=sc.STEPS_TOPO_R3, n_cut=1, R_sim=2.0, background=sc.STEPS_BG_OFF,
                                  precision=sc.STEPS_FP64), pos, np.zeros_like(pos), m, h)
    a = sim.forces()
    sim.close()
    assert np.all(abs(a - ref) <= (32 + n) * EPS * mag), float((abs(a - ref) / mag).max() / EPS)
