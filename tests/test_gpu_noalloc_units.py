"""The allocation-free call for loads in other units than a total mass and a size of order one, on
both its routes: against the oracle, 1e-6 for the median relative error (1e-7 and less for loads of
order one) and 1e-5 for the first particle, which is the heavy one. And particles far away keep their
own accelerations."""
import numpy as np
import pytest

import oracle
from paper_2602_20787_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_20787_gb300 import steps_cyl
    steps_cyl.load()
    return steps_cyl


def accel(sc, pos, m, h, n_cut, precision):
    import torch
    cols = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (*pos.T, m, h)]
    a = [torch.empty_like(cols[0]) for _ in range(3)]
    sc.steps_cyl_pair_accel_noalloc(*cols, 1.0, 1.0, n_cut, precision, *a, stream=torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return torch.stack(a, 1).cpu().numpy()


@pytest.mark.parametrize("n_cut", [5, 16])
@pytest.mark.parametrize("M,soft,R,heavy", [(1.0, 1e-2, 1.0, 1.0), (1e-9, 3e-7, 1.0, 1.0), (1e-15, 1e-10, 1.0, 1.0),
                                            (1e-6, 1e-2, 1.0, 1.0), (1e12, 1e-2, 1.0, 1.0), (1.0, 1e-2, 1e6, 1.0),
                                            (1.0, 1e-2, 1.0, 1e9)])
def test_units(sc, n_cut, M, soft, R, heavy):
    n = 300
    d = ics.particle_load(n, 9, 1.0)
    pos, m = d["pos"] * [R, R, 1.0], d["m"].copy()
    m[1:] /= heavy
    m *= M / m.sum()
    h = np.random.default_rng(4).uniform(0.3, 1.0, n) * soft
    ref = oracle.pair_field(pos, m, h, 1.0, 1.0, n_cut)
    for pre in (sc.STEPS_FP32_KAHAN, sc.STEPS_FP32_PLAIN):
        a = accel(sc, pos, m, h, n_cut, pre)
        err = np.linalg.norm(a - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert np.median(err) <= 1e-6 and err[0] <= 1e-5, (np.median(err), err[0])


@pytest.mark.parametrize("n_cut", [5, 16, 64])
def test_far_particles(sc, n_cut):
    d = ics.particle_load(200, 8, 1.0)
    for f in (1e4, 1e7, 1e10, 1e11):
        pos = np.vstack([d["pos"], [[f, 0.3 * f, 0.25]]])
        m, h = np.append(d["m"], d["m"][0]), np.append(d["h"], d["h"][0])
        a = accel(sc, pos, m, h, n_cut, sc.STEPS_FP32_KAHAN)
        D = pos[-1, :2] - pos[:-1, :2]
        # beyond some n_cut periods all images pull alike: 2 n_cut (one fewer at equal z) of them
        want = -((m[:-1] * 2 * n_cut / ((D ** 2).sum(1) + n_cut ** 2 / 3) ** 1.5)[:, None] * D).sum(0)
        assert np.linalg.norm(a[-1, :2] - want) <= 1e-5 * np.linalg.norm(want), (f, a[-1], want)


@pytest.mark.parametrize("n_cut", [5, 16])
@pytest.mark.parametrize("half", [128, 512, 2048])
def test_both_sides_are_summed_alike(sc, n_cut, half):
    # two points with as many equal particles each: every pair across them has the same terms, the
    # first half adds them up as rows and the other as j sides, in groups of eight either way, and the groups
    # exactly but for Kahan's second order: the accelerations are opposite
    pos = np.repeat([[0.0, 0.0, 0.1], [0.37, 0.21, 0.43]], half, axis=0)
    a = accel(sc, pos, np.full(2 * half, 1.0 / 3.0), np.full(2 * half, 0.05), n_cut, sc.STEPS_FP32_KAHAN)
    assert np.all(a[:half] == a[0]) and np.all(a[half:] == a[half])
    assert np.all(abs(a[0] + a[half]) <= 1e-11 * abs(a[0])), (a[0], a[half])


@pytest.mark.parametrize("n_cut", [5, 16])
def test_one_mass_among_massless_particles(sc, n_cut):
    d = ics.particle_load(300, 9, 1.0)
    m = np.zeros(300)
    m[7] = 2.5
    h = np.full(300, 1e-3)
    a = accel(sc, d["pos"], m, h, n_cut, sc.STEPS_FP32_KAHAN)
    ref = oracle.pair_field(d["pos"], m, h, 1.0, 1.0, n_cut)
    assert np.all(a[7] == 0.0) and np.array_equal(ref[7], np.zeros(3))
    k = np.arange(300) != 7
    err = np.linalg.norm(a[k] - ref[k], axis=1) / np.linalg.norm(ref[k], axis=1)
    assert np.median(err) <= 1e-6 and err.max() <= 1e-4
