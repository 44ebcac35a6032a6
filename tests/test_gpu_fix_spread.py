"""Forces whose sums the symmetric kernels add up in fixed point, for loads in other units than
total mass and length one: R^3 and FP64 contexts against the image sums in extended precision. The
bounds are those of the loads of order one: 1e-6 for the 2-norm of an FP32 force (some 6e-7), and
test_gpu_fp64_closed's for FP64."""
import numpy as np
import pytest

from paper_2602_20787_gb300 import ics
from test_gpu_fp64_closed import EPS, image_sums

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_20787_gb300 import steps_cyl
    steps_cyl.load()
    return steps_cyl


def ball(n, R, M, soft, heavy=0.0):
    d = ics.ball_load(n, 3)
    m = np.full(n, 1.0 / n)
    if heavy:
        m[1:] /= heavy
    return d["pos"] * (R / np.abs(d["pos"]).max()), m * (M / m.sum()), np.full(n, soft * R)


def r3(sc, precision, R):
    return sc.Config(topology=sc.STEPS_TOPO_R3, n_cut=1, R_sim=2.0 * R, background=sc.STEPS_BG_OFF, precision=precision)


@pytest.mark.parametrize("R,M,soft,heavy,sym", [(1.0, 1.0, 0.05, 0, 1), (1e4, 1.0, 0.05, 0, 1), (1e6, 1e-9, 0.05, 0, 1),
                                                (1e8, 1e12, 0.05, 0, 1), (1e-3, 1e12, 1e-3, 0, 1),
                                                (1.0, 1.0, 0.05, 1e4, 1), (1.0, 1.0, 0.05, 1e9, 0),
                                                (1.0, 1.0, 1e-8, 0, 0)])
def test_r3(sc, R, M, soft, heavy, sym):
    n = 160
    pos, m, h = ball(n, R, M, soft, heavy)
    ref, mag = image_sums(pos, m, h, 1, r3=True)
    for pre in (sc.STEPS_FP32_KAHAN, sc.STEPS_FP32_PLAIN, sc.STEPS_FP64):
        sim = sc.Simulation(r3(sc, pre, R), pos, np.zeros_like(pos), m, h)
        a = sim.forces()
        ev = sc.steps_cyl_last_eval(sim.ctx)
        sim.close()
        if pre == sc.STEPS_FP64:
            assert np.all(abs(a - ref) <= (32 + n) * EPS * mag)
        else:
            assert bool(ev["symmetric"]) == bool(sym)
            err = np.linalg.norm(a - ref, axis=1) / np.linalg.norm(mag, axis=1)
            assert np.sqrt((err ** 2).mean()) <= 1e-6 and err[0] <= 1e-5, (np.sqrt((err ** 2).mean()), err[0])


def test_r3_spreads_in_a_run(sc):
    # outward velocities carry the particles from R = 1 to 1e6 within one call, beyond what the sums'
    # unit was looked at for
    n, steps = 160, 80
    pos, m, h = ball(n, 1.0, 1.0, 0.05)
    v = pos * (1e6 / (steps * 1e-2))
    for split in (1, steps):
        sim = sc.Simulation(r3(sc, sc.STEPS_FP32_KAHAN, 1.0), pos, v, m, h)
        for _ in range(split):
            sim.step(1e-2, steps // split)
        a = sim.forces()
        x = sim.state()[0]
        ref, mag = image_sums(x, m, h, 1, r3=True)
        err = np.linalg.norm(a - ref, axis=1) / np.linalg.norm(mag, axis=1)
        assert np.sqrt((err ** 2).mean()) <= 1e-6
        sim.close()


@pytest.mark.parametrize("n_cut", [5, 24])
@pytest.mark.parametrize("M,soft,R", [(1e-15, 1e-10, 1.0), (1e-9, 1e-3, 1.0), (1e12, 1e-2, 1.0), (1.0, 1e-2, 1e9)])
def test_cylinder_fp64(sc, n_cut, M, soft, R):
    n = 97
    d = ics.particle_load(n, 5, 1.0)
    pos = d["pos"] * [R, R, 1.0]
    m, h = d["m"] * M, np.random.default_rng(4).uniform(0.3, 1.0, n) * soft
    ref, mag = image_sums(pos, m, h, n_cut)
    sim = sc.Simulation(sc.Config(n_cut=n_cut, background=sc.STEPS_BG_OFF, precision=sc.STEPS_FP64), pos,
                        np.zeros_like(pos), m, h)
    a = sim.forces()
    sim.close()
    assert np.all(abs(a - ref) <= (32 + n) * EPS * mag), float((abs(a - ref) / mag).max() / EPS)
