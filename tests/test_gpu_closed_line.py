"""GPU parity of the pair forms that take the image line beyond the near images in
closed form (pair2.cuh): the plain window and the modelled tails with n0 = 4.

- One pair at a time against the sum of its images in FP64, over separations from
  coincident to thousands of periods, dz at the edges of its range (0, tiny, 1/2), every
  softening tier (none, centre, several periods, beyond the whole window) and windows on
  both sides of each switch. The bound is 2e-6 of the sum of the images' magnitudes: an
  image carries rsqrt^3 (3 x 2 ulp) and the spline (a few ulp), about 1e-6, and the closed
  part and the sums as much again.
- Loads of every block remainder (one block, a ragged last one, quarter tiles) against
  the FP64 oracle, and the modelled tails against the row kernels, which take them side
  by side with each far end on its own."""
import numpy as np
import pytest

from gpu_helpers import oracle_accel, rel_err, stats
from paper_2602_20787_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_20787_gb300 import shard, steps_cyl
    steps_cyl.load()
    return torch, steps_cyl, shard


def spline_over_r(r, h):
    u = r / h
    with np.errstate(divide="ignore", invalid="ignore"):
        uo = np.maximum(u, 0.25)
        outer = (64 / 3 - 48 * uo + 38.4 * uo ** 2 - 32 / 3 * uo ** 3 - 1 / (15 * uo ** 3)) / h ** 3
        newton = 1.0 / np.maximum(r, 1e-300) ** 3
    return np.where(u < 0.5, (32 / 3 + u * u * (32 * u - 38.4)) / h ** 3, np.where(u < 1.0, outer, newton))


def image_sums(dR, dz, h, n_cut):
    """(sr, sz) and the sums of their magnitudes over |dz + k| < n_cut."""
    o = dz + np.arange(-n_cut, n_cut + 1)
    o = o[np.abs(o) < n_cut]
    f = spline_over_r(np.sqrt(dR * dR + o * o), h)
    return f.sum(), (o * f).sum(), f.sum(), (np.abs(o) * f).sum()


@pytest.mark.parametrize("n_cut", [1, 2, 11, 12, 13, 16, 64, 300])
@pytest.mark.parametrize("hh", [0.02, 0.49, 0.52, 1.3, 3.4, 4.6, 7.9, 9.2, 40.0])
def test_one_pair(env, n_cut, hh):
    torch, sc, shard = env
    m, h = np.array([1.0, 0.75]), np.array([0.4 * hh, 0.6 * hh])
    cfg = sc.Config(n_cut=n_cut, background=sc.STEPS_BG_OFF, reorder_every=-1)
    sim = sc.Simulation(cfg, np.array([[0.0, 0.0, 0.1], [0.3, 0.0, 0.2]]), np.zeros((2, 3)), m, h)
    zero = [np.zeros(2) for _ in range(3)]
    for dR in (0.0, 1e-3, 0.2, 0.9, 2.7, 11.0, 200.0, 5000.0):
        for dz in (0.0, 1e-7, 0.11, -0.4999, 0.5):
            if dR == 0.0 and abs(dz) < 1e-3 and dz != 0.0:
                continue  # coincident but for a rounding
            z = np.array([0.5, 0.5 - dz])
            sc.steps_cyl_set_state(sim.ctx, np.array([dR, 0.0]), np.zeros(2), z, *zero)
            a = sim.forces()
            assert sc.steps_cyl_last_eval(sim.ctx)["symmetric"]
            # the kernels see dz wrapped; z is exact in FP32 but for the 1e-7 case
            d = (z[0] - z[1]) - np.rint(z[0] - z[1])
            sr, sz, ar, az = image_sums(dR, d, hh, n_cut)
            unit = 1e-11  # the fixed-point accumulators' unit, times a few
            assert abs(a[0, 0] + m[1] * dR * sr) <= 2e-6 * m[1] * dR * ar + unit, (dR, dz, a[0, 0], m[1] * dR * sr)
            assert abs(a[0, 1]) <= unit
            if abs(d) != 0.5:  # at half a period the sign of the wrapped dz is the rounding's
                assert abs(a[0, 2] + m[1] * sz) <= 2e-6 * m[1] * az + unit, (dR, dz, a[0, 2], m[1] * sz)
            assert np.allclose(m[0] * a[0], -m[1] * a[1], rtol=0, atol=2e-6 * m[0] * m[1] * (dR * ar + az) + unit)
    sim.close()


@pytest.mark.parametrize("n", [2, 31, 33, 64, 65, 128, 129, 160, 700])
@pytest.mark.parametrize("law", ["literal", "ratio8"])
def test_plain_window_sizes(env, n, law):
    torch, sc, shard = env
    d = ics.particle_load(n, 900 + n, 1.0, displaced=True, eps_law=law)
    sim = sc.Simulation(sc.Config(n_cut=24), d["pos"], d["vel"], d["m"], d["h"])
    med, p999, mx = stats(sim.forces(), oracle_accel(d["pos"], d["m"], d["h"], 24))
    sim.close()
    assert med <= 1e-5 and p999 <= 1e-3, (med, p999, mx)


@pytest.mark.parametrize("n_cut,n0", [(16, 4), (23, 4), (24, 4), (64, 4), (64, 2), (12, 5), (0, 4), (0, 3)])
@pytest.mark.parametrize("law", ["literal", "ratio8"])
@pytest.mark.parametrize("read", ["cic", "tsc"])
def test_table_forms_match_row_kernels(env, n_cut, n0, law, read):
    torch, sc, shard = env
    n = 1100
    w = ics.WORKLOADS["surrogate_n65536"]
    d = ics.particle_load(n, 71, w.M_tot, displaced=True, rho_bar=w.rho_bar, eps_law=law)
    inf = n_cut == 0
    cfg = sc.Config(n_cut=n_cut, n0=n0, rho_bar=w.rho_bar, reorder_every=-1,
                    tail=sc.STEPS_TAIL_TABLE if inf else sc.STEPS_TAIL_FULL,
                    background=sc.STEPS_BG_INFINITE if inf else sc.STEPS_BG_FINITE)

    def forces(rank=None):
        sim = sc.Simulation(cfg, d["pos"], d["vel"], d["m"], d["h"])
        if read == "tsc":
            sc.steps_cyl_set_table_read(sim.ctx, sc.STEPS_TABLE_READ_TSC)
        if not inf or read == "tsc":
            sc.steps_cyl_build_tail_table(sim.ctx, 129, 17, err_median=1.0, err_p999=1.0)
        sc.steps_cyl_set_tail(sim.ctx, sc.STEPS_TAIL_TABLE)
        if rank is not None:
            shard.GpuRows(sim, rank, 2)
        a = sim.forces()
        assert sc.steps_cyl_last_eval(sim.ctx)["symmetric"] == (rank is None)
        sim.close()
        return a

    r = rel_err(forces(), forces(0) + forces(1))
    assert np.median(r) <= 2e-6 and r.max() <= 1e-4, (np.median(r), r.max())
