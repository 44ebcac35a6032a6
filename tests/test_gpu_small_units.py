"""The symmetric kernels' units at small sizes (quarter tiles, their steps split over one, two
and four units) against the FP64 oracle, for the plain window, the table and the network, and
momentum: each pair adds the same to both sides. Bounds as for the FP32 forms elsewhere."""
import numpy as np
import pytest

from gpu_helpers import oracle_accel, seeded_surrogate, stats
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


@pytest.mark.parametrize("n", [2, 65, 128, 129, 700, 1408, 1409, 2050, 3000])
@pytest.mark.parametrize("form", ["plain", "kahan", "table", "network"])
def test_against_oracle(sc, n, form):
    d = ics.particle_load(n, 70 + n, 1.0)
    cfg = sc.Config(n_cut=24, precision=sc.STEPS_FP32_PLAIN if form == "plain" else sc.STEPS_FP32_KAHAN,
                    background=sc.STEPS_BG_OFF)
    sim = sc.Simulation(cfg, d["pos"], d["vel"], d["m"], d["h"])
    if form == "table":
        sc.steps_cyl_build_tail_table(sim.ctx)
        sc.steps_cyl_set_tail(sim.ctx, sc.STEPS_TAIL_TABLE)
    elif form == "network":
        seeded_surrogate(sc, sim.ctx, 5, 24, 4)
        sc.steps_cyl_set_tail(sim.ctx, sc.STEPS_TAIL_SURROGATE)
    a = sim.forces()
    assert sc.steps_cyl_last_eval(sim.ctx)["symmetric"]
    assert np.array_equal(a, sim.forces())
    sim.close()
    net = (d["m"][:, None] * a).sum(0)
    assert np.all(np.abs(net) <= 1e-6 * (d["m"][:, None] * np.abs(a)).sum())
    if form != "network":  # (a seeded network is no model of the tail)
        med, _, mx = stats(a, oracle_accel(d["pos"], d["m"], d["h"], 24, background=0))
        assert med <= 1e-5 and mx <= 1e-3, (med, mx)
