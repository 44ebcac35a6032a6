"""A few particles softened over many periods among narrow ones: steps of a warp that take the walk for a
pair of theirs take it for all. Against the oracle, with the action equal to the reaction; and the forces in
the library's own particle order against those in the caller's."""
import numpy as np
import pytest

import oracle
from paper_2602_20787_gb300 import ics
from gpu_helpers import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_20787_gb300 import steps_cyl
    steps_cyl.load()
    return steps_cyl


@pytest.mark.parametrize("kahan", [True, False])
@pytest.mark.parametrize("n_cut", [12, 16, 24, 64])
@pytest.mark.parametrize("wide", [9.0, 30.0])
def test_wide_among_narrow(sc, n_cut, wide, kahan):
    n = 700
    d = ics.particle_load(n, 31, 1.0)
    h = np.full(n, 0.05)
    h[[5, 130, 131, 600]] = wide
    cfg = sc.Config(n_cut=n_cut, background=sc.STEPS_BG_OFF,
                    precision=sc.STEPS_FP32_KAHAN if kahan else sc.STEPS_FP32_PLAIN)
    sim = sc.Simulation(cfg, d["pos"], d["vel"], d["m"], h)
    a = sim.forces()
    sim.close()
    r = rel_err(a, oracle.pair_field(d["pos"], d["m"], h, 1.0, 1.0, n_cut))
    assert np.median(r) <= 1e-6 and r.max() <= 1e-4, (np.median(r), r.max())
    # a pair's two sides differ by the rounding of its sums' groups
    net = (d["m"][:, None] * a).sum(0)
    assert np.all(np.abs(net) <= 1e-6 * (d["m"][:, None] * np.abs(a)).sum())


@pytest.mark.parametrize("n", [2, 33, 2047, 2049, 5000])
def test_forces_do_not_depend_on_the_order(sc, n):
    d = ics.particle_load(n, 11 + n, 1.0)
    out = []
    for every in (1, -1):
        sim = sc.Simulation(sc.Config(n_cut=4, background=sc.STEPS_BG_OFF, reorder_every=every), d["pos"], d["vel"],
                            d["m"], d["h"])
        out.append(sim.forces())
        sim.close()
    r = rel_err(out[0], out[1])
    assert np.median(r) <= 1e-6 and r.max() <= 1e-4, (np.median(r), r.max())
