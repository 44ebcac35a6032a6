"""A call of ten steps and ten calls of one give the same bits: the kick and drift of a step that follow
the one before in its finalize, and those in a launch of their own, with a re-ordering and a check of the
modelled tail falling inside the run or at its ends."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n", [2, 700, 3000])
@pytest.mark.parametrize("form", ["comoving", "r3", "r3 comoving", "infinite", "table", "fp64"])
def test_split_of_a_run(sc, form, n):
    kw = dict(n_cut=16, reorder_every=4, check_every=3, check_particles=64)
    if "comoving" in form:
        kw.update(comoving=True, a_start=0.1)
    if form.startswith("r3"):
        kw.update(topology=sc.STEPS_TOPO_R3, n_cut=1, R_sim=2.0, background=sc.STEPS_BG_SPHERE)
    if form == "infinite":
        kw.update(n_cut=0, tail=sc.STEPS_TAIL_TABLE, background=sc.STEPS_BG_INFINITE)
    if form == "fp64":
        kw.update(precision=sc.STEPS_FP64)
    d = ics.particle_load(n, 21, 1.0)
    vel = np.random.default_rng(2).normal(0.0, 0.01, (n, 3))
    out = []
    for calls in (1, 10):
        sim = sc.Simulation(sc.Config(**kw), d["pos"], vel, d["m"], d["h"])
        if form == "table":
            sc.steps_cyl_build_tail_table(sim.ctx)
            sc.steps_cyl_set_tail(sim.ctx, sc.STEPS_TAIL_TABLE)
        for _ in range(calls):
            sim.step(1e-3, 10 // calls)
        x, v, a, t = sim.state()
        out.append((x, v, a, t, sim.forces()))
        sim.close()
    for p, q in zip(*out):
        np.testing.assert_array_equal(p, q)
