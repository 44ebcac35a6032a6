"""A step whose position overflows ends with the device error, in every form that can meet it: one
particle's velocity is finite but carries its z beyond FP64's range, so that the wrap leaves no
number. Over the infinite window the softened images of the tail are walked up to a bound, which
tests/test_soft_bound.py shows to be finite for any position."""
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


@pytest.mark.parametrize("form", ["infinite", "infinite n0 = 2", "octree", "window", "walk", "fp64", "r3"])
def test_overflowing_step(sc, form):
    n = 300
    d = ics.particle_load(n, 4, 1.0)
    kw = dict(n_cut=16, background=sc.STEPS_BG_OFF)
    if form.startswith("infinite") or form == "octree":
        kw.update(n_cut=0, tail=sc.STEPS_TAIL_TABLE, n0=2 if "n0" in form else 4)
    if form == "octree":
        kw.update(force=sc.STEPS_FORCE_OCTREE)
    if form == "walk":
        kw.update(n_cut=5)
    if form == "fp64":
        kw.update(precision=sc.STEPS_FP64)
    if form == "r3":
        kw.update(topology=sc.STEPS_TOPO_R3, n_cut=1, R_sim=2.0)
    v = np.zeros_like(d["pos"])
    v[17, 2] = 1e300
    sim = sc.Simulation(sc.Config(**kw), d["pos"], v, d["m"], d["h"])
    with pytest.raises(sc.StepsError) as e:
        sim.step(1e10, 1)
    assert e.value.code == sc.STEPS_EDEVICE
    sim.close()
