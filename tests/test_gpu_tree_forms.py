"""The octree's walk with every leaf opened (theta near 0) is the direct sum: its forms (near
range 4 in closed form, any other, the nearest-image table, R^3) against the direct kernels of the
same form, around the sizes of a group, a leaf and a list, with leaves of one particle to more
than a warp takes at once. Both sides are FP32 with the same tail; the bounds are those of the
octree's tests against the oracle."""
import numpy as np
import pytest

from gpu_helpers import stats
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


def both(sc, d, leaf, theta, frame, **kw):
    out = []
    for force in (sc.STEPS_FORCE_DIRECT, sc.STEPS_FORCE_OCTREE):
        sim = sc.Simulation(sc.Config(force=force, theta=theta, leaf_size=leaf, **kw), d["pos"], d["vel"], d["m"], d["h"])
        if force == sc.STEPS_FORCE_OCTREE and frame:
            sc.steps_cyl_tree_frame(sim.ctx, *frame)
        out.append(sim.forces())
        if force == sc.STEPS_FORCE_OCTREE:
            n = len(d["m"])
            assert sc.steps_cyl_tree_stats(sim.ctx)["interactions"] == n * n
        sim.close()
    return out


@pytest.mark.parametrize("n,leaf", [(2, 1), (31, 1), (33, 4), (95, 64), (129, 64), (700, 1), (1500, 33)])
@pytest.mark.parametrize("n0", [0, 2, 4])
@pytest.mark.parametrize("soft", [0.1, 6.0])
def test_cylinder(sc, n, leaf, n0, soft):
    d = ics.particle_load(n, 40 + n, 1.0, displaced=True, rho_bar=1.0 / (np.pi * ics.R_SIM ** 2), eps_law="ratio8")
    d["h"] = d["h"] * soft
    a, b = both(sc, d, leaf, 1e-3, (0.37, 1.1), n_cut=0, n0=n0, tail=sc.STEPS_TAIL_TABLE,
                background=sc.STEPS_BG_INFINITE)
    med, _, mx = stats(b, a)
    assert med <= 1e-6 and mx <= 2e-5, (med, mx)


@pytest.mark.parametrize("n,leaf", [(31, 1), (129, 64), (1500, 16)])
@pytest.mark.parametrize("soft", [1.0, 40.0])
def test_r3(sc, n, leaf, soft):
    d = ics.ball_load(n, 40 + n)
    d["h"] = d["h"] * soft
    a, b = both(sc, d, leaf, 1e-3, None, topology=sc.STEPS_TOPO_R3, n_cut=1, R_sim=2.0, background=sc.STEPS_BG_OFF)
    med, _, mx = stats(b, a)
    assert med <= 1e-6 and mx <= 2e-5, (med, mx)
