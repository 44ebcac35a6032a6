"""The internal particle order, made on the device at init, set_state and every reorder_every
steps, read back from a checkpoint: the stable order of the Morton keys of (x, y) that the host
gives. Sizes around a sort tile (2,048 keys) and a single column of equal keys."""
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


def spread(v):
    for s, m in ((8, 0x00FF00FF), (4, 0x0F0F0F0F), (2, 0x33333333), (1, 0x55555555)):
        v = (v | (v << s)) & m
    return v


def morton(x, y):
    span = max(x.max() - x.min(), y.max() - y.min(), 1e-300)
    q = [np.clip(np.floor((c - c.min()) / span * 65536.0), 0, 65535).astype(np.uint64) for c in (x, y)]
    return np.argsort(spread(q[0]) | (spread(q[1]) << np.uint64(1)), kind="stable")


def order_of(sc, ctx, n, path):
    sc.steps_cyl_checkpoint(ctx, str(path))
    return np.frombuffer(open(path, "rb").read()[-4 * n:], dtype=np.int32)


@pytest.mark.parametrize("n", [2, 33, 2047, 2048, 2049, 5000])
def test_order(sc, n, tmp_path):
    d = ics.particle_load(n, 11 + n, 1.0)
    sim = sc.Simulation(sc.Config(n_cut=4, reorder_every=1), d["pos"], d["vel"], d["m"], d["h"])
    f = tmp_path / "a.ckpt"
    assert np.array_equal(order_of(sc, sim.ctx, n, f), morton(d["pos"][:, 0], d["pos"][:, 1]))
    a = sim.forces()
    # new positions: another order, masses and softenings carried along
    p = d["pos"][::-1].copy() * [1.0, -0.5, 1.0]
    sc.steps_cyl_set_state(sim.ctx, *(np.ascontiguousarray(p[:, k]) for k in range(3)), *(np.zeros(n) for _ in range(3)))
    perm = order_of(sc, sim.ctx, n, f)
    assert np.array_equal(perm, morton(p[:, 0], p[:, 1]))
    other = sc.Simulation(sc.Config(n_cut=4), p, np.zeros_like(p), d["m"], d["h"])
    assert np.array_equal(sim.forces(), other.forces())
    other.close()
    # a step: the rows of the old order, sorted again (ties keep the old internal order)
    sim.step(1e-4, 1)
    x = np.array(sim.state()[0])
    assert np.array_equal(order_of(sc, sim.ctx, n, f), perm[morton(x[perm, 0], x[perm, 1])])
    sim.close()
    # all on one column, and the caller's order kept
    for every, q in ((1, d["pos"] * [0.0, 0.0, 1.0] + [0.25, 0.5, 0.0]), (-1, d["pos"])):
        sim = sc.Simulation(sc.Config(n_cut=4, reorder_every=every, background=sc.STEPS_BG_OFF), q, d["vel"], d["m"], d["h"])
        assert np.array_equal(order_of(sc, sim.ctx, n, f), np.arange(n))
        sim.close()
    assert a.shape == (n, 3)
