"""Training steps of the learned tail (surrogate_train.cuh) against the oracle's gradient and
Adam step in FP64, from the same samples, initial weights and sample orders: minibatches of one
block, of several, of one with an incomplete last block, and the whole set; and a batch larger
than the cooperative launch takes, against the oracle as well.

Adam moves a weight by about lr per step whatever the gradient's size, so a gradient's relative
error enters: FP32 sums of n terms with cancellation leave 1e-4 of it for all but small gradients
(99% of the weights), and a gradient that is itself rounding moves its weight by lr in either
direction (bounded by 2 lr per step)."""
import math

import numpy as np
import pytest

import oracle
from paper_2602_20787_gb300 import ics

pytestmark = pytest.mark.gpu
N_CUT, N0 = 16, 4


@pytest.fixture(scope="module")
def sc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_20787_gb300 import steps_cyl
    steps_cyl.load()
    return steps_cyl


class SplitMix:
    def __init__(self, s):
        self.s = s

    def next(self):
        m = (1 << 64) - 1
        self.s = (self.s + 0x9E3779B97F4A7C15) & m
        z = self.s
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
        return z ^ (z >> 31)

    def uniform(self):
        return (self.next() >> 11) * 2.0 ** -53


def reference(ns, batch, epochs, lr, seed, dR_max):
    rng, A = SplitMix(seed), N0 + 0.5
    u, r = np.zeros((ns, 3)), np.zeros((ns, 2))
    for s in range(ns):
        dR, dz, h = dR_max * math.sqrt(rng.uniform()), 0.5 * rng.uniform(), A * rng.uniform()
        u[s] = oracle.surrogate_inputs(dR, dz, h, N0, dR_max)
        r[s] = (np.array(oracle.tail_sums(dR, dz, h, 1.0, N_CUT, N0)) - oracle.tail_base(dR, dz, N_CUT, N0)) \
            / oracle.tail_envelope(dR, dz, N0)
    nt = ns - ns // 16
    mu = r[:nt].mean(0)
    t = (r - mu) / r[:nt].std(0)
    w = []
    for cnt, fan in ((96, 3), (32, 3), (1024, 32), (32, 32), (64, 32), (2, 32)):
        w += [np.float32((2.0 * rng.uniform() - 1.0) / math.sqrt(fan)) for _ in range(cnt)]
    w = np.array(w, dtype=np.float64)
    m1, m2, step = np.zeros_like(w), np.zeros_like(w), 0
    for ep in range(epochs):
        order = list(range(nt))
        for k in range(nt - 1, 0, -1):
            j = rng.next() % (k + 1)
            order[k], order[j] = order[j], order[k]
        for first in range(0, nt, batch):
            sel = order[first:first + batch]
            step += 1
            g = oracle.mlp_loss_grad(w, u[sel], t[sel])[1]
            oracle.adam_step(w, g, m1, m2, lr * 0.5 * (1 + math.cos(math.pi * ep / epochs)), 0.9, 0.999, 1e-8, step)
    return w, mu, step


@pytest.mark.parametrize("ns,batch", [(1024, 64), (1024, 192), (1024, 448), (2100, 1024), (1100, 2048), (1024, 65536)])
def test_weights_after_two_epochs(sc, ns, batch):
    d = ics.particle_load(512, 3, 1.0)
    sim = sc.Simulation(sc.Config(n_cut=N_CUT, n0=N0), d["pos"], d["vel"], d["m"], d["h"])
    lr, seed, dR_max = 1e-3, 5, 6.0
    sc.steps_cyl_train_surrogate(sim.ctx, sc.steps_cyl_train_cfg_default(
        n_samples=ns, epochs=2, batch=batch, lr=lr, seed=seed, dR_max=dR_max, err_median=1e9, err_p999=1e9,
        check_particles=64))
    p = sc.steps_cyl_get_surrogate(sim.ctx)
    sim.close()
    w, mu, steps = reference(ns, batch, 2, lr, seed, dR_max)
    assert np.allclose(p[1250:1252], mu, rtol=1e-6, atol=1e-9)
    err = np.abs(p[:1250] - w)
    assert np.quantile(err, 0.99) <= 1e-4 * lr * steps + 2.0 ** -24, np.quantile(err, 0.99) / (lr * steps)
    assert err.max() <= 2 * lr * steps
