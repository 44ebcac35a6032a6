"""Particles very far from the others (up to where dR^2 is infinite in FP32, and in FP64): they are
accepted, and the forces among the others are what they are without them. 2e-6: the relative error of
an FP32 force is some 1e-7 per component, with a wide margin for particles whose sum nearly cancels
(1e-12 for FP64)."""
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


def load(far):
    d = ics.particle_load(200, 8, 1.0)
    pos = np.vstack([d["pos"]] + [[[f, 0.3 * f, 0.25]] for f in far])
    k = len(far)
    return pos, np.append(d["m"], np.full(k, d["m"][0])), np.append(d["h"], np.full(k, d["h"][0]))


def check(a, ref, tol):
    assert np.all(np.isfinite(a))
    # the far particles' own pull, 2 n_cut m / dR^2, is below rounding from dR = 1e9 on
    err = np.linalg.norm(a[:200] - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.quantile(err, 0.95) <= tol and err.max() <= 20 * tol, (np.quantile(err, 0.95), err.max())


@pytest.mark.parametrize("form,n_cut,soft", [("kahan", 12, 1.0), ("plain", 64, 1.0), ("kahan", 24, 40.0), ("kahan", 5, 1.0),
                                             ("fp64", 5, 1.0), ("fp64", 24, 1.0), ("r3", 1, 1.0), ("r3 fp64", 1, 1.0)])
def test_context(sc, form, n_cut, soft):
    pre = {"kahan": sc.STEPS_FP32_KAHAN, "plain": sc.STEPS_FP32_PLAIN, "r3": sc.STEPS_FP32_KAHAN}.get(form, sc.STEPS_FP64)
    kw = dict(n_cut=n_cut, background=sc.STEPS_BG_OFF, precision=pre, R_sim=2.0)
    if form.startswith("r3"):
        kw.update(topology=sc.STEPS_TOPO_R3)
    far = [1e9, 1e11, 1e22] + ([1e160] if "fp64" in form else [])
    out = []
    for f in ([], far):
        pos, m, h = load(f)
        sim = sc.Simulation(sc.Config(**kw), pos, np.zeros_like(pos), m, soft * h)
        out.append(sim.forces())
        sim.close()
    check(out[1], out[0], 1e-12 if "fp64" in form else 2e-6)


@pytest.mark.parametrize("n_cut", [5, 12, 64])
def test_noalloc(sc, n_cut):
    import torch
    out = []
    for f in ([], [1e9, 1e11, 1e22]):
        pos, m, h = load(f)
        cols = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (*pos.T, m, h)]
        a = [torch.empty_like(cols[0]) for _ in range(3)]
        sc.steps_cyl_pair_accel_noalloc(*cols, 1.0, 1.0, n_cut, sc.STEPS_FP32_KAHAN, *a,
                                        stream=torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        out.append(torch.stack(a, 1).cpu().numpy())
    check(out[1], out[0], 2e-6)
