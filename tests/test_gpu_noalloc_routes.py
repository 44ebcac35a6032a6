"""The allocation-free call's two routes: each pair once where the fixed-point sums have a scale, rows
against every j where they have none (softenings too small), both against the FP64 oracle at sizes
around the blocks and the split of a tile's steps; and a coordinate that is not a number, which
makes every acceleration one. Bounds as in the other tests of this call."""
import numpy as np
import pytest

import oracle
from paper_2602_20787_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_20787_gb300 import steps_cyl
    steps_cyl.load()
    return torch, steps_cyl


def accel(torch, sc, d, n_cut, precision):
    cols = [torch.tensor(np.ascontiguousarray(d["pos"][:, k]), device="cuda") for k in range(3)]
    m, h = torch.tensor(d["m"], device="cuda"), torch.tensor(d["h"], device="cuda")
    out = [torch.zeros_like(m) for _ in range(3)]
    st = torch.cuda.current_stream()
    sc.steps_cyl_pair_accel_noalloc(*cols, m, h, 1.0, 1.0, n_cut, precision, *out, stream=st.cuda_stream)
    st.synchronize()
    return torch.stack(out, 1).cpu().numpy()


@pytest.mark.parametrize("n", [2, 129, 700, 3001, 8200])
@pytest.mark.parametrize("soft", [1.0, 1e-4])
@pytest.mark.parametrize("n_cut", [5, 16])
def test_both_routes(env, n, soft, n_cut):
    torch, sc = env
    d = ics.particle_load(n, 90 + n, 1.0)
    d["h"] = d["h"] * soft
    idx = np.unique(np.concatenate([np.arange(min(64, n)), np.arange(max(0, n - 64), n)]))
    ref = oracle.pair_field(d["pos"], d["m"], d["h"], 1.0, 1.0, n_cut, idx=idx)
    for precision in (sc.STEPS_FP32_KAHAN, sc.STEPS_FP32_PLAIN):
        a = accel(torch, sc, d, n_cut, precision)
        r = np.linalg.norm(a[idx] - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert np.median(r) <= 1e-5 and r.max() <= 1e-3, (np.median(r), r.max())
        assert np.array_equal(a, accel(torch, sc, d, n_cut, precision))


@pytest.mark.parametrize("soft", [1.0, 1e-4])
def test_not_a_number(env, soft):
    torch, sc = env
    d = ics.particle_load(300, 4, 1.0)
    d["pos"][17, 0] = np.nan
    d["h"] = d["h"] * soft
    assert np.all(np.isnan(accel(torch, sc, d, 16, sc.STEPS_FP32_KAHAN)[:, 0]))
