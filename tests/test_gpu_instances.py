"""Every step kernel has an instance for one box, which takes the box by value, and one for many, which
takes tables: the same boxes stepped alone and as a batch agree bit for bit, with each physics option and
boundary, in both precisions."""
import numpy as np
import pytest

from paper_1608_08748_gb300 import inputs as I

pytestmark = pytest.mark.gpu

OPTIONS = [{"chem": 0}, {"chem": 1}, {"chem": 1, "heatcool": 1}, {"chem": 1, "heatcool": 1, "ions": 1},
           {"chem": 1, "bc_y": 1}, {"chem": 0, "regul_mode": 1}]


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1608_08748_gb300 import build as B
    B.build()
    import paper_1608_08748_gb300 as M
    return M


def make(M, k, precision):
    ic = I.turbulence(8, mach=3.0, beta=1.0, seed=90 + k, shape=(9 + k, 12, 33), T_K=4000.0 if k % 2 else 100.0)
    ic["rho_h2"] = 0.1 * ic["rho"]
    if OPTIONS[k].get("ions"):
        ic["rho_hp"] = 1e-3 * ic["rho"]
    return M.from_ic(ic, precision=precision, **OPTIONS[k])


@pytest.mark.parametrize("precision", [0, 1])
def test_one_box_and_many_agree(M, precision):
    solo = [make(M, k, precision) for k in range(len(OPTIONS))]
    mixed = [make(M, k, precision) for k in range(len(OPTIONS))]
    batch = M.Batch(mixed)
    for _ in range(4):
        for s in solo:
            s.step(0.4, sync=False)
        batch.step(0.4)
    batch.sync()
    for k, (s, m) in enumerate(zip(solo, mixed)):
        s.sync()
        a, b = s.get_state(), m.get_state()
        for f in ["rho", "mom", "E", "B", "rho_h2"]:
            assert np.array_equal(a[f], b[f]), (k, f)
        assert np.array_equal(s.get_ions(), m.get_ions()), k
        assert s.diagnostics()["t"] == m.diagnostics()["t"], k
