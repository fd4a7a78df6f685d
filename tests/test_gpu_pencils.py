"""Pencils of every length.  The executor picks the pencils' length from the boxes of a launch, and the FP64
kernels gather Step 4 of Sec. 2.1 over each warp: the same boxes, with lines of fewer faces than a
pencil and one more than a multiple and with partly empty warps, stepped alone (short pencils) and
beside a large box (long pencils) agree bit for bit."""
import numpy as np
import pytest

from paper_1608_08748_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 1, 7), (2, 3, 33), (5, 17, 8), (9, 8, 31), (16, 20, 24)]  # (nz, ny, nx)


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1608_08748_gb300 import build as B
    B.build()
    import paper_1608_08748_gb300 as M
    return M


def rough(shape, seed, outflow=-1):
    """Values with jumps, plateaus and ramps, so that every limiter and Step 4 act."""
    rng = np.random.default_rng(seed)

    def field(lo, hi):
        f = rng.uniform(lo, hi, size=shape)
        ramp = np.cumsum(rng.choice([0.0, 0.02, 0.3], size=shape), axis=-1)
        return np.where(rng.random(shape) < 0.5, f, lo + (hi - lo) * (ramp % 1.0))
    rho, p = field(0.5, 1.5), field(0.5, 1.5)
    v = np.stack([field(-0.3, 0.3) for _ in range(3)])
    B = np.stack([np.full(shape, c) for c in (0.4, -0.3, 0.2)])
    ic = I.conserved(rho, v, p, B, 5.0 / 3.0)
    ic.update(gamma=5.0 / 3.0, dx=1.0 / max(shape), options={"bc_x": 0, "bc_y": 0, "bc_z": 0, "chem": 0})
    if outflow >= 0:
        ic["options"]["bc_" + "xyz"[outflow]] = 1
    return ic


@pytest.mark.parametrize("precision", [0, 1])
def test_results_do_not_depend_on_the_length(M, precision):
    solo = [M.from_ic(rough(s, 70 + i), precision=precision) for i, s in enumerate(SHAPES)]
    mixed = [M.from_ic(rough(s, 70 + i), precision=precision) for i, s in enumerate(SHAPES)]
    large = M.from_ic(I.turbulence(8, mach=2.0, beta=1.0, seed=3, shape=(72, 80, 96), chem=0), precision=precision)
    batch = M.Batch(mixed + [large])
    for _ in range(2):
        for s in solo:
            s.step(0.3, sync=False)
        batch.step(0.3)
    batch.sync()
    for s, m in zip(solo, mixed):
        s.sync()
        a, b = s.get_state(), m.get_state()
        for f in ["rho", "mom", "E", "B"]:
            assert np.array_equal(a[f], b[f]), f
