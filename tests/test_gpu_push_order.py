"""The block -> chunk map of the push (spread): every particle is pushed once whatever the order, for launches of one block,
about a group and its tails, in blocks of one warp and of four.  All particles lie far from the hole, where the arithmetic of a
particle does not depend on the others of its warp (the order within a cell is not fixed), so the new state after one step is
the same bits as without spreading."""
import numpy as np
import pytest

from paper_0904_0232_gb300.grpic import Simulation

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _after_step(x4, u4, spread):
    n = x4.shape[1]
    sim = Simulation(28, 24, 26, 1.0, 0.5, 1.0, 0.4, precision="fp32_mixed")
    sim.set_tuning(spread=spread, sort_interval=64)
    sim.set_uniform_field(B=(0.0, 0.0, 0.1))
    sim.load_particles(0, -1.0, 1e-4, x4, u4, np.arange(n, dtype=np.uint32), umode=1)
    sim.step(1)
    x, u, ids = sim.get_particles(0)
    order = np.argsort(ids)
    return x[:, order], u[:, order], ids[order]


@pytest.mark.parametrize("n", [1, 32, 33, 127, 128 * 3, 32 * 17 + 5, 32 * 64, 32 * 67, 20000, 311296, 311297, 700001])
def test_order_does_not_matter(n):
    rng = np.random.default_rng(n)
    x = 2.0 + rng.random((3, n)) * (np.array([[28.0], [24.0], [26.0]]) - 5.0)
    u = rng.standard_normal((4, n)) * 0.1
    # |z - z_c| >= 9 > near radius 8.5 (4 m + |a| + 4)
    x[2] = np.where(rng.random(n) < 0.5, 1.5 + 2.0 * rng.random(n), 21.5 + 2.0 * rng.random(n))
    x4 = np.vstack([x, np.zeros((1, n))])
    want = _after_step(x4, u, 0)
    for spread in (1, 16):
        got = _after_step(x4, u, spread)
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
