"""Charge density by exact integer sums over runs of equal cells (FP32 positions) against cloud-in-cell in numpy: piles that
end before, at and after a run's and a warp's edge, scattered particles, particles on nodes, an order no longer sorted by
cell, and gamma over a narrow and over a wide range (which takes the FP64 sums).

Both sides weigh the same stored state; numpy adds fewer than 2000 terms of one sign to a node in FP64, an error below
2000 * 2^-53 = 2.2e-13 of the largest sum."""
import numpy as np
import pytest

from paper_0904_0232_gb300.grpic import Simulation

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _cic(shape, x, w):
    rho = np.zeros(shape)
    i0 = np.floor(x[:3]).astype(int)
    f = x[:3] - i0
    for dk in (0, 1):
        for dj in (0, 1):
            for di in (0, 1):
                W = (f[0] if di else 1 - f[0]) * (f[1] if dj else 1 - f[1]) * (f[2] if dk else 1 - f[2])
                np.add.at(rho, (i0[2] + dk, i0[1] + dj, i0[0] + di), w * W)
    return rho


def _check(sim, q, c):
    shape = sim.shape
    x, u, _ = sim.get_particles(0)
    for got, w in ((sim.charge_density(), np.full(x.shape[1], q)), (sim.charge_density(with_gamma=True), q * u[3] / c)):
        ref = _cic(shape, x, w)
        assert np.abs(got - ref).max() <= 2.2e-13 * np.abs(ref).max()


def _state(x, umax, rng):
    n = x.shape[1]
    u = np.zeros((4, n))
    u[0] = umax ** rng.random(n) - 1.0
    u[3] = np.sqrt(1.0 + u[0] ** 2)
    return np.vstack([x, np.zeros((1, n))]), u


@pytest.mark.parametrize("prec", ["fp32_mixed", "fp64"])
@pytest.mark.parametrize("umax", [1.0, 30.0, 1e6])
@pytest.mark.parametrize("piles", [[1], [7, 8, 9], [31, 32, 33], [40, 1, 100, 256, 5], []])
def test_piles(piles, umax, prec):
    rng = np.random.default_rng(len(piles) + 7)
    dims = (13, 9, 11)
    sim = Simulation(*dims, 0.0, 0.0, 1.0, 0.4, precision=prec)
    xs = [np.array([[1 + i % 10], [1 + (2 * i) % 6], [1 + (i * i) % 8]]) + rng.random((3, k)) * 0.999
          for i, k in enumerate(piles)]
    # scattered ones as well, some on nodes and in the last cells
    xs.append(1.0 + rng.random((3, 333)) * (np.array(dims).reshape(3, 1) - 3.0))
    xs.append(np.floor(xs[-1][:, :50]))
    xs.append(np.array(dims).reshape(3, 1) - 2.0 - 0.5 * rng.integers(0, 2, (3, 9)))
    x4, u = _state(np.hstack(xs).astype(np.float32).astype(np.float64), umax, rng)
    sim.load_particles(0, 0.0, -0.37, x4, u, np.arange(x4.shape[1], dtype=np.uint32))
    _check(sim, -0.37, 1.0)


def test_unsorted():
    rng = np.random.default_rng(5)
    dims = (20, 17, 15)
    sim = Simulation(*dims, 0.0, 0.0, 1.0, 0.4, precision="fp32_mixed")
    sim.set_tuning(sort_interval=64)
    x = 4.0 + rng.random((3, 4000)) * (np.array(dims).reshape(3, 1) - 8.0)
    x4, u = _state(x.astype(np.float32).astype(np.float64), 4.0, rng)
    sim.load_particles(0, 0.0, 1.5, x4, u, np.arange(4000, dtype=np.uint32))
    sim.step(5)
    _check(sim, 1.5, 1.0)
