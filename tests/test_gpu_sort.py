"""The counting sort of all species in one set of launches: species of very different sizes (none, one, a few, many), bins
that end at, before and after a tile's edge (2048 bins), removed particles, species 2 and 3 with scratch of their own, a
grid of more than 16384 tiles, and repeated loads and sorts whose bins have to be zero again."""
import numpy as np
import pytest

from paper_0904_0232_gb300.grpic import GRPIC_STAGE_SORT, Simulation

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _load(sim, dims, s, k, rng):
    hi = np.array(dims).reshape(3, 1) - 2.0
    x = (1.0 + rng.random((3, k)) * (hi - 1.0)).astype(np.float32).astype(np.float64)
    u = np.vstack([rng.standard_normal((3, k)) * 0.05, np.zeros((1, k))])
    u[3] = np.sqrt(1.0 + (u[:3] ** 2).sum(0))
    sim.load_particles(s, 0.0, 0.0, np.vstack([x, np.zeros((1, k))]), u, np.arange(k, dtype=np.uint32))
    return x


def _check(sim, dims, s, x):
    px, _, ids = sim.get_particles(s)
    assert px.shape[1] == x.shape[1] and np.array_equal(np.sort(ids), np.arange(x.shape[1]))
    assert np.array_equal(px[:3], x[:, ids])
    c = np.floor(px[:3]).astype(np.int64)
    key = (c[2] * dims[1] + c[1]) * dims[0] + c[0]
    assert np.all(np.diff(key) >= 0)


@pytest.mark.parametrize("prec", ["fp32_mixed", "fp64"])
@pytest.mark.parametrize("dims", [(16, 16, 8), (23, 89, 1 + 7), (32, 8, 16), (17, 19, 13)])
@pytest.mark.parametrize("sizes", [(0, 1), (5000, 3, 0, 70000), (31, 32, 33, 1)])
def test_species_of_all_sizes(dims, sizes, prec):
    rng = np.random.default_rng(3)
    sim = Simulation(*dims, 0.0, 0.0, 1.0, 0.4, precision=prec)
    for _ in range(2):  # the second round reuses dirty bins
        xs = [_load(sim, dims, s, k, rng) for s, k in enumerate(sizes)]
        for _ in range(3):
            sim.stage(GRPIC_STAGE_SORT)
        for s, x in enumerate(xs):
            _check(sim, dims, s, x)
    n0 = sum(sizes)
    sim.step(6)  # free flight: particles leave through the faces and are dropped
    st = sim.stats()
    assert st["removed_outer"] > 0 or n0 < 200
    assert [sim.num_particles(s) for s in range(len(sizes))] == st["n_alive"][:len(sizes)]
    assert sum(st["n_alive"]) + st["removed_outer"] == n0
    for s in range(len(sizes)):
        px, _, ids = sim.get_particles(s)
        assert len(np.unique(ids)) == ids.size
        c = np.floor(px[:3]).astype(np.int64)
        assert np.all(np.diff((c[2] * dims[1] + c[1]) * dims[0] + c[0]) >= 0)


def test_more_than_16384_tiles():
    dims = (330, 330, 330)
    sim = Simulation(*dims, 0.0, 0.0, 1.0, 0.4, precision="fp32_mixed")
    rng = np.random.default_rng(5)
    xs = [_load(sim, dims, s, k, rng) for s, k in enumerate((200000, 77))]
    sim.stage(GRPIC_STAGE_SORT)
    for s, x in enumerate(xs):
        _check(sim, dims, s, x)
