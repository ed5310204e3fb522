"""A batch over contexts that change between its steps: reloaded with fewer and then more particles (up to the
counts of its creation), other charges, other stores (a load beyond the capacity moves them) or another launch
shape, it steps them as they stand. Each is compared with the same contexts stepped on their own."""
import numpy as np
import pytest

from paper_0904_0232_gb300 import synth
from paper_0904_0232_gb300.grpic import (GRPIC_U_COV_SPATIAL, GrpicError, Simulation, grpic_batch_create,
                                         grpic_batch_destroy, grpic_batch_step)
from test_gpu_batch import _compare

pytestmark = pytest.mark.gpu
N, M, A, COUNT = 24, 1.5, 1.2, 1000


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _plasma(seed, n):
    rng = np.random.default_rng(seed)
    c = 0.5 * (N - 1)
    x = rng.uniform(2.0, N - 3.0, (3, 2 * n + 64))
    x = x[:, ((x - c) ** 2).sum(0) > 16.0][:, :n]
    assert x.shape[1] == n
    return np.vstack([x, np.zeros((1, n))]), synth.maxwell_juettner(rng, n, 0.01)


def _load(sims, seed, n, scale):
    for k, sim in enumerate(sims):
        for s, qm in enumerate((-1.0, 0.5)):
            x, u = _plasma(seed + 10 * k + s, n)
            sim.load_particles(s, qm * scale, qm * scale * 1e-2, x, u, np.arange(n, dtype=np.uint32),
                               GRPIC_U_COV_SPATIAL)


def _start(prec, count=COUNT):
    sides = []
    for _ in range(2):
        sims = [Simulation(N, N, N, M, A, 1.0, 0.4, precision=prec) for _ in range(2)]
        for sim in sims:
            sim.set_uniform_field(B=(0.0, 0.0, 0.05))
        _load(sims, 1, count, 1.0)
        sides.append(sims)
    return sides, grpic_batch_create([s.handle for s in sides[0]])


def _step_and_compare(sides, b, prec, n=2):
    grpic_batch_step(b, n)
    for x, y in zip(*sides):
        y.step(n)
        _compare(x, y, prec, 1.0 if prec == "fp64" else 16.0)


@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
def test_fewer_then_more_particles_with_other_charges(prec):
    sides, b = _start(prec)
    for seed, n, scale in ((2, COUNT // 2, 1.0), (3, COUNT, 1.0), (4, COUNT - 1, 3.0), (5, 0, 1.0), (6, COUNT, -2.0)):
        for sims in sides:
            _load(sims, seed, n, scale)
        _step_and_compare(sides, b, prec)  # (two steps: the parities are those of the last capture)
    grpic_batch_destroy(b)


@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
def test_moved_stores(prec):
    sides, b = _start(prec)
    _step_and_compare(sides, b, prec)
    for sims in sides:
        _load(sims, 2, 3 * COUNT, 1.0)  # beyond the stores: others are allocated
    with pytest.raises(GrpicError):
        grpic_batch_step(b, 1)  # more than the batch was built for
    for sims in sides:
        _load(sims, 3, COUNT - 7, 1.0)
    _step_and_compare(sides, b, prec)
    grpic_batch_destroy(b)


def test_other_shapes_and_a_species_the_batch_does_not_know():
    sides, b = _start("fp32_mixed")
    _step_and_compare(sides, b, "fp32_mixed")
    for sims in sides:
        for sim in sims:
            t = sim.tuning()
            t.update(far_min_blocks=5, area_table=1, spread=2)
            sim.set_tuning(**t)
    _step_and_compare(sides, b, "fp32_mixed")
    x, u = _plasma(9, 10)
    sides[0][0].load_particles(2, 1.0, 1e-3, x, u, np.arange(10, dtype=np.uint32), GRPIC_U_COV_SPATIAL)
    with pytest.raises(GrpicError):
        grpic_batch_step(b, 1)
    grpic_batch_destroy(b)
