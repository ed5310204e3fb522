"""The push picks blocks of one warp for small launches and of four for large ones, and runs small species beside each
other: particles on either side of the line against the oracle, and in FP64, where a particle's result does not depend
on its warp, the same bits for every number of particles in the last block."""
import numpy as np
import pytest

import oracle as O
from parity_util import TOL
from paper_0904_0232_gb300 import synth
from paper_0904_0232_gb300.grpic import (GRPIC_STAGE_B_HALF, GRPIC_STAGE_PUSH_DEPOSIT, GRPIC_STAGE_ZERO_J,
                                         GRPIC_U_COV_SPATIAL, Simulation)

pytestmark = pytest.mark.gpu
LINE = 311296  # particles of one species up to which a launch is small
N, M, A = 40, 2.0, 1.8
QMS = (-1.0, 1.0)


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _inputs(k):
    rng = np.random.default_rng(7)
    x = rng.uniform(1.0, N - 2.0, (3, k)).astype(np.float32).astype(np.float64)
    c = 0.5 * (N - 1)
    x = x[:, ((x - c) ** 2).sum(0) > 25.0]  # outside r_+, which no particle then reaches in a step
    return x, [synth.maxwell_juettner(rng, x.shape[1], 0.01) for _ in QMS], synth.random_fields((N, N, N), 11)


def _push(x, u, fields, prec, quad=2):
    sim = Simulation(N, N, N, M, A, 1.0, 0.4, precision=prec, quad_order=quad)
    sim.set_fields(*fields)
    k = x.shape[1]
    for s, qm in enumerate(QMS):
        sim.load_particles(s, qm, qm * 1e-3, np.vstack([x, np.zeros((1, k))]), u[s], np.arange(k, dtype=np.uint32),
                           GRPIC_U_COV_SPATIAL)
    for stage in (GRPIC_STAGE_B_HALF, GRPIC_STAGE_ZERO_J, GRPIC_STAGE_PUSH_DEPOSIT):
        sim.stage(stage)
    out = []
    for s in range(2):
        px, pu, ids = sim.get_particles(s)
        full = np.zeros((8, k))
        full[:, ids] = np.vstack([px, pu])
        out.append(full)
    return out, sim.get_fields()[2]


@pytest.mark.parametrize("quad", [1, 2, 3])
@pytest.mark.parametrize("count", [1, 33, 5000, LINE + 9000])
def test_fp32_against_the_oracle(count, quad):
    x, u, fields = _inputs(count)
    k = x.shape[1]
    ref = O.Oracle(N, N, N, M, A, 1.0, 0.4, quad_order=quad, threads=0)
    ref.set_fields(*fields)
    for s, qm in enumerate(QMS):
        ref.load_particles(s, qm, qm * 1e-3, np.vstack([x, np.zeros((1, k))]), np.vstack([u[s], np.zeros((1, k))]),
                           np.arange(k, dtype=np.uint32), umode=1)
    ref.b_half()
    ref.zero_j()
    ref.push_deposit()
    out, J = _push(x, u, fields, "fp32_mixed", quad)
    Jr = ref.get_fields()[2]
    for s in range(2):
        px, pu, ids = ref.get_particles(s)
        assert np.abs(out[s][:3, ids] - px[:3]).max() <= TOL["fp32_mixed"]["particles"] * N
        assert np.abs(out[s][4:, ids] - pu).max() <= TOL["fp32_mixed"]["particles"] * np.abs(pu).max()
    # the split may be decided differently within rounding of a face, which keeps the total flux
    scale = np.abs(Jr).sum(axis=(1, 2, 3))
    assert np.all(np.abs(J.sum(axis=(1, 2, 3)) - Jr.sum(axis=(1, 2, 3))) <= TOL["fp32_mixed"]["J"] * scale)


def test_fp64_bits_on_both_sides_of_the_line():
    x, u, fields = _inputs(LINE + 9000)
    big = x.shape[1]
    ref, J = _push(x, u, fields, "fp64")
    jsum = np.zeros_like(J)
    for lo, hi in ((0, 1), (1, 32), (32, 65), (65, 4096 + 77), (4096 + 77, LINE // 2), (LINE // 2, big)):
        part, Jp = _push(x[:, lo:hi], [v[:, lo:hi] for v in u], fields, "fp64")
        for s in range(2):
            assert np.array_equal(part[s], ref[s][:, lo:hi])
        jsum += Jp
    # the parts' currents add up to the whole's (both sums of the same FP64 contributions)
    assert np.abs(jsum - J).max() <= 1e-12 * np.abs(J).max()
