"""J of one push node by node against the oracle, near the hole (where the FP32-mixed code evaluates nodes inside the
lattice) and outside, for launches on both sides of the small-launch line, every quadrature order and the launch shapes:
the total over the grid, which the face weights cannot change, says nothing of them."""
import numpy as np
import pytest

import oracle as O
from parity_util import TOL, face_ambiguity_mask, rel_l2_masked
from paper_0904_0232_gb300.grpic import (GRPIC_STAGE_B_HALF, GRPIC_STAGE_PUSH_DEPOSIT, GRPIC_STAGE_ZERO_J,
                                         GRPIC_U_COV_SPATIAL, Simulation)
from test_gpu_push_paths import A, LINE, M, N, QMS, _inputs

pytestmark = pytest.mark.gpu
SHAPES = {"default": {}, "five_blocks": dict(far_min_blocks=5), "fits": dict(area_table=1, far_min_blocks=5),
          "fits_four": dict(area_table=1), "tile": dict(j_tile=1), "split": dict(split=1)}


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(scope="module")
def references():
    made = {}

    def get(count, quad):
        if (count, quad) not in made:
            x, u, fields = _inputs(count)
            k = x.shape[1]
            ref = O.Oracle(N, N, N, M, A, 1.0, 0.4, quad_order=quad, threads=0)
            ref.set_fields(*fields)
            for s, qm in enumerate(QMS):
                ref.load_particles(s, qm, qm * 1e-3, np.vstack([x, np.zeros((1, k))]),
                                   np.vstack([u[s], np.zeros((1, k))]), np.arange(k, dtype=np.uint32), umode=1)
            ref.b_half()
            ref.zero_j()
            ref.push_deposit()
            mask = face_ambiguity_mask(ref, (N, N, N), len(QMS))
            made[count, quad] = x, u, fields, ref.get_fields()[2], mask
        return made[count, quad]

    return get


@pytest.mark.parametrize("quad,shape", [(1, "default"), (3, "default")] + [(2, s) for s in SHAPES])
@pytest.mark.parametrize("count", [5000, LINE + 9000])
def test_nodes_against_the_oracle(references, count, quad, shape):
    x, u, fields, Jr, mask = references(count, quad)
    k = x.shape[1]
    assert mask.mean() < 0.25
    sim = Simulation(N, N, N, M, A, 1.0, 0.4, precision="fp32_mixed", quad_order=quad)
    sim.set_tuning(**SHAPES[shape])
    sim.set_fields(*fields)
    for s, qm in enumerate(QMS):
        sim.load_particles(s, qm, qm * 1e-3, np.vstack([x, np.zeros((1, k))]), u[s], np.arange(k, dtype=np.uint32),
                           GRPIC_U_COV_SPATIAL)
    for stage in (GRPIC_STAGE_B_HALF, GRPIC_STAGE_ZERO_J, GRPIC_STAGE_PUSH_DEPOSIT):
        sim.stage(stage)
    J = sim.get_fields()[2]
    r = np.arange(N) - 0.5 * (N - 1)
    R = np.sqrt(r[:, None, None] ** 2 + r[None, :, None] ** 2 + r[None, None, :] ** 2)
    # nodes below r_fp64 = 4 m among them, the other near ones, far
    for lo, hi in ((0.0, 7.0), (7.0, 12.0), (12.0, 60.0)):
        skip = mask | (R < lo) | (R >= hi)
        assert np.abs(Jr[:, ~skip]).max() > 0.0
        assert rel_l2_masked(J, Jr, skip) <= TOL["fp32_mixed"]["J"], (lo, rel_l2_masked(J, Jr, skip))
