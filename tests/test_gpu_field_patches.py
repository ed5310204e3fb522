"""Field updates where the patches of the field kernels begin and end (31 cells by 15 or 7, chunks of z), the outer layers
copied beside them, the FP64 metric table against the evaluation in the kernels, and the E step between two B
half-steps, whose predictor must leave b^{n-1/2} alone.  Tolerances: those of the stages in test_gpu_parity.py."""
import ctypes

import numpy as np
import pytest

import oracle as O
from parity_util import TOL, rel_l2
from paper_0904_0232_gb300 import grpic as G
from paper_0904_0232_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _pair(dims, prec, seed, **layers):
    nx, ny, nz = dims
    m, a = 0.6, 0.5
    d, b = (v.astype(np.float32).astype(np.float64) for v in synth.random_fields((nz, ny, nx), seed))
    ref = O.Oracle(nx, ny, nz, m, a, 1.0, 0.4, threads=0, **layers)
    ref.set_fields(d, b)
    if layers:
        ref.set_absorb_target(d, b)
    sim = G.Simulation(nx, ny, nz, m, a, 1.0, 0.4, precision=prec, **layers)
    sim.set_fields(d, b)
    return ref, sim, d, b


@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
@pytest.mark.parametrize("layers", [{}, dict(absorb_inner=0.3, absorb_outer=0.2, absorb_width=3)], ids=["held", "layers"])
@pytest.mark.parametrize("dims", [(8, 9, 10), (35, 19, 9), (36, 20, 12), (34, 18, 70), (67, 33, 8), (9, 35, 13)])
def test_steps_at_patch_edges(dims, layers, prec):
    ref, sim, d, b = _pair(dims, prec, sum(dims), **layers)
    ref.step(2)
    sim.step(2)
    d1, b1, _ = sim.get_fields()
    dr, br, _ = ref.get_fields()
    assert rel_l2(d1, dr) <= 2 * TOL[prec]["fields"] and rel_l2(b1, br) <= 2 * TOL[prec]["fields"]
    outer = np.ones(d.shape, bool)
    outer[:, 2:-2, 2:-2, 2:-2] = False
    assert np.array_equal(d1[outer], d[outer]) and np.array_equal(b1[outer], b[outer])


@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
def test_e_step_between_the_b_halves(prec):
    ref, sim, d, b = _pair((21, 24, 27), prec, 5)
    for stage, call in ((G.GRPIC_STAGE_B_HALF, ref.b_half), (G.GRPIC_STAGE_E, ref.e_step),
                        (G.GRPIC_STAGE_B_HALF2, ref.b_half2)):
        sim.stage(stage)
        call()
    d1, b1, _ = sim.get_fields()
    dr, br, _ = ref.get_fields()
    assert rel_l2(d1, dr) <= 2 * TOL[prec]["fields"] and rel_l2(b1, br) <= 2 * TOL[prec]["fields"]


def test_metric_table_given_up():
    """An FP64 context whose allocator refuses the table steps to the same bits without it."""
    n = 24
    table = 12 * 16 * n ** 3
    refused = []

    @G.ALLOC_FN
    def alloc(nbytes, user):
        if nbytes == table:
            refused.append(nbytes)
            return None
        return G._torch_alloc(nbytes, user)

    d, b = synth.random_fields((n, n, n), 3)
    out = []
    for fn in (G._torch_alloc, alloc):
        cfg = G.grpic_config(n, n, n, 1.0, 0.9, 1.0, 0.4, G.GRPIC_FP64, 2, 0.0, 0, 1, 0, 0.0, 0.3, 0.2, 4)
        cfg.alloc, cfg.free_fn = fn, G._torch_free
        ctx = G.grpic_create(cfg, ctypes.c_void_p(0))
        G.grpic_set_fields(ctx, d, b)
        G.grpic_step(ctx, 3)
        out.append(G.grpic_get_fields(ctx, (n, n, n))[:2])
        G.grpic_destroy(ctx)
    assert refused == [table]
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
