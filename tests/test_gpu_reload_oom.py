"""A load that has to grow a species' stores and does not get the memory (for the first store, the second or a staging
copy) leaves the species empty: steps, read-back and diagnostics go on without it, and a later load that fits is as good
as a first one."""
import ctypes

import numpy as np
import pytest

from paper_0904_0232_gb300 import grpic as G

pytestmark = pytest.mark.gpu
N = 16


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _particles(n, seed):
    rng = np.random.default_rng(seed)
    x = np.vstack([rng.uniform(3.0, N - 4.0, (3, n)), np.zeros((1, n))])
    u = rng.normal(0.0, 0.1, (3, n))
    return x, np.vstack([u, np.sqrt(1.0 + (u ** 2).sum(0))]), np.arange(n, dtype=np.uint32)


@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
@pytest.mark.parametrize("granted", [0, 1, 2])
def test_load_without_the_memory_to_grow(prec, granted):
    left = [1 << 30]

    @G.ALLOC_FN
    def alloc(nbytes, user):
        left[0] -= 1
        return G._torch_alloc(nbytes, user) if left[0] >= 0 else 0

    cfg = G.grpic_config(N, N, N, 0.0, 0.0, 1.0, 0.4, {"fp64": G.GRPIC_FP64, "fp32_mixed": G.GRPIC_FP32_MIXED}[prec],
                         2, 0.0, 0, 1, 0, 0.0, 0.0, 0.0, 0, 0, 0)
    cfg.alloc, cfg.free_fn = alloc, G._torch_free
    ctx = G.grpic_create(cfg, ctypes.c_void_p(0))
    try:
        G.grpic_load_particles(ctx, 0, 1.0, 1e-3, *_particles(100, 1))
        G.grpic_load_particles(ctx, 1, -1.0, -1e-3, *_particles(50, 2))
        left[0] = granted
        with pytest.raises(G.GrpicError) as err:
            G.grpic_load_particles(ctx, 0, 1.0, 1e-3, *_particles(5000, 3))
        assert err.value.code == 2  # GRPIC_ERR_OOM
        left[0] = 1 << 30
        assert G.grpic_num_particles(ctx, 0) == 0
        G.grpic_step(ctx, 2)
        assert G.grpic_num_particles(ctx, 1) == 50
        assert G.grpic_get_stats(ctx)["particle_steps"] == 100
        G.grpic_charge_density(ctx, (N, N, N), False)
        for n, seed in ((60, 4), (5000, 5)):
            x, u, ids = _particles(n, seed)
            G.grpic_load_particles(ctx, 0, 1.0, 1e-3, x, u, ids)
            xo, uo, io = G.grpic_get_particles(ctx, 0)
            o = np.argsort(io)
            assert np.array_equal(io[o], ids)
            keep = x[:3].astype(np.float32) if prec == "fp32_mixed" else x[:3]
            assert np.array_equal(xo[:3, o], keep)
            G.grpic_step(ctx, 1)
            assert G.grpic_num_particles(ctx, 0) == n
    finally:
        G.grpic_destroy(ctx)
