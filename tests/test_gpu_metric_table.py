"""The metric table of an FP64 context makes room for any other allocation of the library from the same
allocator: another context's, a batch's own tables, its own after it has been in a batch; also while another
thread steps the context. The field takes the same bits with and without it."""
import ctypes
import threading

import numpy as np
import pytest

from paper_0904_0232_gb300 import grpic as G
from paper_0904_0232_gb300 import synth

pytestmark = pytest.mark.gpu
N = 32
TABLE = 12 * 16 * N ** 3


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


class Memory:
    """An allocator with a budget."""

    def __init__(self):
        self.budget, self.used, self.size, lock = 1 << 40, 0, {}, threading.Lock()

        @G.ALLOC_FN
        def alloc(nbytes, user):
            with lock:
                if self.used + nbytes > self.budget:
                    return 0
                self.used += nbytes
            p = G._torch_alloc(nbytes, user)
            self.size[p] = nbytes
            return p

        @G.FREE_FN
        def free(ptr, user):
            if ptr:
                with lock:
                    self.used -= self.size.pop(ptr)
                G._torch_free(ptr, user)

        self.alloc, self.free = alloc, free

    def holds_table(self):
        return TABLE in self.size.values()

    def context(self):
        cfg = G.grpic_config(N, N, N, 1.2, 0.9, 1.0, 0.4, G.GRPIC_FP64, 2, 0.0, 0, 1, 0, 0.0, 0.3, 0.2, 4)
        cfg.alloc, cfg.free_fn = self.alloc, self.free
        return G.grpic_create(cfg, ctypes.c_void_p(0))


def _started(mem):
    ctx = mem.context()
    G.grpic_set_fields(ctx, *synth.random_fields((N, N, N), 3))
    return ctx


@pytest.fixture(scope="module")
def expected():
    mem = Memory()  # (its callbacks have to outlive the context)
    ctx = _started(mem)
    out = {}
    for n in range(1, 41):
        G.grpic_step(ctx, 1)
        out[n] = G.grpic_get_fields(ctx, (N, N, N))[:2]
    G.grpic_destroy(ctx)
    return out


def _same(ctx, want):
    got = G.grpic_get_fields(ctx, (N, N, N))[:2]
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_another_context_takes_its_room(expected):
    mem = Memory()
    a = _started(mem)
    assert mem.holds_table()
    G.grpic_step(a, 1)
    mem.budget = 2 * mem.used - TABLE - (1 << 20)
    b = _started(mem)
    assert not mem.holds_table()
    mem.budget = 1 << 40
    G.grpic_step(a, 2)
    G.grpic_step(b, 3)
    _same(a, expected[3])
    _same(b, expected[3])
    G.grpic_destroy(a)
    G.grpic_destroy(b)
    assert mem.used == 0


@pytest.mark.parametrize("destroyed", [True, False])
def test_given_up_after_and_between_batched_steps(expected, destroyed):
    mem = Memory()
    a = _started(mem)
    batch = G.grpic_batch_create([a])
    G.grpic_batch_step(batch, 1)
    assert mem.holds_table()
    if destroyed:
        G.grpic_batch_destroy(batch)
    mem.budget = mem.used
    n = 1000
    x = np.full((4, n), 0.5 * N)
    x[0] = np.linspace(2.0, 4.0, n)
    u = np.zeros((4, n))
    u[3] = 1.0
    G.grpic_load_particles(a, 0, 0.0, 0.0, x, u, np.arange(n, dtype=np.uint32))
    assert not mem.holds_table()
    mem.budget = 1 << 40
    if destroyed:
        G.grpic_step(a, 2)
        _same(a, expected[3])
    else:
        with pytest.raises(G.GrpicError):  # the batch was built without the species
            G.grpic_batch_step(batch, 1)
        G.grpic_batch_destroy(batch)
        batch = G.grpic_batch_create([a])
        G.grpic_batch_step(batch, 2)
        _same(a, expected[3])
        G.grpic_batch_destroy(batch)
    G.grpic_destroy(a)


def test_a_batch_goes_on_without_it(expected):
    mem = Memory()
    a = _started(mem)
    batch = G.grpic_batch_create([a])
    G.grpic_batch_step(batch, 1)
    mem.budget = 2 * mem.used - TABLE - (1 << 20)
    b = _started(mem)
    assert not mem.holds_table()
    mem.budget = 1 << 40
    G.grpic_batch_step(batch, 2)
    _same(a, expected[3])
    G.grpic_batch_destroy(batch)
    G.grpic_destroy(a)
    G.grpic_destroy(b)


def test_given_up_while_another_thread_steps(expected):
    mem = Memory()
    a = _started(mem)

    def steps():
        for _ in range(40):
            G.grpic_step_async(a, 1)

    t = threading.Thread(target=steps)
    t.start()
    mem.budget = 2 * mem.used - TABLE - (1 << 20)
    b = mem.context()
    t.join()
    assert not mem.holds_table()
    G.grpic_sync(a)
    _same(a, expected[40])
    G.grpic_destroy(a)
    G.grpic_destroy(b)
