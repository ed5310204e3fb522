"""What the server allocates to admit a run stays within the estimate that it charges, for one to four
species, with and without particles, in both precisions. The grids are large enough that a word a cell is more
than the estimate's slack."""
import ctypes

import pytest

from paper_0904_0232_gb300 import grpic as G

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
@pytest.mark.parametrize("ppc", [0, 1])
@pytest.mark.parametrize("nspecies", [1, 2, 3, 4])
def test_admission_within_the_estimate(nspecies, ppc, prec):
    size, peak, used = {}, [0], [0]

    @G.ALLOC_FN
    def alloc(nbytes, user):
        p = G._torch_alloc(nbytes, user)
        size[p] = nbytes
        used[0] += nbytes
        peak[0] = max(peak[0], used[0])
        return p

    @G.FREE_FN
    def free(ptr, user):
        if ptr:
            used[0] -= size.pop(ptr)
            G._torch_free(ptr, user)

    req = G.make_request(n=64, m=1.0, a=0.5, ppc=ppc, nsteps=0, seed=3, precision=prec, r_min=2.0,
                         species=((-1.0,), (1.0,), (0.5,), (-0.5,))[:nspecies])
    h = ctypes.c_void_p()
    assert G.load_library().grpic_server_create(1 << 33, 1, alloc, free, None, ctypes.byref(h)) == G.GRPIC_OK
    t = G.grpic_submit(h.value, req)
    G.grpic_server_tick(h.value)
    assert G.grpic_poll(h.value, t)[0] == G.GRPIC_RUN_DONE
    G.grpic_server_destroy(h.value)
    assert used[0] == 0
    assert 0 < peak[0] <= G.grpic_request_bytes(req)
