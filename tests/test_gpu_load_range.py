"""Velocities at the edge of FP64.  Where the square is beyond it the completed u^4 is infinite, which the load takes (the
first step reports it) except for covariant u_i where the metric is flat, whose completion is not a number; a u^4 of 0 makes
the step infinite."""
import numpy as np
import pytest

from paper_0904_0232_gb300.grpic import (GRPIC_U_CONTRA_SPATIAL, GRPIC_U_COV_SPATIAL, GrpicError, Simulation)

pytestmark = pytest.mark.gpu
N = 24


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
@pytest.mark.parametrize("m,umode,taken", [(1.0, GRPIC_U_COV_SPATIAL, True), (1.0, GRPIC_U_CONTRA_SPATIAL, True),
                                           (0.0, GRPIC_U_CONTRA_SPATIAL, True), (0.0, GRPIC_U_COV_SPATIAL, False)])
def test_u_beyond_the_range_of_its_square(prec, m, umode, taken):
    sim = Simulation(N, N, N, m, 0.5 * m, 1.0, 0.4, precision=prec)
    n = 3
    x = np.full((4, n), 4.25)
    x[3] = 0.0
    u = np.zeros((3, n))
    u[0] = 0.25
    u[:, 1] = (1e160, -3e170, 2e180)
    ids = np.arange(n, dtype=np.uint32)
    if not taken:
        with pytest.raises(GrpicError) as err:
            sim.load_particles(0, 1.0, 1e-3, x, u, ids, umode)
        assert err.value.code == 1  # GRPIC_ERR_INVALID
        return
    sim.load_particles(0, 1.0, 1e-3, x, u, ids, umode)
    xo, uo, io = sim.get_particles(0)
    assert np.array_equal(np.sort(io), ids)
    uo = uo[:, np.argsort(io)]
    assert uo[3, 1] == np.inf and np.all(np.isfinite(uo[:, [0, 2]]))


@pytest.mark.parametrize("umode", [GRPIC_U_COV_SPATIAL, GRPIC_U_CONTRA_SPATIAL])
def test_large_velocities_are_completed(umode):
    """|u|^2 of 1e300: g_mn u^m u^n = -c^2 is |u| to FP64 rounding, at rest in flat space far from a light hole."""
    sim = Simulation(N, N, N, 0.0, 0.0, 1.0, 0.4)
    x = np.full((4, 2), 4.25)
    u = np.array([[1e150, 3.0], [0.0, 0.0], [-2e149, 4.0]])
    sim.load_particles(0, 1.0, 1e-3, x, u, np.arange(2, dtype=np.uint32), umode)
    _, uo, io = sim.get_particles(0)
    want = np.hypot(np.hypot(u[0], u[2]), 1.0)
    assert np.all(np.abs(uo[3, np.argsort(io)] - want) <= 4e-16 * want)


@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
def test_a_step_without_a_clock_rate_is_reported_as_such(prec):
    """u^4 = 0, given in full: the proper-time step dt / gamma is infinite and the state after it not finite."""
    sim = Simulation(N, N, N, 0.0, 0.0, 1.0, 0.4, precision=prec)
    x = np.full((4, 1), 5.25)
    x[3] = 0.0
    sim.load_particles(0, 0.0, 0.0, x, np.array([[0.1], [0.0], [0.0], [0.0]]), np.zeros(1, dtype=np.uint32))
    with pytest.raises(GrpicError) as err:
        sim.step(1)
    assert err.value.code == 5  # GRPIC_ERR_NONFINITE
