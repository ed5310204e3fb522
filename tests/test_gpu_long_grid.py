"""Steps of a grid with very many planes are enqueued as fast as others: the choice of the field launches'
chunks does not grow with the number of planes (4 ms a launch at a million planes where each number of chunks
is tried, 5 us where each length up to 64 is; bound: 2.5 ms a launch)."""
import time

import pytest

from paper_0904_0232_gb300.grpic import Simulation

pytestmark = pytest.mark.gpu


def test_host_time_of_a_step():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sim = Simulation(8, 8, 1000000, 1.0, 0.5, 1.0, 0.4, precision="fp32_mixed")
    sim.set_uniform_field(B=(0.0, 0.0, 0.1))
    sim.step(1)
    t = time.perf_counter()
    sim.step_async(5)  # four field launches a step
    host = time.perf_counter() - t
    sim.sync()
    assert host < 0.05, host
