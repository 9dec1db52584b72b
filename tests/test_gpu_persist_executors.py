"""The two executors of the persistent step on the GPU: small grids step on one
thread-block cluster, larger ones (and those with a barrier timeout of their
own) on the grid-wide launch."""
import math

import numpy as np
import pytest

from paper_2412_16843_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu

GRID_NS = 3_000_000_000  # a barrier timeout other than the default selects the grid-wide launch


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2412_16843_gb300 import build
    build.build()
    cdi.load()


def rel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def on_executor(s, executor):
    s.set_exec(cdi.EXEC_PERSISTENT)
    if executor == "grid":
        s.set_barrier_timeout(GRID_NS)
    return s


def test_cluster_launch_opens_with_a_reduction():
    """gamma = 2.5 |u|_max: the first operation between the CTAs of a step is
    the largest velocity, not a barrier.  50 launches of one step on the
    cluster end where those of the grid-wide launch end: twice the bars that
    the FP64 parity tests set for 50 steps of either against the oracle."""
    nx, ny = 64, 32
    h = 1.0 / nx
    phi = inputs.add_noise(inputs.cap_phi_2d(nx, ny, h, 0.2, math.pi / 2, 0.5, h), 1e-3, 9)
    out = []
    for executor in ("cluster", "grid"):
        s = cdi.Solver(2, (nx, ny), (1.0, ny * h))
        s.set_fluids(1.0, 0.1, 0.05, 0.005, 1.0, h, -0.5)
        s.set_wall(cdi.WALL_BOTH, math.radians(120), h, 0.0)
        s.set_solver(1e-12, 100)
        s.set_state(phi)
        on_executor(s, executor)
        for _ in range(50):
            s.step(5e-5, 1)
        out.append(s.get_fields())
    assert rel(out[0][0], out[1][0]) < 2e-11
    for a in range(2):
        assert rel(out[0][1][a], out[1][1][a]) < 2e-10
