"""The two executors of the persistent step on the GPU: small grids step on one
thread-block cluster, larger ones (and those with a barrier timeout of their
own) on the grid-wide launch."""
import math

import numpy as np
import pytest

import oracle
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


EXECUTORS = pytest.mark.parametrize("executor", ["cluster", "grid"])


def against_oracle(s, o, phi_bar, u_bar):
    phi_g, vel_g, _ = s.get_fields()
    phi_o, vel_o, _ = o.get_state()
    assert rel(phi_g, phi_o) < phi_bar
    for a in range(len(vel_o)):
        assert rel(vel_g[a], vel_o[a]) < u_bar


@EXECUTORS
@pytest.mark.parametrize("grid", [(64, 32), (32, 16), (16, 16, 12)], ids=str)
def test_fp64_step_parity(executor, grid):
    """20 steps of a drop against the FP64 oracle, with the bars of the 50-step
    parity tests (32 x 16: fewer cells than the grid-wide launch has warps)."""
    if len(grid) == 2:
        wl = inputs.drop_2d(*grid)
    else:
        h = 1.0 / 16
        L = tuple(n * h for n in grid)
        phi = inputs.add_noise(inputs.cap_phi_3d(*grid, h, 0.3, math.pi / 2, 0.5, 0.5, h), 1e-3, 3)
    if len(grid) == 2:
        s, o = cdi.from_workload(wl, tol=1e-12), oracle.from_workload(wl, tol=1e-12)
        dt = wl.dt
    else:
        s, o = cdi.Solver(3, grid, L), oracle.Oracle(3, grid, L)
        for x in (s, o):
            x.set_fluids(1.0, 0.1, 0.05, 0.005, 1.0, h, 1.0)
            x.set_solver(1e-12, 100)
        s.set_wall(cdi.WALL_BOTH, math.radians(60), h, 0.0)
        o.set_wall_slip_length(2, math.radians(60), h, 0.0)
        s.set_state(phi)
        o.set_state(phi)
        dt = 5e-5
    on_executor(s, executor)
    s.step(dt, 20)
    o.step(dt, 20)
    against_oracle(s, o, 1e-11, 1e-10)


@EXECUTORS
def test_adaptive_gamma_parity(executor):
    """gamma = 2.5 |u|_max (the maximum over the grid is a reduction) for 50
    steps against the oracle."""
    nx, ny = 64, 32
    h = 1.0 / nx
    phi = inputs.add_noise(inputs.cap_phi_2d(nx, ny, h, 0.2, math.pi / 2, 0.5, h), 1e-3, 9)
    s, o = cdi.Solver(2, (nx, ny), (1.0, ny * h)), oracle.Oracle(2, (nx, ny), (1.0, ny * h))
    for x in (s, o):
        x.set_fluids(1.0, 0.1, 0.05, 0.005, 1.0, h, -0.5)
        x.set_solver(1e-12, 100)
    s.set_wall(cdi.WALL_BOTH, math.radians(120), h, 0.0)
    o.set_wall_slip_length(2, math.radians(120), h)
    s.set_state(phi)
    o.set_state(phi)
    on_executor(s, executor)
    s.step(5e-5, 50)
    o.step(5e-5, 50)
    against_oracle(s, o, 1e-11, 1e-10)


@EXECUTORS
def test_extrapolated_first_guess_parity(executor):
    wl = inputs.couette_2d(128, 32, 1.0)
    s, o = cdi.from_workload(wl, tol=1e-12), oracle.from_workload(wl, tol=1e-12)
    s.set_solver(1e-12, 100, cdi.WARM_EXTRAP)
    s.set_state(wl.phi0)
    on_executor(s, executor)
    s.step(wl.dt, 40)
    o.step(wl.dt, 40)
    against_oracle(s, o, 1e-11, 1e-10)


@EXECUTORS
def test_fp32_mixed_parity(executor):
    """200 FP32-mixed steps of the 64 x 32 drop against the FP64 oracle, with
    the bars of that form (2e-5 in phi, 1e-3 relative in velocity)."""
    wl = inputs.drop_2d(64, 32)
    s = cdi.from_workload(wl, precision=cdi.FP32_MIXED, tol=1e-8)
    o = oracle.from_workload(wl, tol=1e-8)
    on_executor(s, executor)
    s.step(wl.dt, 200)
    o.step(wl.dt, 200)
    phi_g, vel_g, _ = s.get_fields()
    phi_o, vel_o, _ = o.get_state()
    assert np.abs(phi_g - phi_o).max() < 2e-5
    for a in range(2):
        assert rel(vel_g[a], vel_o[a]) < 1e-3


@EXECUTORS
@pytest.mark.parametrize("precision", [cdi.FP64, cdi.FP32_MIXED], ids=["fp64", "fp32"])
def test_no_convergence_is_reported(executor, precision):
    wl = inputs.drop_2d(64, 32)
    s = on_executor(cdi.from_workload(wl, precision=precision, tol=1e-14, max_vcycles=1), executor)
    with pytest.raises(cdi.CdiError) as e:
        s.step(wl.dt, 1)
    assert e.value.status == 4
    assert s.last_stats()["resid"] > 1e-14


def test_grid_barriers_work_after_a_timeout():
    """A zero timeout ends the call with CDI_ETIMEOUT; with a timeout set again
    (not the default, which would select the cluster) the grid-wide launch
    steps the same context."""
    wl = inputs.drop_2d(64, 32)
    s, o = cdi.from_workload(wl, tol=1e-12), oracle.from_workload(wl, tol=1e-12)
    s.set_exec(cdi.EXEC_PERSISTENT)
    s.set_barrier_timeout(0)
    with pytest.raises(cdi.CdiError) as e:
        s.step(wl.dt, 1)
    assert e.value.status == 6
    s.set_barrier_timeout(GRID_NS)
    s.set_state(wl.phi0)
    s.step(wl.dt, 2)
    o.step(wl.dt, 2)
    against_oracle(s, o, 1e-11, 1e-10)


def test_grid_above_the_cluster_sizes_fp64():
    """256 x 64 cells take the grid-wide launch by themselves."""
    wl = inputs.couette_2d(256, 64, 1.0)
    s, o = cdi.from_workload(wl, tol=1e-12), oracle.from_workload(wl, tol=1e-12)
    s.set_exec(cdi.EXEC_PERSISTENT)
    s.step(wl.dt, 4)
    o.step(wl.dt, 4)
    against_oracle(s, o, 1e-11, 1e-10)
