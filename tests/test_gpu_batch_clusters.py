"""GPU test of the batched step's split of an instance over the CTAs of a
cluster: batches of 1, 10, 20, 60 and 160 equal small grids, which the launch
gives clusters of 16, 8, 4, 2 and 1 CTAs on a 152-SM part (fewer where fewer
are resident), against the same grids stepped alone."""
import numpy as np
import pytest

from paper_2412_16843_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2412_16843_gb300 import build
    build.build()
    cdi.load()


@pytest.mark.parametrize("count", [1, 10, 20, 60, 160])
@pytest.mark.parametrize("dim", [2, 3])
def test_cluster_split_ends_where_instances_alone_end(count, dim):
    """FP64 at a pressure tolerance of 1e-12: the sums over a grid are taken in
    another order, so fields agree to the solver tolerance times the bars of
    the batch tests (1e-11 in phi, 1e-9 in velocity)."""
    if dim == 2:
        wls = [inputs.drop_2d(64, 32, 50.0 + (i % 7) * 10.0) for i in range(count)]
    else:
        wls = [inputs.drop_3d(16, 50.0 + (i % 7) * 10.0, noise=0.0) for i in range(count)]
        for w in wls:
            w.dt = inputs.stable_dt(w)
    batched = [cdi.from_workload(w, tol=1e-12) for w in wls]
    b = cdi.Batch(batched)
    for _ in range(2):  # a second launch reuses the split
        b.step(np.array([w.dt for w in wls]), 2)
    for i in {0, count // 2, count - 1}:
        alone = cdi.from_workload(wls[i], tol=1e-12)
        alone.step(wls[i].dt, 4)
        pa, va, _ = alone.get_fields()
        pb, vb, _ = batched[i].get_fields()
        assert b.stats(i)["status"] == 0
        assert np.abs(pb - pa).max() < 1e-11
        for a in range(dim):
            assert np.abs(vb[a] - va[a]).max() <= 1e-9 * max(np.abs(v).max() for v in va)
