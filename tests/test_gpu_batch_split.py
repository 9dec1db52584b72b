"""GPU test of the batched step at a known number of CTAs an instance, in the
forms the equal FP64 grids at 512 threads do not cover."""
import numpy as np
import pytest

from paper_2412_16843_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2412_16843_gb300 import build
    build.build()
    cdi.load()


def rel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def whole_chip():
    """The sizes below hold where 152 CTAs, or 76, 36, 15 and 7 clusters of 2
    to 16, are resident at once."""
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count == 152


@pytest.mark.parametrize("count,ctas", [(1, 16), (10, 8), (20, 4), (60, 2), (304, 1)])
@pytest.mark.parametrize("dim", [2, 3])
def test_equal_grids_run_on_the_expected_clusters(count, ctas, dim):
    if dim == 2:
        wls = [inputs.drop_2d(64, 32, 50.0 + (i % 7) * 10.0) for i in range(count)]
    else:
        wls = [inputs.drop_3d(16, 50.0 + (i % 7) * 10.0, noise=0.0) for i in range(count)]
    ss = [cdi.from_workload(w) for w in wls]
    b = cdi.Batch(ss)
    assert b.cluster() == 1
    b.step(np.array([inputs.stable_dt(w) for w in wls]), 1)
    if whole_chip():
        assert b.cluster() == ctas


@pytest.mark.parametrize("precision", [cdi.FP64, cdi.FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("threads", [256, 1024])
@pytest.mark.parametrize("count,ctas", [(3, 16), (64, 8)])
def test_uneven_grids_on_clusters_end_where_instances_alone_end(count, ctas, threads, precision):
    """The first 3 instances of the 2D sweep, and 64 (more than the 15 clusters
    of 8 that run at once): five steps at a pressure tolerance of 1e-10 end
    where each instance alone ends, within the bars of the batch tests."""
    wls = inputs.sweep_2d()[:count]
    batched = [cdi.from_workload(w, precision=precision, tol=1e-10) for w in wls]
    b = cdi.Batch(batched)
    b.set_threads(threads)
    b.step(np.array([w.dt for w in wls]), 5)
    if whole_chip():
        assert b.cluster() == ctas
    tol = 1e-11 if precision == cdi.FP64 else 1e-5
    sizes = [w.cells for w in wls]
    for i in sorted({0, int(np.argmin(sizes)), int(np.argmax(sizes))}):
        alone = cdi.from_workload(wls[i], precision=precision, tol=1e-10)
        alone.step(wls[i].dt, 5)
        pa, va, _ = alone.get_fields()
        pb, vb, _ = batched[i].get_fields()
        assert b.stats(i)["status"] == 0
        assert rel(pb, pa) < tol, wls[i].name
        for a in range(2):
            assert rel(vb[a], va[a]) < 100 * tol, (wls[i].name, a)


def test_sweep_of_512_runs_on_pairs():
    wls = inputs.sweep_2d()
    b = cdi.Batch([cdi.from_workload(w, precision=cdi.FP32_MIXED) for w in wls])
    b.set_threads(1024)
    b.step(np.array([w.dt for w in wls]), 1)
    assert all(b.stats(i)["status"] == 0 for i in range(len(wls)))
    if whole_chip():
        assert b.cluster() == 2
