"""GPU test of contexts and batches of different size stepped in turn in one
process: the dynamic shared memory a kernel may be launched with belongs to the
kernel, not to the object that set it last."""
import numpy as np
import pytest

from paper_2412_16843_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2412_16843_gb300 import build
    build.build()
    cdi.load()


def equal(a, b, dim):
    assert np.array_equal(a[0], b[0])
    for k in range(dim):
        assert np.array_equal(a[1][k], b[1][k])


@pytest.mark.parametrize("exec_mode", [cdi.EXEC_PERSISTENT, cdi.EXEC_KERNELS], ids=["persistent", "kernels"])
@pytest.mark.parametrize("precision", [cdi.FP64, cdi.FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("dim,big,small", [(2, (64, 64), (32, 16)), (2, (256, 128), (64, 32)), (3, 32, 16)])
def test_large_small_large_context(dim, big, small, precision, exec_mode):
    """The fields of the larger context do not change by a smaller one stepped
    in between."""
    make = (lambda n: inputs.drop_2d(*n)) if dim == 2 else (lambda n: inputs.drop_3d(n, noise=0.0))
    wl, ws = make(big), make(small)
    dt = inputs.stable_dt(wl)
    res = []
    for disturb in (False, True):
        s = cdi.from_workload(wl, precision=precision)
        s.set_exec(exec_mode)
        s.step(dt, 1)
        if disturb:
            t = cdi.from_workload(ws, precision=precision)
            t.set_exec(exec_mode)
            t.step(inputs.stable_dt(ws), 1)
        s.step(dt, 1)
        res.append(s.get_fields())
    equal(res[0], res[1], dim)


@pytest.mark.parametrize("count", [2, 160])
def test_two_batches_with_other_tail_budgets(count):
    """A batch with a small tail budget stepped between two steps of one with a
    large budget: on clusters (2 instances) and one CTA an instance (160)."""
    wls = [inputs.drop_2d(64, 32, 50.0 + i % 7 * 10.0) for i in range(count)]
    dts = np.array([w.dt for w in wls])
    res = []
    for disturb in (False, True):
        ss = [cdi.from_workload(w, precision=cdi.FP32_MIXED) for w in wls]
        b = cdi.Batch(ss)
        b.set_tail_budget(100 * 1024)
        b.step(dts, 1)
        if disturb:
            t = cdi.Batch([cdi.from_workload(w, precision=cdi.FP32_MIXED) for w in wls])
            t.set_tail_budget(16 * 1024)
            t.step(dts, 1)
        b.step(dts, 1)
        res.append(ss[0].get_fields())
    equal(res[0], res[1], 2)
