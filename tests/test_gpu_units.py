"""The unit of length changes neither the result nor the work: a mesh in units 2^e larger, under the
metric that goes with it, takes the same operations with every coordinate scaled exactly.
"""
import numpy as np
import pytest

from mempool import MemPool
from paper_1505_04694_gb300 import inputs
from test_gpu_parity import STAT_KEYS

pytestmark = pytest.mark.gpu

pm = pytest.importorskip("paper_1505_04694_gb300.pm")


def adapt(w, e, kernel=None):
    """Adapts `w` in units of 2^-e: statistics, mesh, launches, counted FP64 operations of `kernel`."""
    g = pm.Mesh.from_host(np.ldexp(w.xy, e), w.tri, device=0)
    g.set_metric(np.ldexp(w.m, -2 * e))
    pm.profile_enable(kernel)
    n0 = pm.kernel_launches()
    st = g.adapt(pm.Params(seed=3, opt_smooth_rounds=2))
    n = pm.kernel_launches() - n0
    work = pm.profile_read()[2] if kernel else 0
    pm.profile_enable(None)
    mesh = g.get_mesh()
    g.close()
    return st, mesh, n, work


@pytest.fixture(scope="module")
def workload():
    return inputs.psi_workload(33, 20000, True, 3)


@pytest.mark.parametrize("kernel", ["k_swap_rounds", "k_smooth_rounds"])
@pytest.mark.parametrize("e", [-32, 32])
def test_unit_changes_neither_result_nor_fp64_work(workload, e, kernel):
    s0, (xy0, tri0, m0), _, f0 = adapt(workload, 0, kernel)
    s1, (xy1, tri1, m1), _, f1 = adapt(workload, e, kernel)
    for k in STAT_KEYS:
        assert s1[k] == s0[k], (k, s1[k], s0[k])
    assert np.array_equal(tri1, tri0)
    assert np.array_equal(np.ldexp(xy1, -e), xy0) and np.array_equal(np.ldexp(m1, 2 * e), m0)
    # the filters' absolute terms alone know the unit: the exact rest is the same to within 1%
    assert f0 > 0 and abs(f1 - f0) <= 0.01 * f0


@pytest.mark.parametrize("e", [-32, 32])
def test_unit_does_not_change_the_storage_estimate(workload, e):
    """One growth of the storage at the start, whatever the unit (each later one is more launches)."""
    assert adapt(workload, e)[2] == adapt(workload, 0)[2]


@pytest.mark.parametrize("aspect", [100.0, 1e3, 1e5])
def test_estimate_of_anisotropic_metrics(aspect):
    """A constant metric at 45 degrees asks for as many elements as an isotropic one of the same
    determinant, so it gets as much storage (an adaptation without iterations only makes room)."""
    xy, tri = inputs.grid_mesh(33)
    n = xy.shape[0]
    d = 5.0e4  # sqrt(det): 115k elements on the unit square
    a, b = d * aspect, d / aspect
    iso = np.tile([d, 0.0, d], (n, 1))
    rot = np.tile([0.5 * (a + b), 0.5 * (a - b), 0.5 * (a + b)], (n, 1))
    grown = []
    for m in (iso, rot):
        with MemPool() as pool:
            g = pm.Mesh.from_host(xy, tri, device=0)
            g.set_metric(m)
            g.adapt(pm.Params(seed=1, max_iter=0, max_smooth_sweeps=0))
            grown.append(pool.high())
            g.close()
    # within the estimate's 5%, and a sixteenth that a block's size may be rounded up by
    assert grown[0] / 1.15 < grown[1] < grown[0] * 1.15
