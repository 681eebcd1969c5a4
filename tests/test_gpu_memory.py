"""Storage where device memory is short: what fits without an optional extra is not refused."""
import numpy as np
import pytest

from mempool import MemPool
from paper_1505_04694_gb300 import inputs

pytestmark = pytest.mark.gpu

pm = pytest.importorskip("paper_1505_04694_gb300.pm")


def make_room(limit=0):
    """A mesh given room for 6M elements (over 2^23 vertex slots); the most bytes in use."""
    xy, tri = inputs.grid_mesh(65)
    d = 6.0e6 * np.sqrt(3.0) / 4.0  # sqrt(det): 6M unit triangles on the unit square
    with MemPool(limit) as pool:
        with pm.Mesh.from_host(xy, tri, device=0) as g:
            g.set_metric(np.tile([d, 0.0, d], (xy.shape[0], 1)))
            g.adapt(pm.Params(seed=1, max_iter=0, max_smooth_sweeps=0))
            out = g.get_mesh()
        high = pool.high()
    return high, out


def test_wide_rows_are_given_up_when_memory_is_short():
    """From 2^23 vertex slots on rows are made 32 entries wide, 320 bytes a slot more than needed: with
    half of that missing the rows stay as they are."""
    high, (xy, tri, _) = make_room()
    _, (xy1, tri1, _) = make_room(high - 160 * 2 ** 23)
    assert np.array_equal(xy1, xy) and np.array_equal(tri1, tri)


def adapt_tiny(n):
    """n meshes of 8 triangles, each refined to about a hundred; the most bytes in use."""
    xy, tri = inputs.grid_mesh(3)
    with MemPool() as pool:
        b = pm.Batch.from_host([(xy, tri)] * n)
        b.set_metric(np.tile(inputs.uniform_metric(xy.shape[0], 0.2), (n, 1)))
        st = b.adapt([pm.Params(seed=1)] * n)
        assert min(s["splits"] for s in st) > 10
        b.close()
        return pool.high()


def test_very_many_tiny_meshes_take_little_more_than_they_need():
    """The spare room of a growth does not rise with the number of meshes beyond 512: what eight times as
    many hold above that are their own few hundred slots each (a twelfth of the spare ones)."""
    assert adapt_tiny(4096) < 2 * adapt_tiny(512)


def test_calls_work_after_one_that_ran_out_of_memory():
    """A refused allocation is that call's error alone."""
    xy, tri = inputs.grid_mesh(65)
    with MemPool(1 << 28):
        with pm.Mesh.from_host(xy, tri, device=0) as g:
            d = 6.0e6
            g.set_metric(np.tile([d, 0.0, d], (xy.shape[0], 1)))
            with pytest.raises(pm.PmError, match="PM_ERR_OOM"):
                g.adapt(pm.Params(seed=1, max_iter=0))
            out = g.get_mesh()
            assert np.array_equal(out[0], xy) and np.array_equal(out[1], tri)
            with pm.Mesh.from_host(xy, tri, device=0) as h:
                h.set_metric(inputs.uniform_metric(xy.shape[0], 0.02))
                assert h.adapt(pm.Params(seed=1))["converged"] == 1
