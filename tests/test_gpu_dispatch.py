"""The routes a round can take (persistent or a kernel per phase, one phase or several, queued behind
another pass or continued after it) against the oracle, bit for bit: which route a list takes depends
on its length alone, so the lengths at which the route changes are moved to those of small meshes,
or the mesh is sized to lie on either side of them.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1505_04694_gb300 import inputs
from test_gpu_parity import STAT_KEYS, _wheel, assert_same_adjacency, assert_same_mesh, assert_same_raw

pytestmark = pytest.mark.gpu

pm = pytest.importorskip("paper_1505_04694_gb300.pm")

ALL = 1 << 30


@pytest.fixture
def tuned():
    yield lambda limits, fuse: pm.set_tuning({"rounds_limit": limits, "fuse_limit": fuse})
    pm.set_tuning(None)


@pytest.fixture(scope="module")
def adapted():
    """Oracle results of the mesh below, by selection mode (computed once)."""
    w = inputs.psi_workload(33, 20000, True, 2)
    res = {}
    for mode in (0, 1):
        o = O.OracleMesh(w.xy, w.tri).set_metric(w.m)
        res[mode] = (o.adapt(O.make_params(seed=2, select_mode=mode)), o.get_mesh())
    return w, res


# collapses hand back while flips do not and the other way round; every list a kernel per phase; lists
# that start so and end in persistent rounds (moves stored by the one are met by the other); flips
# and smoothing never and always in one phase
@pytest.mark.parametrize("limits,fuse", [([0, 0, 0], [ALL, ALL]), ([64, 64, 64], [ALL, ALL]),
                                         ([700, 700, 3000], [ALL, ALL]), ([ALL, 300, 300], [ALL, ALL]),
                                         ([300, ALL, 8000], [ALL, 500]), ([ALL, ALL, ALL], [0, 0]),
                                         ([ALL, ALL, 5000], [1000, 0])])
@pytest.mark.parametrize("mode", [0, 1])
def test_limits_change_the_route_and_nothing_else(adapted, tuned, limits, fuse, mode):
    w, res = adapted
    so, om = res[mode]
    tuned(limits, fuse)
    g = pm.Mesh.from_host(w.xy, w.tri, device=0)
    g.set_metric(w.m)
    sg = g.adapt(pm.Params(seed=2, select=mode))
    assert_same_mesh(g.get_mesh(), om, f"{limits} {fuse}")
    for k in STAT_KEYS:
        assert sg[k] == so[k], (k, sg[k], so[k])


# first lists of 9604 and 9801 entries: one pass of evaluations in two turns of the grid's tiles
# (4864), or one more and so several phases.  A flip's list holds every vertex, a smoothing's the interior ones.
@pytest.mark.parametrize("opname,n", [("swap", 69), ("swap", 70), ("swap", 98), ("swap", 99),
                                      ("smooth", 71), ("smooth", 72), ("smooth", 100), ("smooth", 101)])
def test_lists_on_either_side_of_the_one_phase_bound(opname, n):
    w = inputs.psi_workload(n, 2 * n * n, True, n)
    g = pm.Mesh.from_host(w.xy, w.tri, device=0)
    g.set_metric(w.m)
    o = O.OracleMesh(w.xy, w.tri).set_metric(w.m)
    sg = getattr(g, opname)(pm.Params(seed=n))
    so = getattr(o, opname)(O.make_params(seed=n))
    for k in STAT_KEYS:
        assert sg[k] == so[k], (k, sg[k], so[k])
    assert sg["flips"] + sg["moves"] > 0
    assert_same_raw(g.get_raw(), o.get_raw(), opname)


def _grid(n, h):
    xy, tri = inputs.grid_mesh(n)
    return xy, tri, inputs.uniform_metric(xy.shape[0], h)


def _star(nb, h):
    xy, tri = _wheel(nb)
    return xy, tri, inputs.uniform_metric(xy.shape[0], h)


# collapses with many candidates of equal length (a regular grid), 4 to 124 candidates at one vertex (more
# than a warp's lanes), rows of more than 16, 32 and 64 entries; with a kernel per phase and persistent
@pytest.mark.parametrize("mesh", [_grid(40, 0.3), _grid(9, 3.0), _star(4, 4.0), _star(28, 4.0),
                                  _star(36, 4.0), _star(84, 0.4), _star(124, 4.0), _star(124, 0.2)],
                         ids=["grid40", "grid9", "star4", "star28", "star36", "star84", "star124",
                              "star124fine"])
@pytest.mark.parametrize("limit", [0, ALL])
def test_collapses_with_many_candidates(tuned, mesh, limit):
    xy, tri, m = mesh
    tuned([limit] * 3, [ALL, ALL])
    g = pm.Mesh.from_host(xy, tri, device=0)
    g.set_metric(m)
    o = O.OracleMesh(xy, tri).set_metric(m)
    for opname in ("coarsen", "refine", "coarsen"):
        sg = getattr(g, opname)(pm.Params(seed=3))
        so = getattr(o, opname)(O.make_params(seed=3))
        for k in STAT_KEYS:
            assert sg[k] == so[k], (opname, k, sg[k], so[k])
        rg = g.get_raw()
        assert_same_raw(rg, o.get_raw(), opname)
        assert_same_adjacency(g, o, rg)


def test_many_small_meshes_whose_rows_overflow():
    """A set in which a few meshes outgrow the rows' first width in the middle of an iteration
    (the passes queued behind are taken up again after the rows are rebuilt)."""
    ms = [_star(16, 0.03), _grid(6, 0.05), _star(12, 0.02), _grid(12, 0.5)]
    b = pm.Batch.from_host([(xy, tri) for xy, tri, _ in ms])
    b.set_metric(np.concatenate([m for _, _, m in ms]))
    sb = b.adapt([pm.Params(seed=5)] * len(ms))
    for i, ((xy, tri, m), got) in enumerate(zip(ms, b.get_meshes())):
        o = O.OracleMesh(xy, tri).set_metric(m)
        so = o.adapt(O.make_params(seed=5))
        assert_same_mesh(got, o.get_mesh(), f"mesh {i}")
        for k in ("rounds", "collapses", "splits", "flips", "moves"):
            assert sb[i][k] == so[k], (i, k, sb[i][k], so[k])


# a colouring a kernel per phase throughout; begun so and ended in persistent rounds; persistent alone
@pytest.mark.parametrize("limit,steps", [(0, True), (100, True), (3000, True), (ALL, False)])
def test_colouring_takes_the_limits_route(adapted, tuned, limit, steps):
    w, res = adapted
    so, om = res[1]
    tuned([ALL, ALL, limit], [ALL, ALL])
    count = {}
    for kernel in ("k_colour_propose", "k_colour_rounds"):
        g = pm.Mesh.from_host(w.xy, w.tri, device=0)
        g.set_metric(w.m)
        pm.profile_enable(kernel)
        sg = g.adapt(pm.Params(seed=2, select=1))
        count[kernel] = pm.profile_read()[1]
        pm.profile_enable(None)
        assert_same_mesh(g.get_mesh(), om, f"{limit} {kernel}")
        for k in STAT_KEYS:
            assert sg[k] == so[k], (k, sg[k], so[k])
    assert (count["k_colour_propose"] > 0) == steps
    assert count["k_colour_rounds"] > 0  # (the first launch finds the list too long)


def _hub(nb, offset):
    """A disc: a vertex off its centre joined to a ring of nb interior vertices, which a second ring of
    nb boundary vertices surrounds; coordinates around (offset, offset)."""
    rng = np.random.default_rng(nb)
    t = 2 * np.pi * (np.arange(nb) + rng.uniform(-0.2, 0.2, nb)) / nb
    u = np.stack([np.cos(t), np.sin(t)], axis=1)
    s = 2 * np.pi * (np.arange(nb) + 0.5) / nb
    xy = np.concatenate([[[0.2, 0.15]], 0.6 * u * rng.uniform(0.95, 1.05, (nb, 1)),
                         np.stack([np.cos(s), np.sin(s)], axis=1)]) + offset
    i = np.arange(nb)
    j = (i + 1) % nb
    tri = np.concatenate([np.stack([0 * i, 1 + i, 1 + j], axis=1),
                          np.stack([1 + i, 1 + nb + i, 1 + j], axis=1),
                          np.stack([1 + j, 1 + nb + i, 1 + nb + j], axis=1)]).astype(np.int32)
    return xy, tri, inputs.uniform_metric(xy.shape[0], 2 * np.pi / nb)


# balls of 24 to 124 elements moved in the rounds with a kernel per phase, where one of more than 32
# takes a warp by itself, and in the persistent ones.  At offset 0 the bounds accept the moves and their
# qualities follow; at 2^36 a coordinate's error leaves every quality to the exact pass.
@pytest.mark.parametrize("limit", [0, ALL])
@pytest.mark.parametrize("offset", [0.0, 2.0 ** 36])
@pytest.mark.parametrize("nb", [24, 32, 33, 36, 64, 65, 84, 124])
def test_moves_of_large_balls(tuned, nb, offset, limit):
    xy, tri, m = _hub(nb, offset)
    tuned([limit] * 3, [ALL, ALL])
    for opname in ("smooth", "adapt"):
        g = pm.Mesh.from_host(xy, tri, device=0)
        g.set_metric(m)
        o = O.OracleMesh(xy, tri).set_metric(m)
        sg = getattr(g, opname)(pm.Params(seed=4))
        so = getattr(o, opname)(O.make_params(seed=4))
        for k in STAT_KEYS:
            assert sg[k] == so[k], (opname, k, sg[k], so[k])
        rg = g.get_raw()
        assert_same_raw(rg, o.get_raw(), opname)
        assert_same_adjacency(g, o, rg)
        if opname == "smooth":
            assert sg["moves"] > 0 and not np.array_equal(o.get_mesh()[0][0], xy[0])
