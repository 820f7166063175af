"""The build's splits at the edges of their paths (needs a GB300): numbers of
bins that put three, two or one axis on a warp, the smallest and largest
leaves (nodes of 2 .. 32 records finished by one warp), duplicate Morton keys,
centroids without extent (no usable plane), and nodes of more than 1024
records outside the big-node pools (a scene of more than 4M triangles), each
split the Eq. 2 minimum over the device's candidates by the float64 checker."""
import numpy as np
import pytest

from paper_2208_10008_gb300 import scenes
import eq2_check as E

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rb():
    from paper_2208_10008_gb300 import rtbvh
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    rtbvh.lib()
    return rtbvh


def _build(rb, tris, src, **kw):
    s = rb.rt_scene_upload(tris)
    rb.rt_bvh_build(s, source=src, **kw)
    info = rb.rt_bvh_info(s)
    assert info["status"] == 0 and info["n_leaves"] == info["n_bvh2_internal"] + 1
    return info, rb.rt_bvh_export(s)


@pytest.mark.parametrize("bins", [4, 10, 11, 16, 17, 32])
@pytest.mark.parametrize("max_leaf", [1, 15])
def test_axes_per_warp_and_leaf_sizes(rb, orc, bins, max_leaf):
    sc, _, p = scenes.workload_medium(level=1)
    info, ex = _build(rb, sc.tris, p["source"], alpha=0.7, max_leaf=max_leaf, bins=bins, dist_norm=1)
    assert info["max_leaf_size"] <= max_leaf
    E.check_tree(orc, sc.tris, ex, 0.7, p["source"], 1, bins, sample=1200, seed=bins)


@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 64, 65, 255, 1023, 1024, 1025])
def test_node_sizes(rb, orc, n):
    tris = scenes.tiny_city(seed=2).tris
    tris = np.concatenate([tris, tris + np.float32([300, 0, 0])])[:n]
    _, ex = _build(rb, tris, (50.0, 60.0, 30.0), alpha=0.7, max_leaf=1, bins=16, dist_norm=1)
    E.check_tree(orc, tris, ex, 0.7, (50.0, 60.0, 30.0), 1, 16)
    assert np.array_equal(np.sort(ex["prims"]), np.arange(n))


def test_centroids_without_extent(rb, orc):
    """300 triangles of one box centre: no plane, every node halves its range."""
    rng = np.random.default_rng(1)
    h = rng.integers(1, 9, (300, 1, 1)).astype(np.float32)
    tris = np.float32([[[-1, -1, -1], [1, 1, 1], [1, -1, 0]]]) * h
    info, ex = _build(rb, tris, (0.0, 0.0, 30.0), alpha=0.7, max_leaf=2, bins=16, dist_norm=1)
    st = E.check_tree(orc, tris, ex, 0.7, (0.0, 0.0, 30.0), 1, 16)
    assert st["middle"] > 5 and info["max_leaf_size"] <= 2


def _city(n, seed=4):
    """At least n triangles: copies of one city side by side."""
    city = scenes.workload_batched(seed=seed)[0].tris
    k = -(-n // len(city))
    side = int(np.ceil(np.sqrt(k)))
    return np.concatenate([city + np.float32([3100.0 * (i % side), 3100.0 * (i // side), 0.0]) for i in range(k)])


def _check_nodes(orc, tris, ex, alpha, src, bins, pick, most=1500):
    """Every node x with pick(records of x) true (at most `most`, seeded) is split at an Eq. 2 minimum."""
    first, cnt, nl = E.node_ranges(ex)
    assert np.array_equal(np.sort(ex["prims"]), np.arange(len(tris)))
    chk = E.Checker(orc, tris, alpha, src, dist_norm=1, bins=bins)
    nodes = np.nonzero(pick(cnt))[0]
    nodes = np.random.default_rng(0).permutation(nodes)[:most]
    keys = E.morton_keys(chk.lo, chk.hi)
    for x in nodes:
        ids = ex["prims"][first[x]: first[x] + cnt[x]]
        if len(ids) <= E.MICRO:
            cands = chk.prefix_candidates(ids)
            mine = [c for c in cands if c[0] == nl[x]]
            assert np.all(np.diff(keys[ids]) >= 0)
        else:
            cands = chk.binned_candidates(ids)
            left = np.arange(len(ids)) < nl[x]
            mine = [c for c in cands if np.array_equal(c[1], left)]
        assert mine, "node %d: the split is not one of its candidates" % x
        best = min(cands, key=lambda c: c[-2])
        assert mine[0][-2] - best[-2] <= mine[0][-1] + best[-1]
    return len(nodes)


@pytest.mark.parametrize("n,bins,max_leaf", [(239000, 16, 4), (241000, 16, 4), (241000, 8, 1), (510000, 32, 15),
                                             (510000, 11, 2)])
@pytest.mark.parametrize("alpha", [1.0, 0.7])
def test_small_nodes_of_large_scenes(rb, orc, n, bins, max_leaf, alpha):
    """Either side of the sizes from which nodes of at most 64, then 128 records are left to single warps."""
    tris = _city(n)[:n]
    src = (1500.0, 1500.0, 25.0)
    info, ex = _build(rb, tris, src, alpha=alpha, max_leaf=max_leaf, bins=bins, dist_norm=1)
    assert info["max_leaf_size"] <= max_leaf
    assert _check_nodes(orc, tris, ex, alpha, src, bins, lambda c: (c > max_leaf) & (c <= 140)) > 500
    s = rb.rt_scene_upload(tris)  # and again: the same tree
    rb.rt_bvh_build(s, source=src, alpha=alpha, max_leaf=max_leaf, bins=bins, dist_norm=1)
    again = rb.rt_bvh_export(s)
    assert all(np.array_equal(ex[k], again[k]) for k in ("child", "leaf_first", "leaf_count", "prims"))


@pytest.mark.parametrize("n,bins", [(240000, 16), (300001, 32), (999999, 8), (1000003, 16)])
@pytest.mark.parametrize("alpha", [1.0, 0.7])
def test_big_nodes_of_large_scenes(rb, orc, n, bins, alpha):
    """Chunks of 1024 and 2048 records through shared memory, ragged last ones among them."""
    tris = _city(n)[:n]
    src = (1500.0, 1500.0, 25.0)
    _, ex = _build(rb, tris, src, alpha=alpha, max_leaf=4, bins=bins, dist_norm=1)
    assert _check_nodes(orc, tris, ex, alpha, src, bins, lambda c: (c > 1024) & (c < 20000), 60) == 60
    assert _check_nodes(orc, tris, ex, alpha, src, bins, lambda c: c >= 60000, 3) == 3


def test_centroids_without_extent_in_a_large_scene(rb, orc):
    """Stacks of triangles of one box centre: nodes of k_small's size without a usable plane."""
    rng = np.random.default_rng(3)
    at = rng.uniform(0, 4000, (4000, 1, 1, 3)).astype(np.float32).round()
    h = rng.integers(1, 9, (4000, 64, 1, 1)).astype(np.float32)
    tris = (np.float32([[-1, -1, -1], [1, 1, 1], [1, -1, 0]]) * h + at).reshape(-1, 3, 3)
    info, ex = _build(rb, tris, (0.0, 0.0, 30.0), alpha=1.0, max_leaf=2, bins=16, dist_norm=1)
    assert info["max_leaf_size"] <= 2
    assert np.array_equal(np.sort(ex["prims"]), np.arange(len(tris)))


@pytest.mark.parametrize("alpha", [1.0, 0.7])
def test_nodes_too_large_for_shared_memory(rb, orc, alpha):
    """4.6M triangles: nodes of 1025 .. T / 4096 records are no big nodes."""
    tris = _city(4600000)
    src = (1500.0, 1500.0, 25.0)
    _, ex = _build(rb, tris, src, alpha=alpha, max_leaf=4, bins=16, dist_norm=1)
    big = len(tris) // 4096
    assert big > 1060
    assert _check_nodes(orc, tris, ex, alpha, src, 16, lambda c: (c > 1024) & (c <= big)) >= 20
