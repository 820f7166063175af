"""Boxes of the small subtrees of large scenes (needs a GB300): every node of
at most 128 records, where single warps split, holds the exact union of its
children's triangles, also where no plane splits a node; and rays through such
a scene against brute force."""
import numpy as np
import pytest

from paper_2208_10008_gb300 import scenes
import eq2_check as E
from helpers import compare_closest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rb():
    from paper_2208_10008_gb300 import rtbvh
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    rtbvh.lib()
    return rtbvh


def _range_unions(lo, hi, first, n):
    """Unions of the boxes of leaf positions first .. first + n - 1 (n <= 128): two overlapping powers of two."""
    levels = [(lo, hi)]
    for k in range(7):
        a, b = levels[-1]
        o = 1 << k
        levels.append((np.concatenate([np.minimum(a[:-o], a[o:]), a[-o:]]),
                       np.concatenate([np.maximum(b[:-o], b[o:]), b[-o:]])))
    k = np.floor(np.log2(n)).astype(int)
    out_lo, out_hi = np.empty((len(n), 3), np.float32), np.empty((len(n), 3), np.float32)
    for q in range(8):
        m = k == q
        a, b = first[m], first[m] + n[m] - (1 << q)
        out_lo[m] = np.minimum(levels[q][0][a], levels[q][0][b])
        out_hi[m] = np.maximum(levels[q][1][a], levels[q][1][b])
    return out_lo, out_hi


def _check_boxes(tris, ex):
    """Both children's boxes of every node of at most 128 records; returns (first, n, nl) of all nodes."""
    first, n, nl = E.node_ranges(ex)
    lo, hi = E.tri_boxes(tris)
    lo, hi = lo[ex["prims"]], hi[ex["prims"]]
    x = np.nonzero(n <= 128)[0]
    box = np.asarray(ex["boxes"]).reshape(-1, 12)[x]
    for s, (f, c) in enumerate([(first[x], nl[x]), (first[x] + nl[x], n[x] - nl[x])]):
        ulo, uhi = _range_unions(lo, hi, f, c)
        assert np.array_equal(box[:, 6 * s: 6 * s + 3], ulo) and np.array_equal(box[:, 6 * s + 3: 6 * s + 6], uhi)
    assert len(x) > len(tris) // 8
    return first, n, nl


def _city(n):
    city = scenes.workload_batched(seed=4)[0].tris
    k = -(-n // len(city))
    return np.concatenate([city + np.float32([3100.0 * i, 0.0, 0.0]) for i in range(k)])[:n]


@pytest.mark.parametrize("n,bins,max_leaf", [(241000, 16, 4), (241000, 8, 1), (510000, 32, 1), (510000, 11, 2)])
def test_boxes_of_small_nodes(rb, n, bins, max_leaf):
    tris = _city(n)
    s = rb.rt_scene_upload(tris)
    rb.rt_bvh_build(s, source=(1500.0, 1500.0, 25.0), alpha=0.7, max_leaf=max_leaf, bins=bins, dist_norm=1)
    assert rb.rt_bvh_info(s)["status"] == 0
    _check_boxes(tris, rb.rt_bvh_export(s))


@pytest.mark.parametrize("per", [64, 128])
def test_nodes_without_a_plane(rb, orc, per):
    """Stacks of 64 or 128 triangles of one box centre, in scenes whose single warps take nodes of that size."""
    k = 256000 // 64 if per == 64 else 512000 // 128
    rng = np.random.default_rng(3)
    side = int(np.ceil(np.sqrt(k)))
    at = np.stack([np.arange(k) % side, np.arange(k) // side, np.zeros(k)], 1).astype(np.float32) * 64 + 32
    at[:, 2] = rng.integers(10, 60, k)
    h = rng.integers(1, 30, (k, per, 1, 1)).astype(np.float32)
    t = np.float32([[-1, -1, -1], [1, 1, 1], [1, -1, 0]])
    tris = (t * h + at[:, None, None, :]).reshape(-1, 3, 3)
    s = rb.rt_scene_upload(tris)
    rb.rt_bvh_build(s, source=(0.0, 0.0, 30.0), alpha=1.0, max_leaf=2, bins=16)
    assert rb.rt_bvh_info(s)["status"] == 0
    ex = rb.rt_bvh_export(s)
    first, n, nl = _check_boxes(tris, ex)
    c = E.centres32(*E.tri_boxes(tris))[ex["prims"]]
    same = [x for x in np.nonzero((n > E.MICRO) & (n <= per))[0] if np.ptp(c[first[x]: first[x] + n[x]], axis=0).max() == 0]
    assert len(same) >= k and all(nl[x] == n[x] // 2 for x in same)
    # rays above the stacks, down through them
    rays = np.zeros((1500, 8), np.float32)
    rays[:, :3] = rng.uniform([0, 0, 100], [64 * side, 64 * side, 120], (1500, 3))
    d = rng.normal(size=(1500, 3)) - [0, 0, 3]
    rays[:, 4:7] = d / np.linalg.norm(d, axis=1, keepdims=True)
    rays[:, 7] = 1000.0
    got = rb.rt_trace_closest(s, torch.from_numpy(rays).cuda()).cpu().numpy()
    ref = orc.closest_brute(tris, rays)
    assert (ref.id >= 0).sum() > 300
    compare_closest(got, ref, tris, rays, "stacks")
