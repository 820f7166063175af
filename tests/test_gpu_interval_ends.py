"""Hits at the ends of a ray's interval (needs a GB300): rays that start on a
facet (the facet's own hit lies within rounding of tmin, on either side), rays
that end on one, and intervals that begin before the origin.  Every answer is
the float64 definition's, the lowest id where distances are equal."""
import numpy as np
import pytest

from paper_2208_10008_gb300 import scenes
from helpers import compare_closest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rb():
    from paper_2208_10008_gb300 import rtbvh
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    rtbvh.lib()
    return rtbvh


def _trace(rb, tris, rays, width, quant):
    s = rb.rt_scene_upload(tris)
    rb.rt_bvh_build(s, alpha=0.7, source=(100.0, 100.0, 30.0), max_leaf=4, bins=16, dist_norm=1, width=width,
                    quantize=quant)
    fl = rb.RT_QUANTIZED_NODES if quant else 0
    dev = torch.from_numpy(np.ascontiguousarray(rays)).cuda()
    h, occ = rb.rt_trace_closest(s, dev, flags=fl), rb.rt_trace_any(s, dev, flags=fl)
    torch.cuda.synchronize()
    return h.cpu().numpy(), occ.cpu().numpy()


def _scene():
    return scenes.prism_city(60, 200.0, 6)  # (walls in every direction: distances are rounded)


def _first_hits(orc, sc, n, seed):
    """Skew rays and the float32 points at which they meet the scene."""
    rays = scenes.random_rays(sc, n, seed=seed, tmax=400.0)
    ref = orc.closest_brute(sc.tris, rays)
    rays, t, ids = rays[ref.id >= 0], ref.t[ref.id >= 0], ref.id[ref.id >= 0]
    at = (rays[:, :3] + t[:, None] * rays[:, 4:7]).astype(np.float32)
    return rays, at, ids


@pytest.mark.parametrize("width,quant", [(4, 0), (8, 0), (4, 1)])
def test_rays_that_start_on_a_facet(rb, orc, width, quant):
    sc = _scene()
    _, at, ids = _first_hits(orc, sc, 12000, 8)
    rays = scenes.random_rays(sc, len(at), seed=9, tmax=400.0)  # (new directions, from the points of the hits)
    rays[:, :3] = at
    # some pass to the other side; the facet's hit is at |t| of 1e-5 or less
    ref = orc.closest_brute(sc.tris, rays)
    near = np.abs(ref.t) < 1e-4
    assert near.sum() > len(rays) // 50 and (ref.id[~near] >= 0).sum() > len(rays) // 4
    h, occ = _trace(rb, sc.tris, rays, width, quant)
    compare_closest(h, ref, sc.tris, rays, "start on a facet")
    assert (occ == (ref.id >= 0)).all()


@pytest.mark.parametrize("width,quant", [(4, 0), (8, 0), (4, 1)])
def test_rays_that_end_on_a_facet(rb, orc, width, quant):
    sc = _scene()
    rays, at, _ = _first_hits(orc, sc, 12000, 10)
    rays[:, 4:7] = at - rays[:, :3]
    rays[:, 7] = 1.0  # tmin < t < tmax: the facet is met or not by the float64 rounding of t
    ref = orc.closest_brute(sc.tris, rays)
    assert (ref.id >= 0).sum() > len(rays) // 8 and (ref.id < 0).sum() > len(rays) // 8
    h, occ = _trace(rb, sc.tris, rays, width, quant)
    compare_closest(h, ref, sc.tris, rays, "end on a facet")
    assert (occ == (ref.id >= 0)).all()


@pytest.mark.parametrize("width,quant", [(4, 0), (8, 0), (4, 1)])
def test_equal_distances_before_the_origin(rb, orc, width, quant):
    """Every facet twice, the copies in another order: the lower id, also at t < 0."""
    sc = _scene()
    n = len(sc.tris)
    tris = np.concatenate([sc.tris, sc.tris[np.random.default_rng(2).permutation(n)]])
    rays = scenes.random_rays(sc, 6001, seed=11, tmax=300.0)
    rays[:, 3] = -120.0
    ref = orc.closest_brute(tris, rays)
    assert (ref.t[ref.id >= 0] < 0).sum() > 2000
    h, occ = _trace(rb, tris, rays, width, quant)
    exact = np.isfinite(ref.t) & (ref.t2 == ref.t)
    assert exact.sum() > 2000
    ids = h.view(np.int32)[:, 1]
    assert (ids[exact] == ref.id[exact]).all() and ((ids >= 0) == (ref.id >= 0)).all()
    hit = ref.id >= 0
    assert np.all(np.abs(h[hit, 0] - ref.t[hit]) <= 1e-5 * np.abs(ref.t[hit]) + 1e-6)
    assert (occ == hit).all()
