"""Scenes with triangles that hold no finite box (needs a GB300): vertices
without a number on one axis or on all, infinite ones of either sign.  No ray
meets such a triangle, and every other hit is the float64 definition's."""
import numpy as np
import pytest

from paper_2208_10008_gb300 import scenes
from helpers import compare_closest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NAN, INF = np.float32(np.nan), np.float32(np.inf)


def _bad(tris, kind, rng):
    t = tris[rng.integers(0, len(tris), 9)].copy()
    if kind == "nan":
        t[:] = NAN
    elif kind == "nan axis":
        t[np.arange(9), :, np.arange(9) % 3] = NAN
    elif kind == "nan corner":
        t[np.arange(9), np.arange(9) % 3] = NAN
    elif kind == "inf":
        t[np.arange(9), :, np.arange(9) % 3] = np.where(np.arange(9) < 5, INF, -INF)[:, None]
    elif kind == "inf corner":
        t[np.arange(9), np.arange(9) // 3, np.arange(9) % 3] = np.where(np.arange(9) % 2, INF, -INF)
    elif kind == "both":
        t[np.arange(9), 0, np.arange(9) % 3] = INF
        t[np.arange(9), 1, np.arange(9) % 3] = -INF
    return t


@pytest.mark.parametrize("kind", ["nan", "nan axis", "nan corner", "inf", "inf corner", "both"])
@pytest.mark.parametrize("width,quant", [(4, 0), (8, 0), (4, 1)])
@pytest.mark.parametrize("few", [True, False])
def test_triangles_without_a_finite_box(orc, kind, width, quant, few):
    from paper_2208_10008_gb300 import rtbvh as rb
    rng = np.random.default_rng(3)
    tris = scenes.prism_city(4 if few else 120, 200.0, 2).tris
    tris = tris[:24] if few else tris
    bad = _bad(tris, kind, rng)
    at = np.sort(rng.integers(0, len(tris), len(bad)))
    tris = np.insert(tris, at, bad, axis=0)
    rays = scenes.random_rays(scenes.prism_city(120, 200.0, 2), 3001, seed=8, tmax=400.0)
    if few:  # at points of the facets
        with np.errstate(invalid="ignore"):  # (points of the bad ones)
            d = (rng.dirichlet(np.ones(3), 3001)[:, :, None] * tris[rng.integers(0, len(tris), 3001)]).sum(1) - rays[:, :3]
        ok = np.isfinite(d).all(1)
        rays[ok, 4:7] = d[ok] / np.linalg.norm(d[ok], axis=1, keepdims=True)
    s = rb.rt_scene_upload(tris)
    rb.rt_bvh_build(s, alpha=0.7, source=(100.0, 100.0, 30.0), max_leaf=2, bins=16, dist_norm=1, width=width,
                    quantize=quant)
    assert rb.rt_bvh_info(s)["status"] == 0
    fl = rb.RT_QUANTIZED_NODES if quant else 0
    dev = torch.from_numpy(rays).cuda()
    h, occ = rb.rt_trace_closest(s, dev, flags=fl), rb.rt_trace_any(s, dev, flags=fl)
    torch.cuda.synchronize()
    ref = orc.closest_brute(tris, rays)
    assert (ref.id >= 0).sum() > 1000
    compare_closest(h.cpu().numpy(), ref, tris, rays, kind)
    assert (occ.cpu().numpy() == (ref.id >= 0)).all()
