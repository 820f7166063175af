"""Compaction of the bounce at the edges of its tiles (needs a GB300): ray
counts around 256, 1024 and multiples, all, none and every k-th ray
surviving; and counts past the size up to which the scattering blocks add up
the counts themselves, where one block scans them.  Survivors, parents and
skips against a host compaction, rays against the float64 reflection."""
import numpy as np
import pytest

from paper_2208_10008_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def scene():
    from paper_2208_10008_gb300 import rtbvh
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    sc = scenes.tiny_city(seed=1)
    s = rtbvh.rt_scene_upload(sc.tris)
    rtbvh.rt_bvh_build(s, source=(100.0, 100.0, 30.0), max_leaf=4)
    return rtbvh, s, sc.tris


def _check(rb, s, rays, hits):
    out, skip, src, cnt = rb.rt_reflect(s, rays, hits)
    ids = hits[:, 1].view(torch.int32)
    keep = ((ids >= 0) & (rays[:, 7] - hits[:, 0] > 0)).nonzero()[:, 0]
    m = int(cnt.item())
    assert m == len(keep)
    assert torch.equal(src[:m].long(), keep)
    assert torch.equal(skip[:m], ids[keep])
    assert torch.equal(out[:m, 7], rays[keep, 7] - hits[keep, 0])
    return out[:m], keep


@pytest.mark.parametrize("n", [1, 31, 255, 256, 257, 1023, 1024, 1025, 2049, 65537, 1000003])
@pytest.mark.parametrize("every", [0, 1, 7])
def test_tile_edges(scene, orc, n, every):
    rb, s, tris = scene
    rays = rb.rt_gen_rays(rb.RT_RAYS_FIBONACCI, (100.0, 100.0, 30.0), n, 0.0, 1000.0)
    hits = rb.rt_trace_closest(s, rays)
    k = torch.arange(n, device="cuda")
    if every != 1:
        hits[:, 1].view(torch.int32)[(k % every != 0) if every else (k >= 0)] = -1
    out, keep = _check(rb, s, rays, hits)
    if len(keep):
        pick = keep[:: max(1, len(keep) // 500)]
        at = torch.searchsorted(keep, pick)
        h = hits[pick].cpu().numpy()
        ref = orc.reflect(tris, rays[pick].cpu().numpy(), h.view(np.int32)[:, 1].copy(), h[:, 0].astype(np.float64))
        got = out[at].cpu().numpy()
        assert np.abs(got[:, :3] - ref[:, :3]).max() <= 1e-4 and np.abs(got[:, 4:7] - ref[:, 4:7]).max() <= 1e-5


def test_more_tiles_than_a_block_adds_up(scene):
    rb, s, _ = scene
    n = 16384 * 1024 + 4097
    rays = rb.rt_gen_rays(rb.RT_RAYS_FIBONACCI, (100.0, 100.0, 30.0), n, 0.0, 1000.0)
    hits = rb.rt_trace_closest(s, rays)
    _check(rb, s, rays, hits)
