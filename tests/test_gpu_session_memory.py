"""What a serving session's pool holds (needs a GB300): a request is admitted
when its own buffers fit, 56 bytes a ray and order and a few kilobytes, and
refused when they do not."""
import numpy as np
import pytest

from paper_2208_10008_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("order", [0, 2, 8])
def test_a_request_takes_what_its_buffers_take(order):
    from paper_2208_10008_gb300 import rtbvh as rb
    n = 100_003
    need = 56 * n * (order + 1)
    sc = scenes.tiny_city(seed=1)
    s = rb.rt_scene_upload(sc.tris)
    rb.rt_bvh_build(s, alpha=0.7, source=(100, 100, 25), max_leaf=4, dist_norm=1)
    tx = (100.0, 100.0, 25.0)
    sess = rb.Session(pool_bytes=need + (1 << 16), max_slots=1)
    i = sess.add_scene(s)
    t = sess.submit(i, tx, rb.RT_RAYS_FIBONACCI, n, order, 500.0)
    sess.wait(t, timeout_s=60)
    hits, counts = sess.result(t)
    ref = rb.rt_trace_closest(s, rb.rt_gen_rays(rb.RT_RAYS_FIBONACCI, tx, n, 0.0, 500.0)).cpu().numpy()
    assert np.array_equal(hits.view(np.uint32), ref.view(np.uint32))
    assert counts[0] == n and need <= sess.stats()["peak_pool_bytes"] <= need + (1 << 16)
    with pytest.raises(rb.RtError):  # does not fit
        sess.submit(i, tx, rb.RT_RAYS_FIBONACCI, n + 1200 // (order + 1), order, 500.0)
    sess.destroy()
