"""The caller's events around the recursion (needs a GB300): in a large scene
they enclose the kernel of the small subtrees too."""
import numpy as np
import pytest

from paper_2208_10008_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [300_000, 1_000_000])
def test_split_events_enclose_the_small_subtrees(n):
    """After ev_end only the traversal nodes are left: 6-9% of a build, 24-36% with the small subtrees."""
    from paper_2208_10008_gb300 import rtbvh as rb
    city = scenes.workload_batched(seed=4)[0].tris
    k = -(-n // len(city))
    tris = np.concatenate([city + np.float32([3100.0 * i, 0.0, 0.0]) for i in range(k)])[:n]
    s = rb.rt_scene_upload(tris)
    after = []
    for _ in range(7):
        b0, b1, s0, s1 = (torch.cuda.Event(enable_timing=True) for _ in range(4))
        rb.rt_scene_set_split_events(s, s0, s1)
        b0.record()
        rb.rt_bvh_build(s, alpha=1.0, source=(1500.0, 1500.0, 25.0), max_leaf=4, bins=16)
        b1.record()
        torch.cuda.synchronize()
        assert 0 < s0.elapsed_time(s1) < b0.elapsed_time(b1)
        after.append(s1.elapsed_time(b1) / b0.elapsed_time(b1))
    assert np.median(after[2:]) < 0.15, after
