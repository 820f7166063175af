"""The walk with warps whose lanes part at once (needs a GB300): random rays,
a ragged count, directions with zero, tiny or enormous components, far
origins, open intervals, non-finite triangles, large or moved coordinates.
Every hit is the float64 definition's (brute force), and the lanes' results
do not depend on each other: the rays reversed give the same bits reversed."""
import numpy as np
import pytest

from paper_2208_10008_gb300 import scenes
from helpers import compare_closest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N = 801  # not a multiple of a warp


@pytest.fixture(scope="module")
def rb():
    from paper_2208_10008_gb300 import rtbvh
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    rtbvh.lib()
    return rtbvh


def _rays(rng, tris, kind):
    lo, hi = tris.min((0, 1)), tris.max((0, 1))
    r = np.zeros((N, 8), np.float32)
    r[:, :3] = rng.uniform(lo, hi, (N, 3))
    d = rng.normal(size=(N, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    r[:, 4:7] = d
    r[:, 7] = 1e4
    if kind == "axis":  # one or two components zero of either sign; some in the ground plane, some through vertices
        for i in range(N):
            k = rng.permutation(3)[: rng.integers(1, 3)]
            r[i, 4 + k] = np.where(rng.random(len(k)) < 0.5, np.float32(0.0), np.float32(-0.0))
        r[::5, 2] = 0.0
        r[::5, 6] = 0.0
        v = tris[rng.integers(0, len(tris), N), rng.integers(0, 3, N)]
        r[1::5, :3] = v[1::5]
        r[1::5, 4:7] = rng.permuted(np.tile(np.float32([1, 0, -0.0]), (N, 1)), axis=1)[1::5]
        r[1::5, :3] -= 3.0 * r[1::5, 4:7]
    elif kind == "ratio":
        r[np.arange(N), 4 + rng.integers(0, 3, N)] *= np.float32(10.0) ** rng.integers(-45, -3, N).astype(np.float32)
    elif kind == "scaled":  # the same rays with |d| from 2^-90 to 2^90
        s = np.exp2(rng.integers(-90, 91, N)).astype(np.float32)
        r[:, 4:7] *= s[:, None]
        r[:, 7] /= s
    elif kind == "far":
        at = r[:, :3].copy()
        r[:, :3] = (at - 1e6 * d).astype(np.float32)
        r[:, 7] = 2e6
    elif kind == "open":
        r[::2, 3] = rng.uniform(0.0, 40.0, (N + 1) // 2)
        r[:, 7] = np.inf
        r[::3, 7] = 45.0
    return r


@pytest.mark.parametrize("kind", ["axis", "ratio", "scaled", "far", "open", "nonfinite", "huge", "moved"])
@pytest.mark.parametrize("width,quant", [(4, 0), (8, 0), (4, 1)])
def test_lanes_that_part(rb, orc, kind, width, quant):
    rng = np.random.default_rng(7)
    tris = scenes.tiny_city(seed=3).tris.copy()
    rays = _rays(rng, tris, kind)
    if kind == "nonfinite":
        bad = tris[:6].copy()
        bad[0, 0, 0], bad[1, 1, 2], bad[2, 0] = np.inf, -np.inf, np.nan
        bad[3, 2, 1] = np.nan
        bad[4, :, 0] = np.inf
        tris = np.concatenate([tris, bad])
    elif kind == "huge":
        tris *= np.float32(2.0 ** 30)
        rays[:, :3] *= np.float32(2.0 ** 30)
        rays[:, 7] *= np.float32(2.0 ** 30)
    elif kind == "moved":
        off = np.float32([3e5, -2e5, 1e5])
        tris = tris + off
        rays[:, :3] += off
    s = rb.rt_scene_upload(tris)
    rb.rt_bvh_build(s, alpha=0.7, source=tuple(float(x) for x in tris[0, 0]) if kind not in ("huge",) else (0., 0., 0.),
                    max_leaf=2, bins=16, dist_norm=1, width=width, quantize=quant)
    assert rb.rt_bvh_info(s)["status"] == 0
    fl = rb.RT_QUANTIZED_NODES if quant else 0
    dev = torch.from_numpy(rays).cuda()
    ref = orc.closest_brute(tris, rays)
    h = rb.rt_trace_closest(s, dev, flags=fl)
    back = rb.rt_trace_closest(s, dev.flip(0).contiguous(), flags=fl)
    occ = rb.rt_trace_any(s, dev, flags=fl)
    torch.cuda.synchronize()
    assert (ref.id >= 0).sum() > N // 20
    compare_closest(h.cpu().numpy(), ref, tris, rays, kind)
    assert torch.equal(back.flip(0).view(torch.int32), h.view(torch.int32))
    assert (occ.cpu().numpy() == (ref.id >= 0)).all()
