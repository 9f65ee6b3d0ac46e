"""GPU test of the edge walks (edge_walks in csrc/rbsm_device.cuh): every kind
of fragment (straight edge, corner, dead end, one-texel feature, lone texel)
with walks that end, leave the edge, run into the border or into the cap, on
maps down to one texel wide, against the oracle: codes and silhouette bit for
bit, filtering within 1e-5 (one float32 add and divide per axis against the
oracle's float64).  Once with few fragments (CTAs of 256 threads, walks one
step at a time) and once with the same fragments repeated until the single-map
calls take their CTAs of 1024 threads, whose walks go two steps at a time past
the second."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import rbsm as orc  # noqa: E402
from tests.test_gpu_parity import assert_parity, dev  # noqa: E402


def _map(rng, w, h):
    """Lit and shadowed runs along both axes, with one-texel lines, holes and islands."""
    m = np.ones((h, w), np.float32)
    for _ in range(max(2, w * h // 60)):
        j, i = rng.integers(0, h), rng.integers(0, w)
        n = int(rng.integers(1, 24))
        d = np.float32(rng.choice([0.25, 0.5, 1.0]))
        if rng.random() < 0.5:
            m[j, i:i + n] = d
        else:
            m[j:j + n, i] = d
    return m


CAPS = pytest.mark.parametrize("max_dist", [1, 2, 3, 16, 255])
SIZES = pytest.mark.parametrize("size", [(1, 1), (1, 40), (40, 1), (2, 3), (33, 29), (64, 48), (300, 5)])
TEXTURES = pytest.mark.parametrize("texture", [False, True])


def _case(size, max_dist, texture):
    """(api, map, map on the GPU, fragments)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1711_07793_gb300 import api
    w, h = size
    rng = np.random.default_rng(w * 1000 + h * 10 + max_dist)
    m = _map(rng, w, h)
    # every texel with two offsets and two depths, and points outside the map
    i, j = np.meshgrid(np.arange(w), np.arange(h))
    pts = [((i + fx) / w, (j + fy) / h, np.full(i.shape, z)) for fx, fy, z in
           ((0.25, 0.75, 0.3), (0.5, 0.125, 0.75), (0.9, 0.6, 0.75))]
    pts.append((np.array([-0.5, 1.5, 0.5]), np.array([0.5, 0.5, -2.0]), np.full(3, 0.75)))
    x, y, z = (np.concatenate([p[k].reshape(-1) for p in pts]).astype(np.float32) for k in range(3))
    if texture:
        pitched = torch.zeros((h, (w + 31) // 32 * 32), dtype=torch.float32, device="cuda")[:, :w]
        pitched.copy_(dev(m))
        depth = api.MapTexture(pitched)
    else:
        depth = dev(m)
    return api, m, depth, (x, y, z)


@CAPS
@SIZES
@TEXTURES
def test_walks_match_the_oracle(size, max_dist, texture):
    api, m, depth, (x, y, z) = _case(size, max_dist, texture)
    for fn, mode in ((api.rbsm_visibility, orc.MODE_SILHOUETTE), (api.rsmss_filter, orc.MODE_FILTER)):
        vis, codes = fn(depth, dev(x), dev(y), dev(z), codes=True, max_dist=max_dist)
        torch.cuda.synchronize()
        ref = orc.evaluate(m, x, y, z, mode, max_dist=max_dist)
        assert_parity(vis.cpu().numpy(), codes.cpu().numpy().view(np.uint16), ref, mode, "%s %d" % (size, max_dist))


@CAPS
@SIZES
@TEXTURES
def test_walks_of_large_calls_match_the_oracle(size, max_dist, texture):
    api, m, depth, (x, y, z) = _case(size, max_dist, texture)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    times = 128 * 32 * sms // x.size + 1               # 32 tiles of 128 for every SM
    n = times * x.size
    xyz = [dev(a).repeat(times) for a in (x, y, z)]
    for fn, mode in ((api.rbsm_visibility, orc.MODE_SILHOUETTE), (api.rsmss_filter, orc.MODE_FILTER)):
        ref = orc.evaluate(m, x, y, z, mode, max_dist=max_dist)
        vis, codes = fn(depth, *xyz, codes=True, max_dist=max_dist)
        # every repetition is the first one, and the first one the oracle's
        assert torch.equal(vis, vis[:x.size].repeat(times)) and torch.equal(codes, codes[:x.size].repeat(times))
        assert_parity(vis[:x.size].cpu().numpy(), codes[:x.size].cpu().numpy().view(np.uint16), ref, mode,
                      "%s %d, %d fragments" % (size, max_dist, n))
        # the kernel that writes no codes
        assert torch.equal(fn(depth, *xyz, codes=False, max_dist=max_dist)[0], vis)
