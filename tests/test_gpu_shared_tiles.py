"""GPU test of the kernels whose CTAs share out their tiles (single-map calls,
depth buffers, RPCF): a fragment's answer does not depend on how many
fragments follow it, so the answers of n fragments are the first n of a larger
call's, bit for bit, for n around the strips, runs, CTA shapes and waves the
launches switch at; and nothing past the last fragment is written.  The map
holds runs and one-texel lines, so that the walks end at every step up to the
cap: small and large calls take them one and two steps at a time."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from tests.test_gpu_walks import _map  # noqa: E402


@pytest.fixture(scope="module")
def scene():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1711_07793_gb300 import api
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cuda").manual_seed(3)
    depth = torch.from_numpy(_map(np.random.default_rng(3), 384, 250)).cuda()
    n = sms * 40 * 128 * 3 + 77
    x, y = (torch.rand(n, generator=g, device="cuda") * 1.02 - 0.01 for _ in range(2))
    return api, sms, depth, x, y, torch.full((n,), 0.75, device="cuda")


def _counts(sms):
    return [1, 31, 33, 127, 129, 257, 8 * 32 * sms + 1, 128 * 32 * sms - 127, 128 * 32 * sms + 1, 128 * 40 * sms + 129]


@pytest.mark.parametrize("texture", [False, True])
@pytest.mark.parametrize("what", ["silhouette", "filter", "rpcf1", "rpcf3", "rpcf5"])
def test_a_prefix_gives_the_prefix(scene, what, texture):
    api, sms, depth, x, y, z = scene
    m = api.MapTexture(depth) if texture else depth

    def call(n, out):
        if what.startswith("rpcf"):
            return api.rbsm_rpcf(m, x[:n], y[:n], z[:n], k=int(what[4:]), vis=out)
        return (api.rbsm_visibility if what == "silhouette" else api.rsmss_filter)(m, x[:n], y[:n], z[:n], vis=out)[0]

    full = call(x.numel(), torch.empty_like(x))
    for n in _counts(sms):
        out = torch.full((n + 40,), -7.0, device="cuda")
        call(n, out[:n])
        assert torch.equal(out[:n], full[:n]), n
        assert bool((out[n:] == -7.0).all()), n


def test_a_prefix_of_the_rows_of_a_depth_buffer(scene):
    api, sms, depth, _, _, _ = scene
    w = 997
    full_h = 128 * 40 * sms * 2 // w
    g = torch.Generator(device="cuda").manual_seed(4)
    d = torch.rand((full_h, w), generator=g, device="cuda")
    m = np.eye(4, dtype=np.float32)
    m[0, 0], m[1, 1] = 1.0 / w, 1.0 / full_h
    full = api.GBufferJob(depth, d, m)
    api.rbsm_visibility_gbuffer([full])
    for h in (1, 2, 40, 128 * 20 * sms // w, full_h - 1):
        job = api.GBufferJob(depth, d[:h], m)
        api.rbsm_visibility_gbuffer([job])
        assert torch.equal(job.vis_silhouette, full.vis_silhouette[:h * w])
        assert torch.equal(job.vis_filter, full.vis_filter[:h * w])


@pytest.mark.parametrize("texture", [False, True])
@pytest.mark.parametrize("k", [3, 5, 7])
def test_rpcf_shadow_tests_on_special_depths(scene, k, texture):
    """RPCF takes its block's shadow tests from the signs of sums, the filter
    from comparisons: on maps and fragments of signed zeros, subnormals,
    infinities, NaN and equal depths it is the mean of the filter's answers at
    the shifted positions (exact in float32 on a power-of-two map), within the
    samples' rounding of 2^-21."""
    api = scene[0]
    w = 64
    v = torch.tensor([0.0, -0.0, 1e-45, -1e-45, 1e-38, 1.0, -1.0, 3e38, float("inf"), -float("inf"), float("nan")],
                     device="cuda")
    g = torch.Generator(device="cuda").manual_seed(k)
    depth = v[torch.randint(0, len(v), (w, w), generator=g, device="cuda")].contiguous()
    # runs of one value, so that walks go on
    depth[8:24, 8:56], depth[30:34, 4:60], depth[40:60, 20:22] = 0.0, -0.0, float("inf")
    n = w * w * 8
    i = torch.randint(0, w, (2, n), generator=g, device="cuda")
    x, y = ((t + 0.25 * (1 + (t + s) % 3)).float() / w for s, t in enumerate(i))
    z = v[torch.randint(0, len(v), (n,), generator=g, device="cuda")]
    m = api.MapTexture(depth) if texture else depth
    got = api.rbsm_rpcf(m, x, y, z, k=k)
    half, ref = (k - 1) // 2, torch.zeros(n, dtype=torch.float64, device="cuda")
    for b in range(-half, half + 1):
        for a in range(-half, half + 1):
            ref += api.rsmss_filter(m, x + a / w, y + b / w, z)[0].double()
    assert float((got.double() - ref / (k * k)).abs().max()) <= 2.0 ** -21
