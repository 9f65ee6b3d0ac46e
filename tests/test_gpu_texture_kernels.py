"""GPU test of the kernels made for maps with and without a texture: the two
read the same texels in different ways and give the lanes different fragments,
so their answers and codes agree bit for bit, on full and partial tiles, on
aligned and unaligned planes, and on depth buffers whose rows are about as
long as a lane's steps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scene():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1711_07793_gb300 import api
    g = torch.Generator(device="cuda").manual_seed(11)
    depth = torch.where(torch.rand((130, 192), generator=g, device="cuda") < 0.02, 0.3, 1.0)
    return api, g, depth, api.MapTexture(depth)


@pytest.mark.parametrize("codes", [False, True])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 128 * 300 + 5, 128 * 32 * 160 + 64])
def test_planes(scene, n, codes):
    api, g, depth, tex = scene
    x, y, z = (torch.rand(n + 1, generator=g, device="cuda") * 1.04 - 0.02 for _ in range(3))
    for shift in (0, 1):
        xyz = [t[shift:n + shift] for t in (x, y, z)]
        for call in (api.rbsm_visibility, api.rsmss_filter):
            a, b = call(depth, *xyz, codes=codes), call(tex, *xyz, codes=codes)
            assert torch.equal(a[0], b[0])
            assert not codes or torch.equal(a[1], b[1])


@pytest.mark.parametrize("mode", [1, 2, 3])
@pytest.mark.parametrize("w", [1, 31, 32, 33, 63, 64, 65, 96, 127, 128, 333])
def test_depth_buffers(scene, w, mode):
    api, g, depth, tex = scene
    h = 128 * 7 // w + 5
    d = torch.rand((h, w), generator=g, device="cuda")
    m = np.eye(4, dtype=np.float32)
    m[0, 0], m[1, 1] = 1.0 / w, 1.0 / h
    a, b = (api.GBufferJob(t, d, m, mode=mode, codes=w % 2 == 0) for t in (depth, tex))
    for job in (a, b):
        api.rbsm_visibility_gbuffer([job], mode=mode)
    if w % 2 == 0:
        assert torch.equal(a.codes, b.codes)
    if mode & 1:
        assert torch.equal(a.vis_silhouette, b.vis_silhouette)
    if mode & 2:
        assert torch.equal(a.vis_filter, b.vis_filter)


@pytest.mark.parametrize("codes", [False, True])
@pytest.mark.parametrize("mode", [1, 2, 3])
def test_batches(scene, mode, codes):
    """Jobs of fewer and of more fragments than half the map's texels (24960): the line between the kernels."""
    api, g, depth, tex = scene
    for sizes in ([12480, 129], [12481, 31], [40000, 5000, 127]):
        xyz = [[torch.rand(n, generator=g, device="cuda") * 1.04 - 0.02 for _ in range(3)] for n in sizes]
        runs = []
        for m in (depth, tex):
            batch = api.Batch([m], [api.Job(0, *p, mode=mode, codes=codes or None) for p in xyz])
            api.rbsm_batch_run(batch)
            runs.append(batch.jobs)
        for a, b in zip(*runs):
            for k in ("vis_silhouette", "vis_filter", "codes"):
                assert (getattr(a, k) is None) == (getattr(b, k) is None)
                assert getattr(a, k) is None or torch.equal(getattr(a, k), getattr(b, k))
