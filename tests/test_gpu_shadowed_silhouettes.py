"""GPU test of what a shadowed fragment costs in silhouette recovery on a map
without a texture: it reads its own texel and no neighbours (Listing 1: it stays
shadowed), so where the fragments' rows run across the map's rows, and every load
touches lines of its own, a view in full shadow takes well under the time of the
same view lit (a third of it; four fifths when the neighbours are read as well).
The answers of views half and fully in shadow are the shadow test's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

W, SIDE = 4096, 2828


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1711_07793_gb300 import api as A
    return A


def _call(api, what, depth):
    """(call, its answers): SIDE x SIDE fragments whose rows run along the map's columns."""
    t = (torch.arange(SIDE, device="cuda").float() + 0.5) / SIDE
    x, y, z = t.repeat_interleave(SIDE), t.repeat(SIDE), torch.full((SIDE * SIDE,), 0.75, device="cuda")
    if what == "planes":
        vis = torch.empty_like(x)
        return lambda: api.rbsm_visibility(depth, x, y, z, vis=vis), vis
    if what == "batch":
        job = api.Job(0, x, y, z, mode=1)
        batch = api.Batch([depth], [job])
        return lambda: api.rbsm_batch_run(batch), job.vis_silhouette
    m = np.zeros((4, 4), np.float32)
    m[0, 1] = m[1, 0] = 1.0 / SIDE
    m[2, 2] = m[3, 3] = 1.0
    job = api.GBufferJob(depth, z.view(SIDE, SIDE), m, mode=1)
    return lambda: api.rbsm_visibility_gbuffer([job], mode=1), job.vis_silhouette


def _time(call):
    for _ in range(5):
        call()
    times = []
    for _ in range(9):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(10):
            call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return sorted(times)[4]


@pytest.mark.parametrize("what", ["planes", "batch", "depth buffer"])
def test_shadowed_fragments_read_no_neighbours(api, what):
    depth = torch.full((W, W), 1.0, device="cuda")
    call, vis = _call(api, what, depth)
    lit = _time(call)
    assert bool((vis == 1).all())
    depth.fill_(0.1)
    shadowed = _time(call)
    assert bool((vis == 0).all())
    assert shadowed < 0.6 * lit, (shadowed, lit)
    depth[:, W // 2:] = 1.0
    vis.fill_(-1)
    call()
    # the fragments on either side of the straight edge take their shadow test (an I shape)
    rows = vis.view(SIDE, SIDE)
    assert bool((rows[:SIDE // 2] == 0).all()) and bool((rows[SIDE // 2:] == 1).all())
