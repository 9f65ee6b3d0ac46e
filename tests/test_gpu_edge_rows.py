"""GPU test of how the work of a shadow edge is shared out: where an edge runs
along the rows of fragments, and the rows along the map's columns, all the
fragments of several tiles in a row walk, each over lines of the map of its own.
Such a view (one straight edge through 1414 x 1414 fragments on a 2048^2 map) takes
about twice the time of the same view without the edge; when one SM gets all of the
edge's tiles, four to six times.  The answers on both sides of the edge are
the shadow test's (an I shape)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from tests.test_gpu_shadowed_silhouettes import _time  # noqa: E402

W, SIDE = 2048, 1414


@pytest.mark.parametrize("what", ["depth buffer", "filter", "silhouette", "rpcf1"])
def test_an_edge_along_the_rows(what):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1711_07793_gb300 import api
    depth = torch.full((W, W), 1.0, device="cuda")
    tex = api.MapTexture(depth)
    if what == "depth buffer":
        m = np.zeros((4, 4), np.float32)
        m[0, 1] = m[1, 0] = 1.0 / SIDE
        m[2, 2] = m[3, 3] = 1.0
        job = api.GBufferJob(tex, torch.full((SIDE, SIDE), 0.75, device="cuda"), m, mode=2)
        call, vis = (lambda: api.rbsm_visibility_gbuffer([job], mode=2)), job.vis_filter
    else:
        t = (torch.arange(SIDE, device="cuda").float() + 0.5) / SIDE
        xyz = t.repeat_interleave(SIDE), t.repeat(SIDE), torch.full((SIDE * SIDE,), 0.75, device="cuda")
        vis = torch.empty_like(xyz[0])
        call = {"filter": lambda: api.rsmss_filter(tex, *xyz, vis=vis), "rpcf1": lambda: api.rbsm_rpcf(tex, *xyz, k=1, vis=vis),
                "silhouette": lambda: api.rbsm_visibility(tex, *xyz, vis=vis)}[what]
    plain = _time(call)
    assert bool((vis == 1).all())
    depth[:, :W // 2] = 0.1
    edge = _time(call)
    rows = vis.view(SIDE, SIDE)
    assert bool((rows[:SIDE // 2] == 0).all()) and bool((rows[SIDE // 2:] == 1).all())
    assert edge < 3.3 * plain, (edge, plain)
