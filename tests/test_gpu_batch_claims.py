"""GPU test of how a batched launch hands out its tiles: fragment counts around
one and two tiles per resident warp (the tiles taken by place, the first ones
from the counters, counters that run out at different times), in a workspace of
the full size (several work counters) and of 256 bytes (one), for every claim
size.  Every job's answers are the bits of the single-map call, and nothing
past a job's last fragment is written."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SMALL = 256


def _sizes():
    if not torch.cuda.is_available():
        return [0]
    wave = torch.cuda.get_device_properties(0).multi_processor_count * 40 * 128     # 40 warps of 128 fragments per SM
    return [1, 129, 128 * 64 + 5, wave - 1, wave + 1, 2 * wave - 128, 2 * wave + 129, 5 * wave + 77]


@pytest.mark.parametrize("chunk", [0, 1, 2, 8])
@pytest.mark.parametrize("workspace", ["full", SMALL])
def test_every_tile_is_answered_once(workspace, chunk):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1711_07793_gb300 import _native as N
    from paper_1711_07793_gb300 import api
    g = torch.Generator(device="cuda").manual_seed(5)
    depth = torch.where(torch.rand((300, 420), generator=g, device="cuda") < 0.02, 0.3, 1.0)
    for total in _sizes():
        # jobs of uneven sizes, some empty, that add up to `total`
        parts = [0, total // 3, 0, total - total // 3 - min(5, total // 2), min(5, total // 2)]
        jobs = []
        for n in parts:
            x, y = (torch.rand(n, generator=g, device="cuda") for _ in range(2))
            z = torch.full((n,), 0.75, device="cuda")
            sil, fil = (torch.full((n + 64,), -7.0, device="cuda") for _ in range(2))
            jobs.append((api.Job(0, x, y, z, vis_silhouette=sil[:n], vis_filter=fil[:n]), sil, fil))
        b = api.Batch([depth], [j[0] for j in jobs], chunk_tiles=chunk)
        assert b.workspace_bytes > SMALL
        nbytes = b.workspace_bytes if workspace == "full" else workspace
        b.workspace.fill_(-1)
        for _ in range(2):
            N.check("rbsm_batch_run",
                    N.lib().rbsm_batch_run(ctypes.byref(b.desc), ctypes.c_void_p(b.workspace.data_ptr()), nbytes,
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
        torch.cuda.synchronize()
        assert bool((b.workspace.view(torch.uint8)[nbytes:] == 255).all())      # nothing past the workspace
        for job, sil, fil in jobs:
            n = job.x.shape[0]
            if n:
                assert torch.equal(sil[:n], api.rbsm_visibility(depth, job.x, job.y, job.z)[0]), (total, n)
                assert torch.equal(fil[:n], api.rsmss_filter(depth, job.x, job.y, job.z)[0]), (total, n)
            assert bool((sil[n:] == -7.0).all()) and bool((fil[n:] == -7.0).all())
