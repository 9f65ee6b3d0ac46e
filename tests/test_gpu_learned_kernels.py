"""GPU test of the kernels the guarded surrogate runs in: with a texture and
without, with codes and without, on maps wide and narrow for their fragments
(which choose between fragments in pairs and single ones), with one mode for
all jobs and with mixed modes, and at every CTA size.  The answers, codes and
counts are the same bits in all of them; an answer the network did not give is
the exact filter's, and one it gave is within the surrogate's stated bound."""
import os

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TAU, WORST = 0.01, 0.1          # the guard and the largest error that are stated for the committed checkpoint


@pytest.fixture(scope="module")
def scene():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import rbsm_scenes as sc
    from paper_1711_07793_gb300 import api
    from paper_1711_07793_gb300.surrogate import Surrogate
    net = Surrogate.from_checkpoint(os.path.join(os.path.dirname(api.__file__), "weights", "surrogate_c4.npz"))
    f = sc.config2(41, screen=(960, 540))
    depth = torch.from_numpy(f.depth).cuda()
    xyz = [torch.from_numpy(a).cuda() for a in (f.x, f.y, f.z)]
    n = xyz[0].numel()
    assert depth.numel() >= 2 * n
    assert depth.numel() < 2 * 5 * n             # the narrow case repeats the fragments five times
    return api, net, depth, api.MapTexture(depth), xyz


@pytest.mark.parametrize("threads", [0, 128, 512])
@pytest.mark.parametrize("jobs", ["wide", "narrow", "ragged", "mixed"])
def test_every_kernel_gives_the_same_answers(scene, jobs, threads):
    api, net, depth, tex, xyz = scene
    n = xyz[0].numel()
    sets = {"wide": [(2, xyz)], "narrow": [(2, [t.repeat(5) for t in xyz])],
            "ragged": [(2, [t[k:k + m] for t in xyz]) for k, m in ((1, 100001), (0, 0), (7, 31), (4, n - 4))],
            "mixed": [(2, xyz), (1, xyz), (3, xyz), (2, [t[:5000] for t in xyz])]}[jobs]
    runs = {}
    for texture in (False, True):
        for codes in (False, True):
            made = [api.Job(0, *p, mode=m, codes=codes or None) for m, p in sets]
            b = api.Batch([tex if texture else depth], made, surrogate=net, guard_tau=TAU, tile_threads=threads)
            api.rbsm_batch_run(b)
            torch.cuda.synchronize()
            runs[texture, codes] = made, api.rbsm_batch_surrogate_counts(b)
    base, counts = runs[False, True]
    answered = edges = 0
    for job, (mode, p) in zip(base, sets):
        if p[0].numel() == 0:
            continue
        exact, ex_codes = api.rsmss_filter(depth, *p, codes=True)
        if mode & 1:
            assert torch.equal(job.vis_silhouette, api.rbsm_visibility(depth, *p)[0])
        if mode != 2:
            assert mode == 1 or torch.equal(job.vis_filter, exact)
            continue
        learned = (job.codes >> 10 & 1) == 1
        edge = (ex_codes >> 9 & 1) == 1
        assert not bool((learned & ~edge).any())
        assert torch.equal(job.vis_filter[~learned], exact[~learned])
        assert torch.equal(job.codes[~learned], ex_codes[~learned])
        assert torch.equal(job.codes[learned] & 0x3FF, ex_codes[learned] & 0x1F)
        assert bool(((job.vis_filter[learned] - exact[learned]).abs() <= WORST).all())
        answered += int(learned.sum())
        edges += int(edge.sum())
    assert answered > 1000 and counts == (answered, edges - answered)
    for (texture, codes), (made, got) in runs.items():
        assert got == counts, (texture, codes)
        for a, b in zip(made, base):
            for k in ("vis_silhouette", "vis_filter", "codes"):
                t = getattr(a, k)
                assert t is None or torch.equal(t, getattr(b, k)), (texture, codes, k)
