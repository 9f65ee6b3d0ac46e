"""GPU test of the light pass's forms: tiles of 64 texels (maps of at least two
such tiles per resident CTA), and tiles of 32 with the warps on blocks of rows or
on rows spread over the tile, on both sides of the lines between them.  Odd sizes whose last tiles are partial, thin and wide
rectangles (blocks surely outside, surely covered, and cut), spheres from
sub-texel to several tiles, depth scales that are powers of two and not or
outside the float-float range, no occluders, more than one culling round of them
(which keeps the small tiles), and a pitched output; bit for bit the brute-force oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import rbsm as orc  # noqa: E402


def _occluders(rng, w, h, nr, ns):
    ang = rng.uniform(0, np.pi, nr)
    if nr:
        ang[:3] = (0.0, np.pi / 2, np.pi / 4)
    rects = np.stack([rng.uniform(-50, w + 50, nr), rng.uniform(-50, h + 50, nr), np.cos(ang), np.sin(ang),
                      rng.uniform(0.4, 400, nr), rng.uniform(0.4, 60, nr)], 1)
    rects[:1, :2] = np.floor(rects[:1, :2]) + 0.5                  # ties on texel centres
    rects[:1, 4:] = (64.0, 32.0)
    sph = np.stack([rng.uniform(-50, w + 50, ns), rng.uniform(-50, h + 50, ns), np.exp(rng.uniform(-1, 5.3, ns)),
                    rng.uniform(0.1, 0.9, ns)], 1)
    return rects, rng.uniform(0.05, 0.95, nr).astype(np.float32), sph


@pytest.mark.parametrize("w,h,nr,ns,zs", [(2305, 2241, 40, 25, 2048.0), (2305, 2241, 40, 25, 1000.0),
                                          (2240, 2240, 30, 30, 3.7), (2400, 2200, 0, 40, 0.3),
                                          (2400, 2200, 256, 0, 64.0), (2305, 2241, 250, 20, 777.7),
                                          (9000, 577, 30, 30, 1e3), (2305, 2241, 0, 0, 64.0),
                                          (2305, 2241, 10, 12, 2.0 ** 101),
                                          (160, 192, 20, 10, 64.0), (161, 192, 20, 10, 64.0), (161, 200, 200, 200, 3.0),
                                          (500, 333, 120, 60, 512.0), (500, 333, 300, 290, 77.7),
                                          (777, 768, 30, 20, 1000.0), (1, 1100, 12, 6, 2.0), (1089, 1120, 30, 20, 8.0),
                                          (1121, 1120, 30, 20, 8.0),
                                          (801, 800, 10, 300, 0.3)])
def test_maps(w, h, nr, ns, zs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1711_07793_gb300 import api
    rects, dep, sph = _occluders(np.random.default_rng(w + nr + ns), w, h, nr, ns)
    out = torch.full((h, w + 3), -7.0, device="cuda")
    api.rbsm_shadow_map(api.DeviceOccluders(rects, dep, sph), w, h, zs, ground=0.97, out=out[:, :w])
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    ref = orc.shadow_map(w, h, rects, dep, sph, zs, ground=0.97)
    assert np.array_equal(got[:, :w].view(np.uint32), ref.view(np.uint32))
    assert bool((got[:, w:] == -7.0).all())
