"""The diffraction search tests a wedge against the beam of 32 rays before it tests the rays.  Edges that point
almost at the transmitter, or pass it close by, lose most digits of that angle in FP32 (about 1.3e-7 /
sin^2 of the angle between the edge and the line of sight, rad), so the beam allows for it: every (ray,
wedge) pair that a ray's own test finds, launched by itself, is found with all rays together."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import api, scenes

pytestmark = pytest.mark.gpu


def _spikes(o, count, seed, tilt):
    """Thin tetrahedra whose longest edge points at o up to an angle of about `tilt`, most of them past it."""
    rng = np.random.default_rng(seed)
    unit = lambda v: v / np.linalg.norm(v, axis=1)[:, None]
    r = unit(rng.normal(size=(count, 3)))
    t = unit(np.cross(r, rng.normal(size=(count, 3))))
    e = unit(r + t * (tilt * 10 ** rng.uniform(-1, 1, count))[:, None])
    a = o + r * rng.uniform(5, 60, count)[:, None]
    b = a - e * rng.uniform(5, 100, count)[:, None]
    w = 0.02 * (1 + rng.random(count))[:, None]
    c, d = (a + b) / 2 + t * w, (a + b) / 2 + np.cross(e, t) * w
    verts = np.stack([a, b, c, d], 1).reshape(-1, 3).astype(np.float32)
    tris = np.array([[0, 2, 1], [0, 1, 3], [0, 3, 2], [1, 2, 3]])
    tris = (tris[None] + 4 * np.arange(count)[:, None, None]).reshape(-1, 3)
    return verts, tris


@pytest.mark.parametrize("tilt", [1e-5, 3e-4, 1e-2])
def test_pairs_of_single_rays_are_all_found(gpu_ctx, tilt):
    o = scenes.f32_exact(np.array([[40.3, 25.7, 10.1]]))
    verts, tris = _spikes(o[0], 2000, 4, tilt)
    scene = gpu_ctx.scene_upload(verts, tris, np.arange(len(tris)))
    rxs = gpu_ctx.rx_upload(o.astype(np.float32) + 500.0)
    paths = gpu_ctx.paths_create(1 << 21, 1 << 10)
    n = 60

    def candidates(rng):
        gpu_ctx.launch(scene, o, rxs, paths, n, 0, rx_angle_scale=3.0 ** 0.5, diffraction=True, records_only=True,
                       ray_range=rng)
        return gpu_ctx.launch_stats(paths)["diffraction_candidates"]

    whole, single = [], []
    for b in np.random.default_rng(2).integers(12 + 30 * (n - 1), api.num_rays(n) - 128, 6):   # rays of one group
        whole.append(candidates((int(b), int(b) + 128)))
        single.append(sum(candidates((i, i + 1)) for i in range(int(b), int(b) + 128)))
    for h in (paths, rxs, scene):
        h.close()
    assert sum(whole) > 2000
    assert whole == single
