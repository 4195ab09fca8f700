"""Launches of three million rays and more start their first segments from a frontier computed per
64 places (an interval of directions walked once).  Every ray's faces, the segments and the records
have to be those of the same rays launched in ranges too small for it, which start at the root:
from transmitters over streets, on a node box's plane, in a corner, above and outside the scene."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


def _run(ctx, scene, tx, rxs, paths, n, order, dump, **kw):
    ctx.launch(scene, tx, rxs, paths, n, order, rx_angle_scale=SQ3, sync=True, dump_stride=1, dump=dump,
               records_only=True, **kw)
    return ctx.launch_stats(paths)["segments"], ctx.records(paths)


def _sorted(r):
    rows = np.ascontiguousarray(r).view(np.uint32).reshape(len(r), 16)[:, :14]
    return rows[np.lexsort(rows.T[::-1])]


@pytest.mark.parametrize("make,launcher", [("canyon", 0), ("canyon", 20), ("city", 0), ("city", 8)])
def test_frontier_changes_no_ray(gpu_ctx, make, launcher):
    if make == "canyon":
        sc, tx, rx = scenes.urban_canyon(blocks=10)
        ext = 10 * 55.0
    else:
        sc, tx, rx = scenes.large_city(blocks=8, terrain_cells=93, ntx=1, nrx=100)
        ext = 8 * 55.0
    tx = scenes.f32_exact(np.array([tx[0], [47.5, 102.5, 0.25], [0.0, 0.0, 3.0], [ext / 2, ext / 2, 400.0],
                                    [-300.0, 40.0, 20.0]]))
    n = 250 if launcher != 8 else 390        # 3.0 - 3.1 million rays over the five
    N = (10 if launcher != 8 else 4) * n * n + 2
    order = 2
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx)
    assert scene.info()["bvh_nodes"] >= 1024 and 5 * N >= 3_000_000
    paths = gpu_ctx.paths_create(1 << 20, 64)
    shape = (5, N, order + 1)
    d1 = torch.full(shape, -3, dtype=torch.int32, device="cuda")
    d2 = torch.full(shape, -3, dtype=torch.int32, device="cuda")
    s1, r1 = _run(gpu_ctx, scene, tx, rxs, paths, n, order, d1, launcher=launcher)
    cut = N // 2 + 17
    s2, r2 = 0, []
    for a, b in ((0, cut), (cut, N)):
        s, r = _run(gpu_ctx, scene, tx, rxs, paths, n, order, d2, launcher=launcher, ray_range=(a, b))
        s2 += s
        r2.append(r)
    bad = (d1 != d2).any(-1).nonzero()
    assert len(bad) == 0, (len(bad), bad[:5].tolist())
    assert s1 == s2 and (d1[..., 1] >= 0).any() and (d1[3] == -1).any()
    assert len(r1) > 0 and np.array_equal(_sorted(r1), _sorted(np.concatenate(r2)))
    # and on a range that is large enough for it but cuts faces and groups
    if launcher == 0:
        big = np.concatenate([tx, tx + [1.5, -2.0, 1.0]])
        a, b = 5 * n, N - 333
        lone = torch.full((10, N, order + 1), -3, dtype=torch.int32, device="cuda")
        s3, r3 = _run(gpu_ctx, scene, big, rxs, paths, n, order, lone, ray_range=(a, b))
        assert torch.equal(lone[:5, a:b], d1[:, a:b]) and (lone[:, :a] == -3).all() and (lone[:, b:] == -3).all()
    for h in (paths, rxs, scene):
        h.close()
