"""The 4-wide nodes keep half extents in FP16, rounded up: a scene scaled by a power of two (every
coordinate and distance scales exactly) must give every ray the same faces and every receiver the
same records, whether the extents fall into FP16's subnormals, its normal range or beyond it
(+inf: such a box is visited by every ray)."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


def _trace(ctx, sc, tx, rx, scale, n=40, order=3):
    scene = ctx.scene_upload(sc.verts * scale, sc.tris, sc.tri_face, None, sc.nf)
    rxs, paths = ctx.rx_upload(rx * scale), ctx.paths_create(1 << 16, 1 << 14)
    dump = torch.full((1, 10 * n * n + 2, order + 1), -3, dtype=torch.int32, device="cuda")
    ctx.launch(scene, tx * scale, rxs, paths, n, order, rx_angle_scale=SQ3, sync=True, dump_stride=1, dump=dump)
    r = ctx.records(paths)
    ctx.batch_refine(scene, paths, 8, 9)
    q = ctx.query(paths)
    for h in (paths, rxs, scene):
        h.close()
    r = r[np.lexsort((r["order"], r["rx"], r["ray"]))]
    q = q[np.lexsort((q["order"], q["rx"], q["ray"]))]
    return dump.cpu().numpy(), r, q


@pytest.mark.parametrize("k", [-20, -10, 7, 11, 13, 16])
def test_scaled_scene_traces_alike(gpu_ctx, k):
    sc, tx, rx = scenes.random_clutter(nrx=6)
    d1, r1, q1 = _trace(gpu_ctx, sc, tx, rx, 1.0)
    d2, r2, q2 = _trace(gpu_ctx, sc, tx, rx, 2.0 ** k)
    assert np.array_equal(d1, d2)
    assert len(r1) > 50 and (d1[..., 1:] >= 0).any()
    for f in ("tx", "rx", "ray", "order", "faces", "err"):
        assert np.array_equal(r1[f], r2[f]), f
    for f in ("rx", "ray", "order", "faces", "valid"):   # occlusion walks the same nodes
        assert np.array_equal(q1[f], q2[f]), f
