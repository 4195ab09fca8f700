"""With many paths the validity test walks the bounce points in one kernel and tests the legs in
another, a thread per (path, leg); with few a warp takes a path.  Both give every path the same
verdict and outputs, for orders 0 to 8 (nine legs), diffraction paths, blocked legs, points off
their faces and traces that fail; the one-lane form always takes the first way."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import _binding as B
from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


def _by_key(q):
    return q[np.lexsort(tuple(q["faces"][:, j] for j in range(7, -1, -1)) + (q["order"], q["ray"], q["rx"], q["tx"]))]


@pytest.mark.parametrize("make", ["room", "office", "street"])
def test_legs_alike_in_both_forms(gpu_ctx, make):
    kw = {}
    if make == "room":
        sc, tx, _ = scenes.shoebox_config()
        rng = np.random.default_rng(5)
        rx = scenes.f32_exact(rng.uniform([0.4, 0.4, 0.4], [9.6, 7.6, 2.6], (3, 3)))
        n, order = 48, 8
    elif make == "office":
        sc, tx, rx = scenes.office(nbox=60, ntx=2, nrx=40, g_shell=8, g_box=1)
        n, order = 48, 3
    else:
        sc, tx, rx = scenes.urban_canyon(blocks=4)
        n, order, kw = 96, 3, dict(diffraction=True)
    sc.face_eps = np.where(np.arange(sc.nf) % 3 == 0, 0.0, 5.0)
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx)
    paths = gpu_ctx.paths_create(1 << 21, 1 << 20)
    gpu_ctx.launch(scene, tx, rxs, paths, n, order, rx_angle_scale=SQ3, sync=True, **kw)
    rough = _by_key(gpu_ctx.query(paths))
    many = 16 * 32 * gpu_ctx.num_sms
    few = len(rough) < many
    res = []
    for lanes, copies in ((16, 1), (1, 1), (16, many // len(rough) + 1)):
        gpu_ctx.paths_import(paths, np.concatenate([rough] * copies), tx, rxs, n)   # the last: past the line
        gpu_ctx.batch_refine(scene, paths, 6, 9, lanes_per_path=lanes, freq=3e9, ptx_dbm=10.0)
        q = gpu_ctx.query(paths)
        for c in range(1, copies):
            assert q[c * len(rough):(c + 1) * len(rough)].tobytes() == q[:len(rough)].tobytes()
        res.append(q[:len(rough)])
    gpu_ctx.paths_import(paths, rough, tx, rxs, n)
    gpu_ctx.refine(scene, paths, 6, 9, freq=3e9, ptx_dbm=10.0)
    res.append(gpu_ctx.query(paths))
    a = res[0]
    assert few or make == "room"
    assert 0 < np.sum(a["valid"]) < len(a)
    if make == "street":
        d = (a["flags"] & B.PATH_DIFFRACTED) != 0
        assert 0 < np.sum(a["valid"][d]) < np.sum(d)
    if make == "room":
        assert (a["order"] == 8).any()
    for b in res[1:]:
        for f in ("iters", "valid", "flags", "dir", "err", "delay"):
            assert np.array_equal(a[f], b[f]), f
        for f in ("aod", "aoa", "power_dbm"):   # FP32, at most an ulp of pi or of the power apart
            ulp = 2.4e-7 if f != "power_dbm" else 1.6e-5
            assert np.nanmax(np.abs(a[f] - b[f])) <= ulp, f
    for h in (paths, rxs, scene):
        h.close()
