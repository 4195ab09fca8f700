"""The batched refinement changes from a warp per path (validity test) to a thread per path and per
leg at 16 paths an SM.  The same paths, copied up to one below the line, onto it and past it, get the
same directions, verdicts, flags, errors and delays, bit for bit, whatever the lanes per path and
with FP64 iterations; the angles and powers, computed from those by either form, agree to 4 units in
the last place."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


@pytest.mark.parametrize("lanes", [8, 16, 32])
@pytest.mark.parametrize("off", [-1, 0, 1])
@pytest.mark.parametrize("make,iters", [("room", 24), ("street", 5)])
def test_forms_agree_at_the_line(gpu_ctx, make, iters, off, lanes):
    line, kw = 16 * gpu_ctx.num_sms, {}
    if make == "room":
        sc, tx, rx = scenes.shoebox_config()
        n, order = 32, 4
    else:
        sc, tx, rx = scenes.urban_canyon(blocks=4)
        n, order, kw = 64, 2, dict(diffraction=True)
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx)
    paths = gpu_ctx.paths_create(1 << 18, 1 << 16)
    gpu_ctx.launch(scene, tx, rxs, paths, n, order, rx_angle_scale=SQ3, sync=True, **kw)
    rough = gpu_ctx.query(paths)[: line // 2]
    m = len(rough)
    assert m > 10
    i = np.arange(line + off) % m
    res = []
    for r in (rough, rough[i]):
        gpu_ctx.paths_import(paths, r, tx, rxs, n)
        gpu_ctx.batch_refine(scene, paths, iters, 9, lanes_per_path=lanes)
        res.append(gpu_ctx.query(paths))
    for h in (paths, rxs, scene):
        h.close()
    few, many = res[0][i], res[1]
    assert 0 < np.sum(few["valid"]) and (make != "street" or np.sum(few["valid"]) < len(few))
    for f in ("tx", "rx", "ray", "order", "faces", "iters", "valid", "flags", "dir", "err", "delay"):
        assert np.array_equal(few[f], many[f]), f
    for f in ("aod", "aoa", "power_dbm"):
        assert np.all(np.abs(few[f] - many[f]) <= 4 * np.spacing(np.abs(few[f]))), f
