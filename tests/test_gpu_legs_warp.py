"""The batched refinement's few-path form gives a warp the nine legs of an order-8 path; the many-path form
walks it in a thread and tests each leg in one.  A set of paths below the line (16 paths an SM), long and
short ones, blocked ones and traces that fail among them, gets the same verdicts and outputs from both."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import _binding as B
from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


@pytest.mark.parametrize("make", ["room", "office"])
def test_nine_legs_alike(gpu_ctx, make):
    if make == "room":
        sc, tx, _ = scenes.shoebox_config()
        rx = scenes.f32_exact(np.random.default_rng(5).uniform([0.4, 0.4, 0.4], [9.6, 7.6, 2.6], (3, 3)))
    else:
        sc, tx, rx = scenes.office(nbox=60, ntx=2, nrx=40, g_shell=8, g_box=1)
        rx = rx[:8]
    sc.face_eps = np.where(np.arange(sc.nf) % 3 == 0, 0.0, 5.0)
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx)
    paths = gpu_ctx.paths_create(1 << 22, 1 << 20)
    gpu_ctx.launch(scene, tx, rxs, paths, 48, 8, rx_angle_scale=SQ3, sync=True)
    rough = gpu_ctx.query(paths)
    line = 16 * gpu_ctx.num_sms
    rng = np.random.default_rng(2)
    keep = [rng.permutation(np.flatnonzero(rough["order"] == k))[: line // 10] for k in range(9)]
    rough = rough[rng.permutation(np.concatenate(keep))]
    rough["faces"][:20, 2] = rough["faces"][:20, 1]   # a face twice in a row: no such trace
    assert len(rough) < line
    res = []
    for r in (rough, np.concatenate([rough] * (line // len(rough) + 1))):
        gpu_ctx.paths_import(paths, r, tx, rxs, 48)
        gpu_ctx.batch_refine(scene, paths, 6, 9, lanes_per_path=16, freq=3e9, ptx_dbm=10.0)
        res.append(gpu_ctx.query(paths)[: len(rough)])
    for h in (paths, rxs, scene):
        h.close()
    few, many = res
    long = few["order"] == 8
    assert np.sum(long) > 100 and 0 < np.sum(few["valid"][long]) < np.sum(long)
    assert np.any(few["flags"] & B.PATH_TRACE_FAIL)
    for f in ("iters", "valid", "flags", "dir", "err", "delay"):
        assert np.array_equal(few[f], many[f]), f
    for f in ("aod", "aoa", "power_dbm"):   # FP32: 4 units in the last place
        assert np.all(np.abs(few[f] - many[f]) <= 4 * np.spacing(np.abs(few[f]))), f
