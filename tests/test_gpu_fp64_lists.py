"""FP64 iterations of short lists: the tail of the batched refinement shares a path among 32 to 4
lanes, by the list's length and the iterations to come, the plain form among 32 or 8, and longer
lists take a thread a path.  Every length makes the decisions and results of the longest list's form,
bit for bit, and a list takes no longer than one many times as long."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import scenes

from parity_util import in_key_order

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))
PER_SM = 4 * 32   # lanes of the warps that a list in shared lanes may have an SM


def _rough(ctx, nrx):
    """Scene, transmitter, receivers, their rough paths of a room (about 63 a receiver) and a container."""
    sc, tx, _ = scenes.shoebox_config()
    rng = np.random.default_rng(nrx)
    rx = scenes.f32_exact(rng.uniform([0.4, 0.4, 0.4], [9.6, 7.6, 2.6], (nrx, 3)))
    scene, rxs = ctx.scene_from(sc), ctx.rx_upload(rx)
    paths = ctx.paths_create(1 << 18, 1 << 15)
    ctx.launch(scene, tx, rxs, paths, 16, 3, rx_angle_scale=SQ3, sync=True)
    rough = in_key_order(ctx.query(paths))[0]
    return scene, tx, rxs, rough[np.random.default_rng(1).permutation(len(rough))], paths


def _refined(ctx, scene, tx, rxs, rough, paths, K, iters, lanes):
    ctx.paths_import(paths, rough, tx, rxs, 16)
    log = torch.full((paths.path_cap, iters), -1, dtype=torch.int8, device="cuda")
    if lanes:
        ctx.batch_refine(scene, paths, iters, K, fp64_below=10.0, choice_log=log, lanes_per_path=lanes)
    else:
        ctx.refine(scene, paths, iters, K, fp64_below=10.0, choice_log=log)
    return ctx.query(paths), log.cpu().numpy()[: len(rough)]


@pytest.mark.parametrize("K,iters", [(6, 60), (7, 12), (9, 44), (16, 60), (16, 1)])
def test_lengths_alike(gpu_ctx, K, iters):
    scene, tx, rxs, rough, paths = _rough(gpu_ctx, 130)
    sms = gpu_ctx.num_sms
    lines = [PER_SM * sms // g for g in (32, 16, 8, 4)]   # the longest list of each number of lanes
    assert len(rough) > 48 * sms + 33
    want, choice = _refined(gpu_ctx, scene, tx, rxs, rough, paths, K, iters, 16)
    for n in [1, 33, 12 * sms, 12 * sms + 1, 48 * sms, 48 * sms + 1] + lines + [x + 1 for x in lines]:
        for lanes in (16, 1, 0):   # 0: the plain form
            got, log = _refined(gpu_ctx, scene, tx, rxs, rough[:n], paths, K, iters, lanes)
            assert np.array_equal(log, choice[:n]), (n, lanes)
            for f in ("iters", "valid", "flags", "dir", "err", "delay"):
                assert np.array_equal(got[f], want[f][:n]), (n, lanes, f)
    for h in (paths, rxs, scene):
        h.close()


def _time(ctx, scene, tx, rxs, rough, paths, K, lanes):
    best = np.inf
    for _ in range(5):
        ctx.paths_import(paths, rough, tx, rxs, 16)
        torch.cuda.synchronize()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        if lanes:
            ctx.batch_refine(scene, paths, 60, K, lanes_per_path=lanes)
        else:
            ctx.refine(scene, paths, 60, K)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("K", [6, 16])
@pytest.mark.parametrize("form", ["batch", "plain"])
def test_short_list_takes_no_longer(gpu_ctx, form, K):
    """900 and 4,000 paths against the whole list, run to the double floor.  (All lanes of a warp on the
    same path and sub-ray: 900 paths 1.3 times as long as 10,000 in the batched form, 4,000 four times
    in the plain one.)"""
    scene, tx, rxs, rough, paths = _rough(gpu_ctx, 150)
    assert len(rough) > 9000
    lanes = 16 if form == "batch" else 0
    whole, mid, short = (_time(gpu_ctx, scene, tx, rxs, rough[:n], paths, K, lanes) for n in (len(rough), 4000, 900))
    assert mid < 1.15 * whole and short < 1.15 * whole, (short, mid, whole)
    for h in (paths, rxs, scene):
        h.close()
