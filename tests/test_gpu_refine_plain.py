"""The plain and per-pair refinement give a path to a warp while there are few and to a thread
when there are many; on both sides of the line the records are those of the batched form: the
iterations' results and decisions bit for bit, the outputs to the last place."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import scenes

from parity_util import in_key_order

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


@pytest.mark.parametrize("nrx,K,target,below", [(1, 6, 0.0, 0.0), (3, 16, 1.7e-4, 0.0), (90, 9, 0.0, 0.03),
                                                (300, 7, 1.7e-4, 1e-3)])
def test_warp_and_thread_per_path_alike(gpu_ctx, nrx, K, target, below):
    """About 25 paths a receiver: below and above three paths a warp of the plain launch."""
    sc, tx, _ = scenes.random_clutter(nrx=1)
    rng = np.random.default_rng(nrx)
    rx = scenes.f32_exact(rng.uniform([1, 1, 1], [19, 15, 5], (nrx, 3)))
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx)
    paths = gpu_ctx.paths_create(1 << 17, 1 << 15)
    kw = dict(target=target, fp64_below=below)
    res = []
    for form in ("batch", "plain", "pair"):
        gpu_ctx.launch(scene, tx, rxs, paths, 64, 3, rx_angle_scale=SQ3, sync=True)
        log = torch.full((paths.path_cap, 10), -1, dtype=torch.int8, device="cuda")
        if form == "batch":
            gpu_ctx.batch_refine(scene, paths, 10, K, choice_log=log, **kw)
        elif form == "plain":
            gpu_ctx.refine(scene, paths, 10, K, choice_log=log, **kw)
        else:
            for r in range(nrx):
                gpu_ctx.refine_pair(scene, paths, 0, r, 10, K, **kw)
        got, choice = in_key_order(gpu_ctx.query(paths), log.cpu().numpy())
        res.append((got, choice))
    ref, choice = res[0]
    assert (len(ref) > 5472 if nrx == 300 else len(ref) > 20)
    assert np.array_equal(choice, res[1][1])
    for got, _ in res[1:]:
        for f in ("rx", "ray", "order", "faces", "iters", "valid", "flags", "dir", "err", "delay"):
            assert np.array_equal(ref[f], got[f]), f
        for f in ("aod", "aoa", "power_dbm"):   # FP32, at most an ulp of pi or of the power apart
            ulp = 2.4e-7 if f != "power_dbm" else 1.6e-5
            assert np.nanmax(np.abs(ref[f] - got[f])) <= ulp, f
    for h in (paths, rxs, scene):
        h.close()
