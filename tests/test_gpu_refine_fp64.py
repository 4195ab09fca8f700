"""The FP64 iteration of the precise algorithm (§III.B) ranks its sub-rays in FP32 and evaluates
in FP64 only those that may win.  Every decision it logs has to be the FP64 argmin of the cone
it stood on: the test walks the logged decisions in FP64 from the same start (the rough
direction, an FP32 vector taken as it is) and asks the oracle for the error angle of all K
sub-rays of every iteration, down to the double floor."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import scenes

from parity_util import in_key_order

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))
# Both sides run the same FP64 steps; they differ by rounding: at most a few 1e-16 rad in each
# of 44 centres and in each error angle, so a sub-ray chosen over a better one is at most
# 2 (44 x 2.2e-16 + 4e-16) = 2e-14 rad behind it.
TIE = 2e-14


@pytest.mark.parametrize("K,nrx", [(6, 1), (7, 20), (9, 20), (16, 1)])
def test_ranked_iteration_takes_the_fp64_argmin(gpu_ctx, oracle_mod, K, nrx):
    """K sub-rays, one receiver (a warp a path in the FP64 tail) or twenty (over 912 paths: a
    thread a path), every iteration in FP64, in the batched forms and the plain one."""
    sc, tx, _ = scenes.shoebox_config()
    rng = np.random.default_rng(K)
    rx = scenes.f32_exact(rng.uniform([0.4, 0.4, 0.4], [9.6, 7.6, 2.6], (nrx, 3)))
    n, order, cap = 16, 3, 44
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx)
    paths = gpu_ctx.paths_create(1 << 16, 1 << 13)
    S = oracle_mod.Scene.from_generated(sc)
    tl = float(np.float32(oracle_mod.theta_launch(n)))
    results = []
    for lanes in (16, 1, 0):   # 0: the plain form
        gpu_ctx.launch(scene, tx, rxs, paths, n, order, rx_angle_scale=SQ3, sync=True)
        rough = in_key_order(gpu_ctx.query(paths))[0]
        log = torch.full((paths.path_cap, cap), -1, dtype=torch.int8, device="cuda")
        kw = dict(fp64_below=10.0, choice_log=log)
        if lanes:
            gpu_ctx.batch_refine(scene, paths, cap, K, lanes_per_path=lanes, **kw)
        else:
            gpu_ctx.refine(scene, paths, cap, K, **kw)
        results.append(in_key_order(gpu_ctx.query(paths), log.cpu().numpy()))
    got, choice = results[0]
    assert len(got) > (912 if nrx > 1 else 60)
    for other, log in results[1:]:
        assert np.array_equal(choice, log)
        for field in ("iters", "dir", "err"):   # what the iteration writes
            assert np.array_equal(other[field], got[field]), field
    rho, phi, shrink = oracle_mod.subray_pattern(K)
    deep = 0
    for i in range(0, len(got), max(1, len(got) // 60)):
        r = got[i]
        it = int(r["iters"])
        faces = tuple(int(f) for f in r["faces"][: r["order"]])
        R0 = max(tl, float(r["rough_err"]))
        rep = oracle_mod.refine_ex(S, tx[0], rx[r["rx"]], faces, rough["dir"][i], R0, K, it,
                                   forced=choice[i][:it].astype(np.int32), stall=False)
        assert rep["iters"] == it
        c, R = rough["dir"][i].astype(np.float64), R0
        for j in range(it):
            u = np.cross(c, np.eye(3)[int(choice[i][j]) >> 4])
            u /= np.linalg.norm(u)
            a = (np.cos(phi)[:, None] * u + np.sin(phi)[:, None] * np.cross(c, u)) * np.sin(rho * R)[:, None]
            d = c * np.cos(rho * R)[:, None] + a
            e = np.array([oracle_mod.path_errors(S, tx[0], rx[r["rx"]], faces, x)[0] for x in d])
            e[~np.isfinite(rep["sub_err"][j])] = np.inf      # met a face out of order
            c = d[int(choice[i][j]) & 15]
            c, R = c / np.linalg.norm(c), R * shrink
            assert e[int(choice[i][j]) & 15] - np.min(e) <= TIE, (faces, j, e)
        deep += it == cap
    assert deep > 20
    for h in (paths, rxs, scene):
        h.close()
