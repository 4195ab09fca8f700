"""The diffraction search walks the wedge tree once per group of 128 places of the schedule, by
the beam that holds their rays; rays that do not bundle walk it alone.  Its records on coarse
lattices (no group bundles), ordinary ones, in id order (other groups), on ray ranges that cut
groups and with a record array too small for the queue of exact tests are the same, and those of
the oracle's brute force over every wedge."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import api, scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


def _records(ctx, scene, tx, rxs, paths, n, **kw):
    ctx.launch(scene, tx, rxs, paths, n, 0, rx_angle_scale=SQ3, sync=True, diffraction=True, records_only=True, **kw)
    r = ctx.records(paths)
    r = r[(r["order"] == 1) & (r["faces"][:, 0] < 0)]
    return r[np.lexsort((r["rx"], r["faces"][:, 0], r["ray"], r["tx"]))]


@pytest.mark.parametrize("n", [1, 2, 3, 6, 24, 81])
def test_beams_find_every_wedge(gpu_ctx, oracle_mod, n):
    sc, tx, rx = scenes.urban_canyon(blocks=3)
    rng = np.random.default_rng(n)
    rx = scenes.f32_exact(rng.uniform([0, 0, 1], [165, 165, 20], (20, 3)))
    tx = scenes.f32_exact(np.concatenate([tx, tx + [3.0, -2.0, 9.0]]))
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx)
    paths = gpu_ctx.paths_create(1 << 20, 1 << 10)
    whole = _records(gpu_ctx, scene, tx, rxs, paths, n)
    assert len(whole) > 0
    assert _records(gpu_ctx, scene, tx, rxs, paths, n, id_order=True).tobytes() == whole.tobytes()
    N = 10 * n * n + 2
    for a, b in ((0, 1), (7, N), (N // 3, N // 3 + 50), (N // 2, N - 1)):
        a, b = min(a, N), min(b, N)
        part = whole[(whole["ray"] >= a) & (whole["ray"] < b)]
        assert _records(gpu_ctx, scene, tx, rxs, paths, n, ray_range=(a, b)).tobytes() == part.tobytes(), (a, b)
    # the smallest container (grown from the record count in steps of 1.25) that holds the launch,
    # receptions waiting for their occlusion query included: the least room for the queue
    cap = len(whole) + 64
    while True:
        small = gpu_ctx.paths_create(int(cap), 64)
        try:
            assert _records(gpu_ctx, scene, tx, rxs, small, n).tobytes() == whole.tobytes()
            break
        except api.SbrError as e:
            assert e.status == 5
        small.close()
        cap *= 1.25
    S = oracle_mod.Scene.from_generated(sc)
    cone = SQ3 * oracle_mod.theta_launch(n)
    for t in range(len(tx)):
        dr = oracle_mod.diffract(S, tx[t], oracle_mod.lattice(n), rx, cone)
        want = set(zip(dr.rec_ray.tolist(), dr.rec_wedge.tolist(), dr.rec_rx.tolist()))
        g = whole[whole["tx"] == t]
        got = set(zip(g["ray"].tolist(), (-1 - g["faces"][:, 0]).tolist(), g["rx"].tolist()))
        # decisions within FP32 rounding of the cone, the first-hit gate or an occluder's edge
        assert len(got ^ want) <= max(2, len(want) // 50), (t, sorted(got ^ want)[:8])
    for h in (small, paths, rxs, scene):
        h.close()
