"""Double-count removal on record sets made on the host: a warp appends its winners together and
skips atomics that cannot change a slot.  Whatever the duplicates (none, a few, every record one
path) and wherever the last warp ends, each key's smallest (error angle, ray) wins, once."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


@pytest.mark.parametrize("world", [1, 3])
@pytest.mark.parametrize("keys", [1, 7, 0])      # 0: every record a path of its own
@pytest.mark.parametrize("n", [1, 31, 33, 257, 5000, 300001])
def test_winners(gpu_ctx, n, keys, world):
    g = np.random.default_rng(n + keys)
    sc = scenes.shoebox()
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(np.array([[6.0, 3.0, 1.0], [2.0, 2.0, 2.0]], np.float32))
    paths = gpu_ctx.paths_create(n + 64, n + 64)
    gpu_ctx.launch(scene, np.array([[3.1, 4.2, 1.4]], np.float32), rxs, paths, 180, 0, rx_angle_scale=SQ3, sync=True)
    r = np.zeros(n, gpu_ctx.records(paths).dtype)
    k = np.arange(n) if keys == 0 else g.integers(0, keys, n)
    r["rx"], r["order"] = k & 1, 8
    r["faces"] = 1 + (k[:, None] >> np.arange(0, 24, 3)) % 8
    r["faces"][:, 0] += 8 * (k >> 1).astype(np.int32)
    r["err"] = g.integers(0, 4, n).astype(np.float32) * 2.0 ** -12      # many ties, broken by the ray id
    r["ray"] = g.permutation(n)   # a ray reports a path once
    r["slot"], r["pad"] = g.integers(-9, 9, n), 0                       # whatever the caller left there
    order = np.lexsort((r["ray"], r["err"], k))
    first = order[np.concatenate([[True], np.diff(k[order]) != 0])]
    want = r[first]
    want = want[(want["tx"] * 2 + want["rx"]) % world == world - 1]
    gpu_ctx.records_dedup(paths, r, rank=world - 1, world=world)
    got = gpu_ctx.query(paths)
    st = gpu_ctx.launch_stats(paths)
    for h in (paths, rxs, scene):
        h.close()
    assert len(got) == len(want) == st["paths"]
    a = {(int(p["rx"]), p["faces"].tobytes()): (int(p["ray"]), float(p["rough_err"])) for p in got}
    b = {(int(p["rx"]), p["faces"].tobytes()): (int(p["ray"]), float(p["err"])) for p in want}
    assert a == b
