"""The receivers' tree is a median tree built on the device from 64 to 131,072 receivers and the
host builder's otherwise.  The same receivers, padded past that line with far ones outside the closed
room, must give the same reception records bit for bit: the trees only choose which receivers a segment
tests."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
LINE = 131072   # kRxDeviceMax in capi.cu
SQ3 = float(np.sqrt(3.0))


def _layout(kind, n, lo, hi):
    g = np.random.default_rng(n)
    u = g.random((n, 3))
    if kind == "grid":       # equal keys on every axis, one height
        k = int(np.ceil(np.sqrt(n)))
        u = np.stack([np.arange(n) % k / k, np.arange(n) // k / k, np.full(n, 0.5)], 1)
    elif kind == "one":      # every receiver at the same place
        u = np.repeat(u[:1], n, 0)
    elif kind == "streets":  # thin lines, far denser at one end
        u = np.stack([u[:, 0] ** 4, np.where(u[:, 1] < 0.5, 0.25, 0.75), np.full(n, 0.4)], 1)
    return (lo + (hi - lo) * (0.02 + 0.96 * u)).astype(np.float32)


def _records(ctx, scene, tx, rx, n):
    rxs, paths = ctx.rx_upload(rx), ctx.paths_create(1 << 23, 1 << 21)
    ctx.launch(scene, tx, rxs, paths, 12, 1, rx_angle_scale=SQ3, sync=True)
    r = ctx.records(paths)
    for h in (paths, rxs):
        h.close()
    r = r[r["rx"] < n]
    return r[np.lexsort((r["order"], r["rx"], r["ray"]))]


@pytest.mark.parametrize("kind,n", [("random", k) for k in (63, 64, 65, 97, 127, 128, 129, 255, 257, 1025, 4099)] +
                         [("grid", 64), ("grid", 700), ("grid", 4096), ("one", 64), ("one", 600), ("streets", 3000),
                          ("random", LINE)])
def test_device_tree_receives_what_the_host_tree_does(gpu_ctx, kind, n):
    sc, tx = scenes.shoebox(), np.array([[3.1, 4.2, 1.4]], np.float32)
    rx = _layout(kind, n, sc.verts.min(0), sc.verts.max(0))
    far = np.random.default_rng(1).uniform(1e3, 2e3, (LINE + 1 - n, 3)).astype(np.float32)
    scene = gpu_ctx.scene_from(sc)
    a = _records(gpu_ctx, scene, tx, rx, n)
    b = _records(gpu_ctx, scene, tx, np.concatenate([rx, far]), n)
    scene.close()
    assert len(a) >= n and len(a) == len(b)
    for f in ("tx", "rx", "ray", "order", "faces", "err", "dray"):
        assert np.array_equal(a[f], b[f]), f
