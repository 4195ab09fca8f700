"""Transmitters on the device are read by the ray generation, or copied first where it cannot read them well:
from any address, any number of them, and from the host, a launch gets the same records."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import _binding as B
from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu


def _sorted(r):
    r["slot"] = 0
    return r[np.lexsort((r["order"], r["rx"], r["ray"], r["tx"]))].tobytes()


@pytest.mark.parametrize("shift", [0, 1, 2, 4, 6, 12])
def test_any_address(gpu_ctx, shift):
    sc, _, rx = scenes.shoebox_config()
    tx = scenes.f32_exact(np.random.default_rng(shift).uniform(0.5, 2.5, (5, 3))).astype(np.float32)
    scene, rxs, paths = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx), gpu_ctx.paths_create(1 << 14, 1 << 12)
    gpu_ctx.launch(scene, tx, rxs, paths, 24, 2, rx_angle_scale=3.0 ** 0.5, sync=True)
    want = _sorted(gpu_ctx.records(paths))
    buf = torch.zeros(64 + shift, dtype=torch.uint8, device="cuda")
    buf[shift:shift + 60] = torch.from_numpy(tx.view(np.uint8).reshape(-1)).cuda()
    prm = B.LaunchParams(24, 2, 3.0 ** 0.5, B.LAUNCH_SYNC, 0, None, 0, 0, 0, 0, 0, 0, 0)
    gpu_ctx._check(gpu_ctx.lib.sbr_launch(gpu_ctx.handle, scene.handle, ctypes.c_void_p(buf.data_ptr() + shift), 5,
                                          rxs.handle, ctypes.byref(prm), paths.handle))
    assert _sorted(gpu_ctx.records(paths)) == want
    for h in (paths, rxs, scene):
        h.close()


def test_many_transmitters(gpu_ctx):
    """16,384 are read by the ray generation, more are copied."""
    sc, _, rx = scenes.shoebox_config()
    scene, rxs, paths = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx), gpu_ctx.paths_create(1 << 20, 1 << 10)
    t = torch.rand(40_000, 3, device="cuda") * 2 + 0.5
    for n in (16384, 16385, 40000):
        got = []
        for x in (t[:n], t[:n].cpu().numpy()):
            gpu_ctx.launch(scene, x, rxs, paths, 2, 1, rx_angle_scale=3.0 ** 0.5, records_only=True, sync=True)
            got.append(_sorted(gpu_ctx.records(paths)))
        assert got[0] == got[1] and len(got[0]) > 64 * 1000
    for h in (paths, rxs, scene):
        h.close()
