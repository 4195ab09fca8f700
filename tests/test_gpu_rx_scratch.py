"""An upload whose allocator has no room for the device build's scratch builds the receivers' tree on the host
instead: the same reception records, and nothing but the set's own block stays."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import api, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [129, 1000])
def test_upload_without_scratch(monkeypatch, n):
    live, refused = set(), []
    alloc, free = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete

    def _alloc(size, *a):
        if size == 96 * n and refused:
            refused.append(size)
            raise torch.cuda.OutOfMemoryError
        p = alloc(size, *a)
        live.add(p)
        return p

    def _free(p):
        live.discard(p)
        return free(p)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", _alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", _free)
    ctx = api.Context(0)
    sc, tx, _ = scenes.shoebox_config()
    rx = scenes.f32_exact(np.random.default_rng(n).uniform([0.4, 0.4, 0.4], [9.6, 7.6, 2.6], (n, 3)))
    scene, res = ctx.scene_from(sc), []
    for _ in range(2):
        before = len(live)
        rxs = ctx.rx_upload(rx)
        assert len(live) == before + 1
        paths = ctx.paths_create(1 << 20, 1 << 10)
        ctx.launch(scene, tx, rxs, paths, 24, 2, rx_angle_scale=3.0 ** 0.5, records_only=True, sync=True)
        r = ctx.records(paths)
        res.append(r[np.lexsort((r["order"], r["rx"], r["ray"]))])
        paths.close()
        rxs.close()
        refused.append(0)   # from the second upload on
    assert refused == [0, 96 * n, 0]
    assert len(res[0]) > n and res[0].tobytes() == res[1].tobytes()
    scene.close()
    ctx.close()
    assert not live
