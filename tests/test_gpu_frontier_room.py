"""The room for the first segments' lists is one block of a container: launches that need more replace
it, and only a block that a captured launch uses stays beside its successor."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import api, scenes

pytestmark = pytest.mark.gpu


def test_outgrown_lists_are_given_back(monkeypatch):
    live = set()
    alloc, free = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete

    def _alloc(*a):
        p = alloc(*a)
        live.add(p)
        return p

    def _free(p):
        live.discard(p)
        return free(p)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", _alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", _free)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = api.Context(0, stream=stream)
        sc, tx, rx = scenes.urban_canyon(blocks=10)
        scene, rxs = ctx.scene_from(sc), ctx.rx_upload(rx)
        paths = ctx.paths_create(1 << 18, 64)
        t = torch.from_numpy(scenes.f32_exact(np.repeat(tx[:1], 6, 0))).float().cuda()

        def launch(k):
            ctx.launch(scene, t[:k], rxs, paths, 560, 1, rx_angle_scale=3.0 ** 0.5, records_only=True)
            torch.cuda.synchronize()
            return len(live)

        counts = [launch(k) for k in (1, 2, 3, 5, 2)]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            ctx.launch(scene, t[:2], rxs, paths, 560, 1, rx_angle_scale=3.0 ** 0.5, records_only=True)
        after = launch(6)
        del graph
        for h in (paths, rxs, scene, ctx):
            h.close()
        torch.cuda.synchronize()
    assert len(set(counts)) == 1, counts
    assert after == counts[0] + 2   # the captured launch's lists and transmitters
    assert not live
