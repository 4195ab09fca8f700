"""Blocks that a captured call uses (directions, lattice tables, transmitters, pairs) outlive larger calls
on the same handles: nothing allocated by then is freed before the handles close, replays give the
records of the captured launch whatever ran between, and a launch at the captured division level takes
its blocks up again.  Everything is given back in the end."""
import gc

import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import api, scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


class Blocks:
    """The device blocks that the library holds."""

    def __init__(self, monkeypatch):
        self.live, self.freed, self.allocs = set(), [], 0
        alloc, free = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete

        def _alloc(*a):
            p = alloc(*a)
            self.live.add(p)
            self.allocs += 1
            return p

        def _free(p):
            self.live.discard(p)
            self.freed.append(p)
            return free(p)

        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", _alloc)
        monkeypatch.setattr(torch.cuda, "caching_allocator_delete", _free)


def _rows(ctx, paths):
    q = ctx.query(paths)
    keys = [q["faces"][:, j] for j in range(7, -1, -1)] + [q["order"], q["ray"], q["rx"], q["tx"]]
    return q[np.lexsort(tuple(keys))]


@pytest.mark.parametrize("launcher", [0, 8, 20])
def test_blocks_stay_for_replays(monkeypatch, launcher):
    blocks = Blocks(monkeypatch)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = api.Context(0, stream=stream)
        sc, tx, rx = scenes.random_clutter(nrx=6)
        rng = np.random.default_rng(3)
        many = torch.from_numpy(scenes.f32_exact(rng.uniform([1, 1, 1], [19, 15, 5], (7, 3)))).float().cuda()
        one = torch.from_numpy(scenes.f32_exact(tx[:1])).float().cuda()
        scene, rxs, few = ctx.scene_from(sc), ctx.rx_upload(rx), ctx.rx_upload(rx[:2])
        mine, other = ctx.paths_create(1 << 16, 1 << 14), ctx.paths_create(1 << 18, 1 << 16)

        def step(t, paths, n, r=rxs, **kw):
            ctx.launch(scene, t, r, paths, n, 2, rx_angle_scale=SQ3, launcher=launcher, **kw)
            ctx.refine(scene, paths, 6, 9)

        step(one, mine, 24)
        want = _rows(ctx, mine)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            step(one, mine, 24)
        ctx.launch(scene, one, few, mine, 24, 2, rx_angle_scale=SQ3, launcher=launcher)   # for its pairs
        ctx.refine_pair(scene, mine, 0, 1, 6)
        pair = torch.cuda.CUDAGraph()
        with torch.cuda.graph(pair, stream=stream, capture_error_mode="thread_local"):
            ctx.refine_pair(scene, mine, 0, 1, 6)
        torch.cuda.synchronize()
        captured = set(blocks.live)
        blocks.freed.clear()
        for paths, t, n in ((other, many, 57), (mine, many, 40), (other, many, 30)):
            step(t, paths, n)
            ctx.refine_pair(scene, paths, 3, 4, 6)
            ctx.launch(scene, t, rxs, paths, 9, 1, launcher=8 if launcher == 0 else 0)
        torch.cuda.synchronize()
        assert not captured & set(blocks.freed)   # before any replay: it would touch freed memory
        for paths, t, n in ((None, None, 0), (other, many, 57), (mine, many, 33)):
            if paths is not None:
                step(t, paths, n)
            graph.replay()
            torch.cuda.synchronize()
            assert _rows(ctx, mine).tobytes() == want.tobytes()
        # records of the replay's launch removed of double counts on this context: its own directions
        count = ctx.launch_stats(mine)["records"]
        step(one, mine, 24)
        step(one, mine, 57)
        held = len(blocks.live), blocks.allocs
        for n in (33, 24, 57, 24, 33, 57, 24):   # back and forth: no block made or given back
            step(one, mine, n)
        assert (len(blocks.live), blocks.allocs) == held and count == ctx.launch_stats(mine)["records"]
        assert _rows(ctx, mine).tobytes() == want.tobytes()
        graph.replay()
        torch.cuda.synchronize()
        assert _rows(ctx, mine).tobytes() == want.tobytes()
        del graph, pair
        gc.collect()
        for h in (mine, other, few, rxs, scene, ctx):
            h.close()
        torch.cuda.synchronize()
    assert len(want) > 20 and not blocks.live
