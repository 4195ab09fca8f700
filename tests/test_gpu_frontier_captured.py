"""A captured launch keeps its frontier when other containers of the context launch larger sets of
rays, and when its own container outgrows the room later; captured before there is any room, its
walks start at the root.  Replays give the records of an eager launch."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import api, scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


def _sorted(r):
    rows = np.ascontiguousarray(r).view(np.uint32).reshape(len(r), 16)[:, :14]
    return rows[np.lexsort(rows.T[::-1])]


@pytest.mark.parametrize("warm", [True, False])
def test_replay_after_larger_launches(warm):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = api.Context(0, stream=stream)
        sc, tx, rx = scenes.urban_canyon(blocks=10)
        scene, rxs = ctx.scene_from(sc), ctx.rx_upload(rx)
        n, kw = 560, dict(rx_angle_scale=SQ3, records_only=True)          # 3,136,002 rays
        one = torch.from_numpy(scenes.f32_exact(tx[:1])).float().cuda()
        three = torch.from_numpy(scenes.f32_exact(np.array([tx[0], [47.5, 102.5, 0.25], [200.0, 100.0, 90.0]]))).float().cuda()
        mine, other, eager = (ctx.paths_create(1 << 18, 64) for _ in range(3))
        ctx.launch(scene, three, rxs, mine, 8, 1, sync=True, **kw)        # room for three transmitters
        ctx.launch(scene, one, rxs, eager, n, 1, sync=True, **kw)
        want = _sorted(ctx.records(eager))
        ctx.launch(scene, one, rxs, mine, n, 1, sync=True, **(kw if warm else kw | dict(ray_range=(0, 1000))))
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            ctx.launch(scene, one, rxs, mine, n, 1, **kw)
        got = []
        for between in (None, other, mine):
            if between is not None:
                ctx.launch(scene, three, rxs, between, n, 1, sync=True, **kw)
                filler = torch.full((1 << 22,), -1, dtype=torch.int32, device="cuda")   # takes freed room
            graph.replay()
            torch.cuda.synchronize()
            got.append(_sorted(ctx.records(mine)))
        del graph
        for h in (eager, other, mine, rxs, scene):
            h.close()
        ctx.close()
    assert len(want) > 100
    for g in got:
        assert np.array_equal(g, want)
