"""A batched refinement whose launches fail half way (made up on the host, in the checked build) leaves its
container's queue head and lists as they were then; the next call starts from clean ones, also when the
first of them is captured and never run."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import api, scenes

from parity_util import in_key_order

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


@pytest.mark.parametrize("lanes,below", [(16, 0.0), (1, 1e-2)])
@pytest.mark.parametrize("fail", [1, 2, 3, 4, 5])
def test_next_call_is_whole(monkeypatch, lanes, below, fail):
    ctx = api.Context(0, stream=torch.cuda.Stream(), checked=True)
    sc, tx, rx = scenes.shoebox_config()
    scene, rxs = ctx.scene_from(sc), ctx.rx_upload(rx)
    # room for the many-path form: five launches
    paths, own = ctx.paths_create(1 << 16, 1 << 14), ctx.paths_create(1 << 16, 1 << 14)

    def refine(p):
        ctx.batch_refine(scene, p, 8, 9, lanes_per_path=lanes, fp64_below=below)

    def refined(p):
        ctx.launch(scene, tx, rxs, p, 32, 3, rx_angle_scale=SQ3, sync=True)
        refine(p)
        return in_key_order(ctx.query(p))[0]

    want = refined(own)
    assert len(want) > 20 and np.sum(want["valid"]) > 0
    for captured in (False, True):
        ctx.launch(scene, tx, rxs, paths, 32, 3, rx_angle_scale=SQ3, sync=True)
        monkeypatch.setenv("SBR_CHECKED_FAIL_LAUNCH", str(fail))
        with pytest.raises(api.SbrError):
            refine(paths)
        monkeypatch.delenv("SBR_CHECKED_FAIL_LAUNCH")
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=ctx.stream):
                refine(paths)
        assert refined(paths).tobytes() == want.tobytes()
        if captured:   # the captured call on a container that is clean by now
            ctx.launch(scene, tx, rxs, paths, 32, 3, rx_angle_scale=SQ3, sync=True)
            g.replay()
            torch.cuda.synchronize()
            assert in_key_order(ctx.query(paths))[0].tobytes() == want.tobytes()
    for h in (paths, own, rxs, scene):
        h.close()
    ctx.close()
