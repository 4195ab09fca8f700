"""A container that holds a launch's records but not the diffraction receptions that wait for their occlusion
queries: the launch reports an overflow and later calls see the records that were written, nothing else of
the record array."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import api, scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


def _set(r):
    r = r.copy()
    r["slot"] = 0
    return sorted(x.tobytes() for x in r)


@pytest.mark.parametrize("many", [20, 60])
def test_only_written_records_are_seen(gpu_ctx, many):
    sc, tx, rx = scenes.urban_canyon(blocks=6)
    rx = scenes.jitter(np.random.default_rng(many), np.repeat(rx, many, 0), 1.0)   # many receptions a candidate
    scene, rxs = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx)
    kw = dict(rx_angle_scale=SQ3, diffraction=True)
    big = gpu_ctx.paths_create(1 << 21, 1 << 16)
    gpu_ctx.launch(scene, tx, rxs, big, 96, 2, sync=True, **kw)
    st = gpu_ctx.launch_stats(big)
    want, diffracted = _set(gpu_ctx.records(big)), st["diffraction_records"]
    trace = st["records"] - diffracted
    cap = max(int(st["diffraction_candidates"] / 1.25) + 1, trace + 100)   # room for the candidates
    assert diffracted > 100 and trace > 10
    torch.full((1 << 22,), -1, dtype=torch.int32, device="cuda")   # what the container's memory held before
    small = gpu_ctx.paths_create(cap, 1 << 16)
    gpu_ctx.launch(scene, tx, rxs, small, 96, 2, **kw)
    st = gpu_ctx.launch_stats(small)
    assert st["records"] > cap and st["diffraction_candidates"] <= st["candidate_cap"]
    got = _set(gpu_ctx.records(small))
    assert trace <= len(got) <= cap and set(got) <= set(want) and len(set(got)) == len(got)
    assert len(got) == trace + st["diffraction_records"]
    gpu_ctx.refine(scene, small, 4, 9)
    q = gpu_ctx.query(small)
    assert 0 < len(q) <= len(got) and np.all((q["tx"] == 0) & (q["rx"] >= 0) & (q["rx"] < len(rx)))
    assert st["paths"] == len(q) and st["collisions"] == 0
    with pytest.raises(api.SbrError) as e:
        gpu_ctx.launch(scene, tx, rxs, small, 96, 2, sync=True, **kw)
    assert e.value.status == 5
    # records put in place of the launch's are complete
    again = np.frombuffer(b"".join(got), gpu_ctx.records(small).dtype)
    gpu_ctx.records_dedup(small, again)
    assert gpu_ctx.launch_stats(small)["records"] == len(got) and gpu_ctx.paths_count(small) == len(q)
    for h in (small, big, rxs, scene):
        h.close()
