"""Before its exact test a diffraction reception passes a filter in the frame of the edge, which may let none go
that the test accepts.  The checked build tests what the filter rejects as well and reports the first
that it should have kept: transmitters and receivers close to an edge's line, where the frame loses digits,
near the origin and a kilometre from it."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import api, scenes

pytestmark = pytest.mark.gpu


TURN = np.array([[0.8, -0.6, 0.0], [0.6, 0.8, 0.0], [0.0, 0.0, 1.0]])   # edges off the axes


def _wall(at, length):
    """A thin wall (a closed box of 12 triangles, 6 faces)."""
    v = np.array([[i * length, j * 0.3, k * 4.0] for i in (0, 1) for j in (0, 1) for k in (0, 1)]) @ TURN.T + at
    quads = [(0, 1, 3, 2), (4, 6, 7, 5), (0, 4, 5, 1), (2, 3, 7, 6), (0, 2, 6, 4), (1, 5, 7, 3)]
    tris = np.array([t for a, b, c, d in quads for t in ((a, b, c), (a, c, d))])
    return v.astype(np.float32), tris, np.repeat(np.arange(6), 2)


@pytest.mark.parametrize("at,length", [((2.0, 3.0, 0.0), 6.0), ((903.1, 850.7, 20.0), 30.0)])
@pytest.mark.parametrize("near", [0.02, 0.3, 3.0])
def test_filter_keeps_what_the_test_accepts(at, length, near):
    ctx = api.Context(0, checked=True)
    scene = ctx.scene_upload(*_wall(at, length))
    rng = np.random.default_rng(int(1000 * near) + int(length))

    def beside(count):   # around the edge along the wall's top, above it or before its face
        a, r = rng.uniform(0, np.pi, count), near * 10 ** rng.uniform(-1, 0, count)
        p = np.stack([length * rng.uniform(-1, 2, count), -r * np.sin(a), 4.0 + r * np.cos(a)], 1)
        return scenes.f32_exact(p @ TURN.T + at)

    tx, rx = beside(6), beside(4096)
    rxs, paths = ctx.rx_upload(rx), ctx.paths_create(1 << 24, 1 << 10)
    ctx.launch(scene, tx, rxs, paths, 1000, 0, rx_angle_scale=3.0 ** 0.5, diffraction=True, records_only=True, sync=True)
    st = ctx.launch_stats(paths)
    for h in (paths, rxs, scene, ctx):
        h.close()
    assert st["diffraction_candidates"] > 100 and st["diffraction_records"] > 1000
    assert st["check_flags"] == 0
