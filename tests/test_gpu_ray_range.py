"""Ray ranges (SBR_LAUNCH_RAY_RANGE) are taken in the schedule's order, whole faces at a time with
the ids outside the range passed over: the segments and records of any range have to be those of
the same range traced in id order, and of a range's part of the whole launch."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


def _ranges(n, launcher, rng):
    """The empty, whole and single-ray ranges, cuts at the vertex, edge and face blocks' borders
    and inside them, and random ones."""
    N = (4 if launcher == 8 else 10) * n * n + 2
    E = 12 + 30 * (n - 1)
    per = max((n - 1) * (n - 2) // 2, 1)
    marks = [0, 1, 11, 12, E - 1, E, E + 1, E + per - 1, E + per, E + per + 1, E + 7 * per + per // 2, N - 1, N]
    marks = sorted({min(max(m, 0), N) for m in marks})
    pairs = list(zip(marks[:-1], marks[1:])) + [(0, N), (5 % N, 5 % N), (0, N - 1), (1, N), (N - 1, N)]
    pairs += [(min(E + per // 3, N), min(E + 3 * per + per // 2, N))]
    for _ in range(4):
        a, b = sorted(rng.integers(0, N + 1, 2))
        pairs.append((int(a), int(b)))
    return N, pairs


@pytest.mark.parametrize("n,ntx,launcher", [(1, 1, 0), (2, 2, 0), (3, 1, 0), (4, 1, 0), (7, 3, 0), (24, 2, 0), (31, 5, 0),
                                            (9, 2, 8), (10, 1, 20)])
def test_range_equals_id_order(gpu_ctx, n, ntx, launcher):
    sc = scenes.shoebox()
    rng = np.random.default_rng(n)
    tx = scenes.f32_exact(rng.uniform([0.5, 0.5, 0.5], [9.5, 7.5, 2.5], (ntx, 3)))
    rx = scenes.f32_exact(rng.uniform([0.5, 0.5, 0.5], [9.5, 7.5, 2.5], (6, 3)))
    scene, rxs, paths = gpu_ctx.scene_from(sc), gpu_ctx.rx_upload(rx), gpu_ctx.paths_create(1 << 18, 1 << 16)

    def records(**kw):
        gpu_ctx.launch(scene, tx, rxs, paths, n, 2, rx_angle_scale=SQ3, launcher=launcher, records_only=True, sync=True,
                       **kw)
        st = gpu_ctx.launch_stats(paths)
        r = gpu_ctx.records(paths)
        r = r[np.lexsort((r["order"], r["rx"], r["ray"], r["tx"]))]
        return st["rays"], st["segments"], r

    N, pairs = _ranges(n, launcher, rng)
    whole = records()
    assert whole[0] == ntx * N
    for a, b in pairs:
        got, want = records(ray_range=(a, b)), records(ray_range=(a, b), id_order=True)
        assert got[0] == want[0] == ntx * (b - a) and got[1] == want[1]
        assert got[2].tobytes() == want[2].tobytes(), (a, b)
        part = whole[2][(whole[2]["ray"] >= a) & (whole[2]["ray"] < b)]
        assert got[2].tobytes() == part.tobytes(), (a, b)
    for h in (paths, rxs, scene):
        h.close()
