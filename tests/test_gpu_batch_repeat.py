"""The batched refinement leaves its queue head, group sizes and cursors zero for the next call: calls
in a row on one container, with none, few and many paths, with and without FP64 iterations, give
the results of a container of their own."""
import numpy as np
import pytest

from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu
SQ3 = float(np.sqrt(3.0))


@pytest.mark.parametrize("lanes", [1, 16])
def test_calls_in_a_row_equal_fresh_containers(gpu_ctx, lanes):
    sc, tx, rx = scenes.office(nbox=40, ntx=3, nrx=300, g_shell=6, g_box=1)
    scene = gpu_ctx.scene_from(sc)
    far = gpu_ctx.rx_upload(np.array([[500.0, 500.0, 2.0]], np.float32))   # outside: no path
    sets = [gpu_ctx.rx_upload(rx[:k]) for k in (1, 300)]
    shared = gpu_ctx.paths_create(1 << 20, 1 << 18)

    def refined(paths, rxs, n, iters, below):
        gpu_ctx.launch(scene, tx, rxs, paths, n, 4, rx_angle_scale=SQ3, sync=True)
        gpu_ctx.batch_refine(scene, paths, iters, 9, target=1.7e-4, lanes_per_path=lanes, fp64_below=below)
        q = gpu_ctx.query(paths)
        return q[np.lexsort((q["faces"][:, 1], q["faces"][:, 0], q["order"], q["ray"], q["rx"], q["tx"]))]

    counts = []
    for rxs, n, iters, below in ((sets[0], 48, 6, 0.0), (far, 16, 6, 0.0), (sets[1], 96, 6, 0.0), (sets[0], 48, 12, 1e-2),
                                 (sets[1], 96, 0, 0.0), (sets[1], 96, 12, 1e-2), (far, 16, 6, 0.0), (sets[0], 24, 6, 0.0)):
        own = gpu_ctx.paths_create(1 << 20, 1 << 18)
        want, got = refined(own, rxs, n, iters, below), refined(shared, rxs, n, iters, below)
        again = None
        if len(got):   # and twice on the same paths: the second call starts from refined ones
            for p in (own, shared):
                gpu_ctx.batch_refine(scene, p, iters, 9, target=1.7e-4, lanes_per_path=lanes, fp64_below=below)
            again = [np.sort(gpu_ctx.query(p)["err"]) for p in (own, shared)]
        assert got.tobytes() == want.tobytes()
        assert again is None or np.array_equal(*again)
        counts.append(len(got))
        own.close()
    assert min(counts) == 0 and max(counts) > 16 * 32 * gpu_ctx.num_sms   # past the many-path line
    for h in (shared, far, scene, *sets):
        h.close()
