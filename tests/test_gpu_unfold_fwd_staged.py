"""The forward map's staged form (bulk copies of whole 32-path chunks into shared memory, the
ragged last chunk from global memory) gives, path for path, the bits of the direct form, which
runs when an input array is not 16-byte aligned or the batch is small; an output buffer that is
not 16-byte aligned gets the same values."""
import numpy as np
import pytest
import torch

from paper_2208_10009_gb300 import scenes

pytestmark = pytest.mark.gpu


def _shifted(t):
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    u = flat[1:].view(t.shape)
    u.copy_(t)
    assert u.data_ptr() % 16 == 4
    return u


@pytest.mark.parametrize("extra", [-1, 0, 1, 31, 32 * 152 * 40 + 5])
def test_staged_forward_equals_direct(gpu_ctx, extra):
    sc, _, _ = scenes.urban_canyon()
    scene = gpu_ctx.scene_from(sc)
    n = 32 * 16 * gpu_ctx.num_sms + extra   # around the size from which the staged form runs
    rng = np.random.default_rng(n)
    dev = "cuda"
    T, R = (torch.tensor(rng.uniform(0, 1000, (n, 3)), dtype=torch.float32, device=dev) for _ in range(2))
    AE = torch.tensor(np.stack([rng.uniform(-np.pi, np.pi, n), rng.uniform(-1.2, 1.2, n)], -1), dtype=torch.float32,
                      device=dev)
    faces = rng.integers(0, sc.nf, (n, 8)).astype(np.int32)
    order = rng.integers(0, 9, n).astype(np.int32)
    order[:4] = [0, 8, 12, -3]              # clamped to [0, 8]
    faces[7, 0], order[7] = sc.nf, 1        # ids out of range: NaN outputs
    faces[8, 5], order[8] = -1, 6
    faces[9, 5], order[9] = -1, 5           # past the order: not looked at
    F, O = torch.tensor(faces, device=dev), torch.tensor(order, device=dev)
    got = gpu_ctx.unfold_fwd(scene, T, R, AE, F, O)
    direct = gpu_ctx.unfold_fwd(scene, _shifted(T), R, AE, F, O)
    shifted = gpu_ctx.unfold_fwd(scene, T, R, AE, F, O, out=_shifted(torch.empty_like(got)))
    got, direct, shifted = (x.cpu().numpy() for x in (got, direct, shifted))
    assert np.array_equal(got, direct, equal_nan=True) and np.array_equal(got, shifted, equal_nan=True)
    assert np.isnan(got[7:9]).all() and np.isfinite(np.delete(got, [7, 8], 0)).all()
    scene.close()
