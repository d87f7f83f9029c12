"""Training rays (fpo_camera_ray_batch) against the same formula in plain torch."""

import numpy as np
import pytest

from paper_2202_08614_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("n,size", [(1, (5, 3)), (255, (1, 1)), (4097, (800, 800)), (0, (8, 8))])
def test_ray_batch_matches_torch(n, size):
    from paper_2202_08614_gb300.finetune import camera_basis, camera_ray_batch

    cams = synth.ring_cameras(5, *size, fov_y_deg=37.0)
    gen = lambda: torch.Generator(device="cuda").manual_seed(n)
    o, d, t = camera_ray_batch(cams, n, gen(), n_frames=60)
    g, (W, H) = gen(), size
    v, p, f = (torch.randint(0, k, (n,), device="cuda", generator=g) for k in (5, W * H, 60))
    b = camera_basis(cams)[v]
    th = np.tan(np.radians(37.0) / 2)
    sx = ((2 * ((p % W).float() + 0.5) / W - 1) * th * W / H)[:, None]
    sy = ((1 - 2 * ((p // W).float() + 0.5) / H) * th)[:, None]
    e = b[:, 3:6] + sx * b[:, 6:9] + sy * b[:, 9:12]
    assert o.shape == d.shape == (n, 3) and torch.equal(o, b[:, :3]) and torch.equal(t, f.float())
    # the same operations in the same order: equal, or a few units in the last
    # place where torch contracts or reorders one of them
    assert n == 0 or float((d - e / e.norm(dim=1, keepdim=True)).abs().max()) <= 4 * 2.0 ** -24
