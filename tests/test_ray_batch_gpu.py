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


def test_other_bases_as_torch_takes_them():
    from paper_2202_08614_gb300.finetune import camera_basis, camera_ray_batch

    cams = synth.ring_cameras(4, 33, 21, fov_y_deg=37.0)
    gen = lambda: torch.Generator(device="cuda").manual_seed(3)
    base = camera_basis(cams)
    draw = lambda b: camera_ray_batch(cams, 777, gen(), basis=b)
    o, d, t = draw(base)
    # wider, longer or strided: the same rows, the same bits
    wide = torch.cat([base, torch.full((4, 5), torch.nan, device="cuda")], 1)
    long = torch.cat([base, torch.full((3, 12), torch.nan, device="cuda")])
    for b in (wide, long, base.t().contiguous().t()):
        assert all(torch.equal(x, y) for x, y in zip(draw(b), (o, d, t)))
    # other types keep their precision; float64 differs by the float32 rounding
    # of a dozen operations, float16 by that of its inputs (2^-11 each)
    o8, d8, t8 = draw(base.double())
    assert o8.dtype == d8.dtype == torch.float64 and torch.equal(t8, t)
    assert torch.equal(o8, o.double()) and float((d8 - d).abs().max()) <= 16 * 2.0 ** -24
    oh, dh, _ = draw(base.half())
    assert oh.dtype == torch.float16 and dh.dtype == torch.float32 and float((dh - d).abs().max()) <= 8 * 2.0 ** -11
    # gradients reach a basis that asks for them
    leaf = base.clone().requires_grad_()
    og, dg, _ = draw(leaf)
    (og.sum() + dg[:, 0].sum()).backward()
    assert leaf.grad is not None and float(leaf.grad.abs().max()) > 0
    assert float((dg.detach() - d).abs().max()) <= 16 * 2.0 ** -24
    # any field of view, as before
    for c in cams:
        c.fov_y_deg = 0.0
    _, d0, _ = draw(base)
    assert torch.isfinite(d0).all()
    with torch.no_grad():
        assert torch.equal(draw(leaf)[1], d0)
