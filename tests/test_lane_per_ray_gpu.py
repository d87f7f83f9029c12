"""The fused mode's two ways, a warp evaluating its visits together and one lane
a ray (large calls on small trees, whole images), against each other, and the
adjoint of batches larger than its list against that of their parts."""

import numpy as np
import pytest

from paper_2202_08614_gb300 import fpo, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

LANES = 1 << 17  # rays from which a tree of fewer than 4096 leaves takes one lane a ray
ASKED = 3 << 16  # ... and from which explicit rays on one of up to 2^17 leaves do, if they are coherent


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _rays(n, seed):
    rng = np.random.default_rng(seed)
    dev = lambda x: torch.as_tensor(x, dtype=torch.float32, device="cuda")
    o = rng.uniform(-0.6, 1.6, (n, 3))
    return dev(o), dev(rng.uniform(0.2, 0.8, (n, 3)) - o), dev(rng.uniform(0, 60, n)), dev(rng.normal(size=(n, 3)))


def _close_grad(a, b, visits):
    # FP32 sums of up to `visits` visits a leaf in another order, as a random walk
    # of roundings: sqrt(visits) * 2^-24 of a sum of |terms| that is up to some
    # ten times the largest element
    tol = 40 * visits ** 0.5 * 2.0 ** -24
    assert float(b.abs().max()) > 0 and float((a - b).abs().max()) <= tol * float(b.abs().max())


def _tree(kind, n1, n2):
    if kind == "octree":
        return synth.random_tree(11, max_depth=5, n1=n1, n2=n2)
    t = synth.shell_tree(4, 5, n1, n2)  # every other leaf
    return synth.Tree(t.leaf_depth[::2].copy(), t.leaf_xyz[::2].copy(), t.coeffs[::2].copy(), t.max_depth, n1, n2)


@pytest.mark.parametrize("n1,n2", [(31, 5), (11, 5), (21, 5), (31, 11)])
@pytest.mark.parametrize("kind", ["bricks", "octree"])
@pytest.mark.parametrize("own", [True, False])
def test_lanes_equal_warps(n1, n2, kind, own):
    tree = _tree(kind, n1, n2)
    assert tree.n_leaves < 4096
    r = fpo.Renderer(n1=n1, n2=n2, idft_mode="fused")
    r.upload(tree)
    n = LANES + 33
    o, d, t, g = _rays(n, n1 + n2)
    d[:9] = torch.eye(3, device="cuda").repeat(3, 1)  # axis-parallel
    args = lambda s: dict(rays_o=o[s], rays_d=d[s], t_per_ray=t[s] if own else None, t=7.0)
    whole = slice(0, n)
    stats = [torch.zeros(3, dtype=torch.int64, device="cuda") for _ in range(2)]
    marks = [torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda") for _ in range(4)]
    a = r.render(**args(whole), visit_cap=96, want_T=True, leaf_mark=marks[0], stats=stats[0])
    plain = r.render(**args(whole))["rgb"]
    assert torch.equal(plain, a["rgb"])
    ga, gb = (torch.zeros(tree.coeffs.shape, device="cuda") for _ in range(2))
    r.render_backward(a["rgb"], g, ga, **args(whole), leaf_mark=marks[2])
    cuts = [0, 1, n // 2, n - 31, n]
    for lo, hi in zip(cuts[:-1], cuts[1:]):
        s = slice(lo, hi)
        b = r.render(**args(s), visit_cap=96, want_T=True, leaf_mark=marks[1], stats=stats[1])
        # the same walk; sums of n1 and 27 n2 products in another order, and their
        # sigmoids and exponentials along at most 96 visits
        assert float((a["rgb"][s] - b["rgb"]).abs().max()) <= 2e-5
        assert float((a["T"][s] - b["T"]).abs().max()) <= 2e-5
        # (a transmittance at stop_T to within that may stop a visit apart)
        same = (a["visit_count"][s] == b["visit_count"]) & (a["visit_log"][s] == b["visit_log"]).all(1)
        assert int((~same).sum()) <= 3 + n // 20000
        r.render_backward(b["rgb"], g[s].contiguous(), gb, **args(s), leaf_mark=marks[3])
    r.status()
    r.close()
    assert torch.equal(stats[0][2:], stats[1][2:]) and int(stats[0][1]) > n
    assert int((marks[0] != marks[1]).sum()) <= 1 and int((marks[2] != marks[3]).sum()) <= 1
    assert torch.equal(marks[0], marks[2])
    _close_grad(ga, gb, 4 * n / tree.n_leaves + 1000)


@pytest.mark.parametrize("own", [True, False])
@pytest.mark.parametrize("n", [ASKED - 1, ASKED, (1 << 18) + 41])
def test_large_calls_look_at_their_rays(n, own):
    # an image's rays go by lanes from ASKED on (their adjoint, from more than one
    # list holds on), a random batch by warps; both as parts of them by warps, the
    # latter in the same bits
    tree = synth.shell_tree(6)
    assert tree.n_leaves >= 4096
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    cam = synth.shell_camera(640, 480)
    image = _camera_rows(cam, 0, 480)
    o, d, t, g = _rays(n, 3)
    for coherent, (o, d) in ((True, (image["rays_o"][:n], image["rays_d"][:n])), (False, (o, d))):
        args = lambda s: dict(rays_o=o[s], rays_d=d[s], t_per_ray=t[s] if own else None, t=7.0)
        a = r.render(**args(slice(0, n)))["rgb"]
        b = torch.cat([r.render(**args(s))["rgb"] for s in (slice(0, n // 2), slice(n // 2, n))])
        assert float((a - b).abs().max()) <= 2e-5
        assert torch.equal(a, b) == (not coherent or n < ASKED)
        log = r.render(**args(slice(0, n)), visit_cap=64, want_T=True)
        assert torch.equal(log["rgb"], a)
        ga, gb = (torch.zeros(tree.coeffs.shape, device="cuda") for _ in range(2))
        r.render_backward(a, g, ga, **args(slice(0, n)))
        mark = torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda")
        for s in (slice(0, n // 2), slice(n // 2, n)):
            r.render_backward(b[s], g[s], gb, **args(s), leaf_mark=mark)
        assert mark.any() and float(ga[mark == 0].abs().sum()) == 0.0
        _close_grad(ga, gb, 4 * n / tree.n_leaves + 1000)
    r.status()
    r.close()


def _camera_rows(cam, y0, y1):
    """Rows y0 .. y1 of a camera as explicit rays."""
    from test_grad_gpu import camera_rays

    o, d = camera_rays(cam)
    s = slice(y0 * cam.width, y1 * cam.width)
    dev = lambda x: torch.as_tensor(x[s], dtype=torch.float32, device="cuda")
    return dict(rays_o=dev(o), rays_d=dev(d))


@pytest.mark.parametrize("w,h", [(512, 257), (1, 131072), (32769, 4)])
def test_lanes_of_a_camera_frame(w, h):
    tree = synth.shell_tree(6)
    cam = synth.shell_camera(w, h)
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    img = r.render(camera=cam, t=11.0)["rgb"]
    table = fpo.Renderer()
    table.upload(tree)
    assert float((img - table.render(camera=cam, t=11.0)["rgb"]).abs().max()) <= 2e-5
    g = torch.randn(img.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    a, b = (torch.zeros(tree.coeffs.shape, device="cuda") for _ in range(2))
    r.render_backward(img, g, a, camera=cam, t=11.0)
    for y in range(0, h, max(1, h // 3)):
        y1 = min(h, y + max(1, h // 3))
        s = slice(y * w, y1 * w)
        r.render_backward(img[s].contiguous(), g[s].contiguous(), b, t=11.0, **_camera_rows(cam, y, y1))
    r.status()
    r.close()
    table.close()
    # (the explicit rays are rounded from the camera's FP64 frame: 2^-24 of a
    # coordinate moves a segment's ends by as much of a cell)
    assert float(a.abs().max()) > 0 and float((a - b).abs().max()) <= 2e-3 * float(a.abs().max())


@pytest.fixture(scope="module")
def big():
    """A tree of 2^17 leaves and more: batches past the list's 2^18 rays go in parts."""
    k = np.arange(52 ** 3)
    xyz = (6 + np.stack([k % 52, k // 52 % 52, k // 52 ** 2], 1)).astype(np.uint32)
    rng = np.random.default_rng(2)
    c = rng.normal(size=(len(xyz), 146)).astype(np.float32) * 0.1
    c[:, 0] = 10.0
    tree = synth.Tree(np.full(len(xyz), 6, np.uint8), xyz, c, 6, 11, 5)
    r = fpo.Renderer(n1=11, n2=5, idft_mode="fused")
    r.upload(tree)
    yield tree, r
    r.close()


@pytest.mark.parametrize("n", [(1 << 18) + 1, 500_001])
def test_large_batches_in_parts(big, n):
    tree, r = big
    o, d, t, g = _rays(n, 9)
    rgb = r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"]
    a, b = (torch.zeros(tree.coeffs.shape, device="cuda") for _ in range(2))
    ma, mb = (torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda") for _ in range(2))
    r.render_backward(rgb, g, a, rays_o=o, rays_d=d, t_per_ray=t, leaf_mark=ma, defer=True)
    for at in range(0, n, 100_000):
        s = slice(at, min(n, at + 100_000))
        r.render_backward(rgb[s].contiguous(), g[s].contiguous(), b, rays_o=o[s], rays_d=d[s], t_per_ray=t[s], leaf_mark=mb)
    r.status()
    assert torch.equal(ma, mb)
    _close_grad(a, b, 60 * n / tree.n_leaves + 500)


# (a row of tiles of the last is more than the list holds: no parts)
@pytest.mark.parametrize("w,h,fov", [(640, 480, 40.0), (333, 1001, 40.0), (40000, 7, 0.01)])
def test_camera_adjoint_in_parts(big, w, h, fov):
    tree, r = big
    cam = synth.Camera(eye=(2.2, 0.7, 0.9), width=w, height=h, fov_y_deg=fov)
    img = r.render(camera=cam, t=5.0)["rgb"]
    g = torch.randn(img.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    a = torch.zeros(tree.coeffs.shape, device="cuda")
    r.render_backward(img, g, a, camera=cam, t=5.0)
    # the FP64 replay takes the frame whole
    b64 = torch.zeros(tree.coeffs.shape, dtype=torch.float64, device="cuda")
    r.render_backward(img, g, b64, camera=cam, t=5.0, fp64=True)
    r.status()
    assert float(b64.abs().max()) > 0
    # norm-wise, as the FP32 adjoint against the oracle's
    assert float((a.double() - b64).norm() / b64.norm()) <= 2e-4
