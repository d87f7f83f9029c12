"""Gradients as visit lists: the second pass of fpo_render_backward and the
deferred form that fpo_adam_leaves takes, against the replay that adds every
row itself (large batches take it) and against each other."""

import numpy as np
import pytest

from paper_2202_08614_gb300 import fpo, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _rays(n, seed):
    rng = np.random.default_rng(seed)
    o = torch.as_tensor(rng.uniform(-0.6, 1.6, (n, 3)), dtype=torch.float32, device="cuda")
    d = torch.as_tensor(rng.uniform(0.2, 0.8, (n, 3)), dtype=torch.float32, device="cuda") - o
    t = torch.as_tensor(rng.uniform(0, 60, n), dtype=torch.float32, device="cuda")
    g = torch.as_tensor(rng.normal(size=(n, 3)), dtype=torch.float32, device="cuda")
    return o, d, t, g


def _close(a, b):
    # FP32 sums of at most 4000 visits of a leaf in another order: each within
    # 4000 * 2^-24 = 2.4e-4 of its sum of |terms| in the worst case, and within
    # a few sqrt(4000) * 2^-24 = 4e-6 of it as a random walk; terms of both
    # signs make that sum up to about ten times the largest element
    assert float((a - b).abs().max()) <= 1e-4 * float(b.abs().max())


@pytest.mark.parametrize("n1,n2", [(31, 5), (11, 5), (21, 5), (31, 11)])
@pytest.mark.parametrize("deep", [False, True])
def test_list_pass_equals_the_replays_own_adds(n1, n2, deep):
    # with 270,000 more rays of zero gradient the batch is beyond the list's
    # 2^18 rays, and the replay adds the rows of the 300
    tree = synth.random_tree(11, max_depth=5, n1=n1, n2=n2) if deep else synth.shell_tree(3, 5, n1, n2)
    r = fpo.Renderer(n1=n1, n2=n2, idft_mode="fused")
    r.upload(tree)
    o, d, t, g = _rays(300, n1 + n2)
    rgb = r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"]
    one = torch.zeros(tree.coeffs.shape, device="cuda")
    mark = torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda")
    r.render_backward(rgb, g, one, rays_o=o, rays_d=d, t_per_ray=t, leaf_mark=mark)
    many, mark2 = torch.zeros_like(one), torch.zeros_like(mark)
    rep = lambda x: x.repeat(901, *([1] * (x.dim() - 1))).contiguous()
    g2 = torch.zeros((300 * 901, 3), device="cuda")
    g2[:300] = g
    r.render_backward(rep(rgb), g2, many, rays_o=rep(o), rays_d=rep(d), t_per_ray=rep(t), leaf_mark=mark2)
    r.status()
    r.close()
    assert float(one.abs().max()) > 0 and torch.equal(mark, mark2)
    _close(many, one)


@pytest.mark.parametrize("parts", [20000, 40, 7])
def test_list_pass_at_every_share_of_a_warp(parts):
    # 20,000 rays' visits give a warp 32 entries at a time; those of 1, 500 or
    # 2858 rays fewer, down to the least, and leave most warps without any
    tree = synth.shell_tree(4)
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    n = 20000
    o, d, t, g = _rays(n, 5)
    rgb = r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"]
    whole, cut = (torch.zeros(tree.coeffs.shape, device="cuda") for _ in range(2))
    r.render_backward(rgb, g, whole, rays_o=o, rays_d=d, t_per_ray=t)
    step = -(-n // parts)
    for i in range(0, n, step):
        k = slice(i, min(i + step, n))
        r.render_backward(rgb[k].contiguous(), g[k].contiguous(), cut, rays_o=o[k].contiguous(),
                          rays_d=d[k].contiguous(), t_per_ray=t[k].contiguous())
    r.status()
    r.close()
    assert float(whole.abs().max()) > 0
    _close(cut, whole)


def _step(defer, calls, overflow=False):
    tree = synth.shell_tree(7)
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    p = torch.as_tensor(tree.coeffs, device="cuda")
    p, m, v, grad = p.clone(), torch.full_like(p, 1e-3), torch.full_like(p, 1e-4), torch.zeros_like(p)
    mark = torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda")
    if overflow:  # the list has the room of its first batch: 4096 rays, 32 visits each
        o, d, t, g = _rays(8, 1)
        rgb = r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"]
        r.render_backward(rgb, g * 0, grad, rays_o=o, rays_d=d, t_per_ray=t, leaf_mark=mark, defer=defer)
    for k in range(calls):
        o, d, t, g = _rays(4000, 20 + k)
        rgb = r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"]
        r.render_backward(rgb, g, grad, rays_o=o, rays_d=d, t_per_ray=t, leaf_mark=mark, defer=defer)
    r.adam_leaves(p, grad, m, v, mark, 5)
    rows = (p != torch.as_tensor(tree.coeffs, device="cuda")).any(1)
    img = r.render(camera=synth.shell_camera(64, 48), t=9.0)["rgb"].clone()
    r.set_coeffs(p)
    img2 = r.render(camera=synth.shell_camera(64, 48), t=9.0)["rgb"]
    r.status()
    r.close()
    assert not grad.any() and not mark.any() and torch.equal(img, img2)
    return p, m, v, rows


# one batch; three of which the list has room for the first (the others' rows go to
# grad); one beside a first, of zero gradient, that sized the list
@pytest.mark.parametrize("calls,overflow", [(1, False), (3, False), (1, True)])
def test_deferred_step_equals_the_dense_one(calls, overflow):
    a, b = _step(False, calls, overflow), _step(True, calls, overflow)
    assert torch.equal(a[3], b[3]) and int(a[3].sum()) > 1000
    for x, y in zip(a[:3], b[:3]):
        _close(x, y)


def test_set_coeffs_drops_a_pending_list():
    tree = synth.shell_tree(7)
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    p = torch.as_tensor(tree.coeffs, device="cuda").clone()
    m, v, grad = torch.zeros_like(p), torch.zeros_like(p), torch.zeros_like(p)
    mark = torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda")
    o, d, t, g = _rays(500, 3)
    rgb = r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"]
    r.render_backward(rgb, g, grad, rays_o=o, rays_d=d, t_per_ray=t, leaf_mark=mark, defer=True)
    r.set_coeffs(p)
    r.adam_leaves(p, grad, m, v, mark, 1)
    r.status()
    assert not m.any() and torch.equal(p, torch.as_tensor(tree.coeffs, device="cuda"))
    with pytest.raises(fpo.FPOError):  # needs the marks
        r.render_backward(rgb, g, grad, rays_o=o, rays_d=d, t_per_ray=t, defer=True)
    r.close()


@pytest.mark.parametrize("tensor_cores", [False, True])
def test_a_decoder_drops_a_pending_list(tensor_cores):
    from paper_2202_08614_gb300.latent import LatentModel

    tree = synth.shell_tree(7)
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    p = torch.as_tensor(tree.coeffs, device="cuda").clone()
    m, v, grad = torch.zeros_like(p), torch.zeros_like(p), torch.zeros_like(p)
    mark = torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda")
    o, d, t, g = _rays(500, 3)
    rgb = r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"]
    r.render_backward(rgb, g, grad, rays_o=o, rays_d=d, t_per_ray=t, leaf_mark=mark, defer=True)
    model = LatentModel(tree.n_leaves)
    r.set_coeffs_from_decoder(model._mlp(model.p), model.p["lat"], tensor_cores=tensor_cores)
    r.adam_leaves(p, grad, m, v, mark, 1)
    r.status()
    r.close()
    assert not m.any() and torch.equal(p, torch.as_tensor(tree.coeffs, device="cuda"))


def _coarse_tree():
    """A leaf of an eighth of the cube, in front of 32^3 finest cells."""
    k = np.arange(32 ** 3)
    xyz = np.concatenate([[[0, 0, 0]], 32 + np.stack([k % 32, k // 32 % 32, k // 1024], 1)]).astype(np.uint32)
    depth = np.array([1] + [6] * len(k), np.uint8)
    c = np.random.default_rng(7).normal(size=(len(depth), 166)).astype(np.float32) * 0.1
    c[:, 0] = np.where(depth == 1, 0.5, 20.0)
    return synth.Tree(depth, xyz, c, 6)


def _through_both(n, seed):
    rng = np.random.default_rng(seed)
    dev = lambda x: torch.as_tensor(x, dtype=torch.float32, device="cuda")
    o = rng.uniform(-0.6, -0.1, (n, 3))
    return dev(o), dev(rng.uniform(0.55, 0.75, (n, 3)) - o), dev(rng.uniform(0, 60, n)), dev(rng.normal(size=(n, 3)))


def _run(tree, batches, defer, times=None):
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    p0 = torch.as_tensor(tree.coeffs, device="cuda")
    p, m, v, grad = p0.clone(), torch.full_like(p0, 1e-3), torch.full_like(p0, 1e-4), torch.zeros_like(p0)
    mark = torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda")
    rgb = [r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"] for o, d, t, _ in batches]
    for k in range(1 if times is None else 5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for (o, d, t, g), y in zip(batches, rgb):
            r.render_backward(y, g, grad, rays_o=o, rays_d=d, t_per_ray=t, leaf_mark=mark, defer=defer)
        r.adam_leaves(p, grad, m, v, mark, 5)
        b.record()
        r.status()
        assert not grad.any() and not mark.any()
        if times is not None:
            times.append(a.elapsed_time(b))
    r.close()
    return p, m, v, (p != p0).any(1)


# several batches on one list (4096 rays fit), leaves with none to thousands of
# visits, and more rays than the tree has leaves (the rows go to grad)
@pytest.mark.parametrize("coarse,sizes", [(False, (1000, 1, 1500)), (False, (40, 40, 40)), (True, (1000, 1500)),
                                          (True, (20000,)), (False, (6000,)), (False, (2000, 6000))])
def test_deferred_batches_add_up(coarse, sizes):
    tree = _coarse_tree() if coarse else synth.shell_tree(7)
    batches = [(_through_both if coarse else _rays)(n, 50 + i) for i, n in enumerate(sizes)]
    a, b = _run(tree, batches, False), _run(tree, batches, True)
    assert torch.equal(a[3], b[3]) and int(a[3].sum()) > 100
    for x, y in zip(a[:3], b[:3]):
        _close(x, y)


def test_a_coarse_leaf_does_not_hold_up_the_step():
    # 30,000 visits of one leaf, summed one after another, took twenty times
    # what the dense step takes
    tree, batches = _coarse_tree(), [_through_both(30000, 9)]
    dense, deferred = [], []
    _run(tree, batches, False, dense)
    _run(tree, batches, True, deferred)
    assert min(deferred) <= 3.0 * min(dense)


def test_a_first_small_adjoint_allocates_nothing():
    tree = synth.shell_tree(7)

    def grads(n, r):
        o, d, t, g = _rays(n, 3)
        rgb = r.render(rays_o=o, rays_d=d, t_per_ray=t)["rgb"]
        grad = torch.zeros(tree.coeffs.shape, device="cuda")
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        r.render_backward(rgb, g, grad, rays_o=o, rays_d=d, t_per_ray=t)
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0], grad

    warm = fpo.Renderer(idft_mode="fused")  # (the kernels' code is loaded at their first launch)
    warm.upload(tree)
    grads(300, warm)
    warm.close()
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    used, a = grads(4096, r)
    assert used == 0
    more, _ = grads(8192, r)  # a list of its own, and then that one for fewer rays too
    assert more > 0
    used, b = grads(4096, r)
    assert used == 0
    r.upload(tree)  # back to the first room
    used, c = grads(4096, r)
    r.status()
    r.close()
    assert used == 0
    _close(b, a)
    _close(c, a)
