"""The brick index of trees whose leaves are all finest cells against the octree
descent: the compaction schedule walks the octree for every tree, so the two
must give the same visits and the same bits."""

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


def _uniform_tree(depth, seed, n1=31, n2=5, block=0):
    """Finest cells in clumps of 1, 2, 4 and 8 cells a side and single ones, in
    shuffled upload order: partly filled bricks, bricks in every corner of a
    block, empty cubes of every size.  block: a full cube of that side besides,
    for trees with the leaves that the index of a deep grid asks for."""
    rng = np.random.default_rng(seed)
    g = 1 << depth
    cells = {(0, 0, 0), (g - 1, g - 1, g - 1), (g - 1, 0, 0), (0, g - 1, 3)}
    for s in (1, 1, 2, 2, 4, 8):
        for lo in rng.integers(0, max(1, g - s + 1), (12 if s < 8 else 3, 3)):
            cells |= {(int(lo[0]) + i, int(lo[1]) + j, int(lo[2]) + k)
                      for i in range(s) for j in range(s) for k in range(s) if rng.random() < 0.8}
    xyz = np.array(sorted(cells), np.uint32)
    if block:
        lo, k = g // 2 - 7, np.arange(block ** 3)
        cube = lo + np.stack([k % block, k // block % block, k // block ** 2], 1).astype(np.uint32)
        xyz = np.concatenate([xyz[((xyz < lo) | (xyz >= lo + block)).any(1)], cube.astype(np.uint32)])
    xyz = xyz[rng.permutation(len(xyz))]
    coeffs = synth.draw_coefficients(rng, len(xyz), n1, n2)
    return synth.Tree(np.full(len(xyz), depth, np.uint8), xyz, coeffs, depth, n1, n2)


# 4: the smallest grid the index serves; 3 and 12, and 9 and 11 with so few leaves, walk the octree both times
@pytest.mark.parametrize("depth", [3, 4, 5, 6, 9, 11, 12])
def test_brick_walk_equals_octree_descent(depth):
    _same_walk(_uniform_tree(depth, 40 + depth), depth)


# the leaves that a grid of this depth needs for its index, and no more than a few hundred besides
@pytest.mark.parametrize("depth,block", [(9, 12), (11, 50)])
def test_brick_walk_of_deep_grids(depth, block):
    tree = _uniform_tree(depth, 40 + depth, 1, 1, block + 1)
    assert tree.n_leaves >= 8 ** (depth - 4) // 16
    _same_walk(tree, depth, 512, n1=1, n2=1)


def _same_walk(tree, depth, cap=128, **sizes):
    rng = np.random.default_rng(depth)
    # rays at the leaves (the grid is mostly empty), axis-parallel ones among them
    n = 4000
    to = (tree.leaf_xyz[rng.integers(0, tree.n_leaves, n)] + rng.uniform(0, 1, (n, 3))) / (1 << depth)
    d = rng.normal(size=(n, 3))
    d[:60] = np.eye(3)[rng.integers(0, 3, 60)] * rng.choice([-1, 1], (60, 1))
    o = torch.as_tensor(to - d * rng.uniform(0.1, 2.0, (n, 1)), dtype=torch.float32, device="cuda")
    d = torch.as_tensor(d, dtype=torch.float32, device="cuda")
    out = []
    for kw in ({}, {"refill_min": 16}):
        r = fpo.Renderer(**kw, **sizes)
        r.upload(tree)
        log = r.render(rays_o=o, rays_d=d, t=7.0, visit_cap=cap, stop_T=0.0, want_T=True)
        rgb = r.render(rays_o=o, rays_d=d, t=7.0, stop_T=0.0)["rgb"]
        r.status()
        out.append((log["visit_count"], log["visit_log"], log["T"], log["rgb"], rgb))
        r.close()
    assert int(out[0][0].sum()) > n // 2
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_brick_renumbering_keeps_the_leaf_ids():
    # leaves are renumbered inside bricks: coefficient updates, marks and
    # gradients stay in upload order
    tree = _uniform_tree(6, 3)
    rng = np.random.default_rng(8)
    o = torch.as_tensor(rng.uniform(-0.5, 1.5, (3000, 3)), dtype=torch.float32, device="cuda")
    d = torch.as_tensor(rng.uniform(0.2, 0.8, (3000, 3)), dtype=torch.float32, device="cuda") - o
    a, b = fpo.Renderer(idft_mode="fused"), fpo.Renderer()
    co = torch.as_tensor(tree.coeffs, device="cuda")
    for r in (a, b):
        r.upload(synth.Tree(tree.leaf_depth, tree.leaf_xyz, np.zeros_like(tree.coeffs), 6))
        r.set_coeffs(co)
    ref = fpo.Renderer()
    ref.upload(tree)
    img = ref.render(rays_o=o, rays_d=d, t=3.0)["rgb"]
    assert torch.equal(b.render(rays_o=o, rays_d=d, t=3.0)["rgb"], img)
    rgb = a.render(rays_o=o, rays_d=d, t=3.0, visit_cap=64)
    assert float((rgb["rgb"] - img).abs().max()) < 1e-4
    mark = torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda")
    grad = torch.zeros_like(co)
    a.render_backward(rgb["rgb"], torch.ones_like(img), grad, rays_o=o, rays_d=d, t=3.0, leaf_mark=mark)
    a.status()
    log, cnt = rgb["visit_log"].cpu().numpy(), rgb["visit_count"].cpu().numpy()
    ids = np.unique(np.concatenate([log[i, :cnt[i]] for i in range(len(cnt))]))
    assert np.array_equal(np.flatnonzero(mark.cpu().numpy()), ids)
    assert float(grad[mark == 0].abs().max()) == 0.0
    for r in (a, b, ref):
        r.close()
