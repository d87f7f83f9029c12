"""The adjoint and the fine-tuning update inside CUDA graphs: what a graph does
depends on nothing that later calls of the context change."""

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


class Batch:
    def __init__(self, r, n, seed):
        rng = np.random.default_rng(seed)
        dev = lambda x: torch.as_tensor(x, dtype=torch.float32, device="cuda").contiguous()
        o = rng.uniform(-0.6, 1.6, (n, 3))
        self.kw = dict(rays_o=dev(o), rays_d=dev(rng.uniform(0.2, 0.8, (n, 3)) - o), t_per_ray=dev(rng.uniform(0, 60, n)))
        self.g = dev(rng.normal(size=(n, 3)))
        self.rgb = r.render(**self.kw)["rgb"]

    def backward(self, r, grad, **kw):
        r.render_backward(self.rgb, self.g, grad, **self.kw, **kw)


def _close(a, b):
    # FP32 sums of up to a few hundred visits a leaf in another order: each within
    # 300 * 2^-24 = 2e-5 of its sum of |terms|, itself a few times the largest element
    assert float(b.abs().max()) > 0 and float((a - b).abs().max()) <= 1e-4 * float(b.abs().max())


def _setup():
    tree = synth.shell_tree(5)
    r = fpo.Renderer(idft_mode="fused")
    r.upload(tree)
    p = torch.as_tensor(tree.coeffs, device="cuda").clone()
    return r, p, torch.zeros(tree.n_leaves, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("n", [300, 70000])  # adds by warps, and by one lane a ray
def test_captured_adjoint_outlives_a_larger_call_and_deferred_visits(n):
    r, p, mark = _setup()
    a, b, c = Batch(r, n, 1), Batch(r, n + 9000, 2), Batch(r, 500, 3)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    want, got, big, pend = (torch.zeros_like(p) for _ in range(4))
    a.backward(r, want)  # the context has its workspace for 4096 rays now
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.backward(r, got)
    b.backward(r, big)  # ... and a larger one
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    _close(got, want)
    # a replay between a deferred adjoint and its update changes neither
    q = p.clone()
    r.set_coeffs(p)
    c.backward(r, pend, leaf_mark=mark, defer=True)
    got.zero_()
    graph.replay()
    r.adam_leaves(p, pend, m, v, mark, 1)
    r.status()
    _close(got, want)
    m2, v2, mark2, dense = torch.zeros_like(m), torch.zeros_like(v), torch.zeros_like(mark), torch.zeros_like(pend)
    r.set_coeffs(q)
    c.backward(r, dense, leaf_mark=mark2)
    r.adam_leaves(q, dense, m2, v2, mark2, 1)
    r.status()
    r.close()
    _close(m, m2)


def test_captured_step_replays_and_waiting_visits_are_not_captured():
    r, p, mark = _setup()
    a = Batch(r, 700, 4)
    p0, grad = p.clone(), torch.zeros_like(p)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    r.set_coeffs(p)
    a.backward(r, grad, leaf_mark=mark, defer=True)
    r.adam_leaves(p, grad, m, v, mark, 7)
    want = m.clone()
    for x, y in ((p, p0), (m, None), (v, None)):
        x.zero_() if y is None else x.copy_(y)
    r.set_coeffs(p)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.backward(r, grad, leaf_mark=mark, defer=True)
        r.adam_leaves(p, grad, m, v, mark, 7)
    graph.replay()
    r.status()
    _close(m, want)
    assert not grad.any() and not mark.any()
    # visits that wait belong to the calls made now, not to a graph
    a.backward(r, grad, leaf_mark=mark, defer=True)
    other = torch.cuda.CUDAGraph()
    with torch.cuda.graph(other):
        for call in (lambda: r.adam_leaves(p, grad, m, v, mark, 8), lambda: r.set_coeffs(p)):
            with pytest.raises(fpo.FPOError, match="deferred visits wait"):
                call()
        want.add_(1.0)
    m.zero_()
    r.adam_leaves(p, grad, m, v, mark, 8)
    r.status()
    r.close()
    assert m.any()


def test_first_adjoint_beside_another_streams_capture():
    # the workspace's allocation does not end a capture under way elsewhere
    r, p, _ = _setup()
    a = Batch(r, 300, 5)
    want, got, x = torch.zeros_like(p), torch.zeros_like(p), torch.zeros(4, device="cuda")
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        x.add_(1.0)
        a.backward(r, got, stream=side)
    torch.cuda.synchronize()
    graph.replay()
    a.backward(r, want)
    r.status()
    r.close()
    assert float(x[0]) == 1.0
    _close(got, want)
