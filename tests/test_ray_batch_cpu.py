"""camera_ray_batch refuses a basis that its kernel could not read (no launch)."""

import pytest

torch = pytest.importorskip("torch")

from paper_2202_08614_gb300 import synth  # noqa: E402
from paper_2202_08614_gb300.finetune import camera_ray_batch  # noqa: E402


class _OnCuda:
    """What camera_ray_batch looks at before it draws, said to be on the GPU."""

    is_cuda, device = True, "cuda:0"

    def __init__(self, t):
        self.shape, self.dtype, self.dim = t.shape, t.dtype, t.dim


@pytest.mark.parametrize("basis", [torch.zeros(5, 12), _OnCuda(torch.zeros(4, 12)), _OnCuda(torch.zeros(5, 11)),
                                   _OnCuda(torch.zeros(60))])
def test_refused_bases(basis):
    with pytest.raises(ValueError, match="basis must be"):
        camera_ray_batch(synth.ring_cameras(5, 8, 8), 16, None, basis=basis)
