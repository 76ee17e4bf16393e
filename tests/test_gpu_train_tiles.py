"""The training gradient over the edges of its tiling: one row, ragged 128-row
tiles, one and several tiles per CTA group, more tiles than one pass over the
two kernels takes (608).

The mean loss over two halves of m points is the mean of the halves' losses,
and so is the gradient. dL/dy of the whole is exactly half of a half's (the
same value times a power of two), so every BF16 rounding on the way is the same
and the two sides differ by the order of FP32 sums only: at most a few hundred
partial sums of up to 128 terms each, some 1e-6 relative; 2e-5 of each
parameter block's norm."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")
H = W.MLP_HIDDEN
BLOCKS = np.cumsum([0, 3 * H, H, H * H, H, H * H, H, H * H, H, H, 1])


def _grad(net, pts, f):
    g = torch.empty(sft.sft_mlp_nparam(), dtype=torch.float32, device=DEV)
    loss = sft.sft_mlp_loss_grad(net, pts, f, g)
    return loss, g.double().cpu().numpy()


@pytest.mark.parametrize("m", [1, 63, 64, 65, 127, 128, 200, 9800, 19456, 29187, 39001])
def test_gradient_of_two_halves(m):
    net = sft.sft_mlp_create(W.mlp_init(2))
    g = torch.Generator(device=DEV)
    g.manual_seed(m)
    pts = torch.rand((2 * m, 3), device=DEV, generator=g)
    f = torch.sin(7 * pts[:, 0]) + pts[:, 1] * pts[:, 2]
    loss, whole = _grad(net, pts, f)
    la, a = _grad(net, pts[:m].contiguous(), f[:m].contiguous())
    lb, b = _grad(net, pts[m:].contiguous(), f[m:].contiguous())
    assert loss == pytest.approx(0.5 * (la + lb), rel=1e-6)
    halves = 0.5 * (a + b)
    for lo, hi in zip(BLOCKS[:-1], BLOCKS[1:]):
        assert np.linalg.norm(whole[lo:hi] - halves[lo:hi]) <= 2e-5 * np.linalg.norm(halves[lo:hi]) + 1e-30
