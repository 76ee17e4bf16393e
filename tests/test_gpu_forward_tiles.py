"""The network forward at the edges of its tiling (128-row tiles dealt to two
alternating groups of each persistent CTA: one tile, a ragged last tile, odd
and even tile counts per CTA) and the network pass of the surrogate transfer
over several chunks of samples.

A row's value depends on its own input only and is computed by the same
operations wherever the row falls, so the values are compared bit for bit
with those of the rows in reversed order and of small calls. With a constant
network and alpha = 0 the estimator is b_i = |T| / N sum_j k lambda_i summed
over elements, so sum_i b_i = k sum |T| up to FP32 rounding of the weights
(about 1e-7 relative, against 1.4e-5 for one element of 72,000 missing)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")
SMS = torch.cuda.get_device_properties(0).multi_processor_count
ROUND = 128 * SMS


@pytest.mark.parametrize("n", [1, 127, 128, 129, 300, ROUND - 1, ROUND, ROUND + 1, 2 * ROUND + 1, 3 * ROUND + 130,
                               4 * ROUND + 64])
def test_forward_rows_do_not_depend_on_the_tiling(n):
    net = sft.sft_mlp_create(W.mlp_init(3))
    g = torch.Generator(device=DEV)
    g.manual_seed(n)
    pts = torch.rand((n, 3), device=DEV, generator=g)
    y = torch.empty(n, device=DEV)
    sft.sft_mlp_forward(net, pts, y)
    r = torch.empty(n, device=DEV)
    sft.sft_mlp_forward(net, pts.flip(0).contiguous(), r)
    assert torch.equal(y, r.flip(0))
    for a in sorted({0, max(0, n // 2 - 20), max(0, n - 40)}):
        part = torch.empty(min(40, n - a), device=DEV)
        sft.sft_mlp_forward(net, pts[a:a + 40].contiguous(), part)
        assert torch.equal(part, y[a:a + 40])


@pytest.mark.parametrize("N", [64, 50, 130])
def test_network_pass_over_several_chunks(N):
    k = 0.75
    p = W.mlp_init(1)
    p[-257:-1] = 0.0     # w5
    p[-1] = k
    net = sft.sft_mlp_create(p)
    m = W.jittered_tri_mesh(230 if N < 128 else 140, 4)   # a chunk holds 4 Mi samples: two chunks
    t = sft.mesh_target(m, device=DEV)
    u = torch.zeros(m.nnodes, dtype=torch.float64, device=DEV)
    b = torch.zeros_like(u)
    sf = torch.zeros((m.nelems, N), dtype=torch.float32, device=DEV)
    _, st, _ = sft.sft_transfer_surrogate(net, None, t, N, alpha=0.0, u_out=u, b_out=b, sample_f_out=sf)
    assert m.nelems * N > 4 << 20
    assert st["net_queries"] == m.nnodes + m.nelems * N
    assert bool((sf == k).all())
    assert abs(float(b.sum()) / k - 1.0) < 1e-6
