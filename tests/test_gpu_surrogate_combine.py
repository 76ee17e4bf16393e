"""The network pass's sums: warps whose 32 rows belong to one element (N a
multiple of 32) and warps that hold several (or part of one), in both
dimensions, against the FP64 sums of the sample values and control values that
the call returns. Each FP32 contribution takes at most seven roundings (value
of the control at the sample 4, residual, product, weight) on a compensated
sum: bound 8 x 2^-24 of the sum of the terms' magnitudes."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402


@pytest.mark.parametrize("dt", [2, 3])
@pytest.mark.parametrize("N", [20, 32, 33, 64, 96, 128, 160, 256])
def test_sums_equal_the_terms(orc, dt, N):
    alpha, seed = 0.7, 9
    m = W.as_precision(W.jittered_tri_mesh(5, 4) if dt == 2 else W.jittered_kuhn_mesh(2, 4), np.float32)
    nv, ne = m.nnodes, m.nelems
    net = sft.sft_mlp_create(W.mlp_init(2))
    b, g, u, sf = np.zeros(nv), np.zeros(nv), np.zeros(nv), np.zeros((ne, N), np.float32)
    sft.sft_transfer_surrogate(net, None, sft.mesh_target(m), N, seed=seed, alpha=alpha, u_out=u, b_out=b, g_out=g,
                               sample_f_out=sf)
    ref, mag = np.zeros(nv), np.zeros(nv)
    x, gd = m.coords.astype(np.float64), g.astype(np.float64)
    for t in range(ne):
        c = m.conn[t]
        e = x[c[1:]] - x[c[0]]
        vol = np.linalg.det(e) / (2.0 if dt == 2 else 6.0)
        lam = orc.sample_element(1, dt, seed, 0, t, N, m.coords[c])[0].astype(np.float64)
        gX = lam @ gd[c]
        ctl = alpha * vol / ((dt + 1) * (dt + 2)) * (gd[c].sum() + gd[c])
        ref[c] += ctl + vol / N * (lam.T @ (sf[t] - alpha * gX))
        mag[c] += alpha * vol / ((dt + 1) * (dt + 2)) * (np.abs(gd[c]).sum() + np.abs(gd[c]))
        mag[c] += vol / N * (lam.T @ (np.abs(sf[t]) + alpha * (lam @ np.abs(gd[c]))))
    assert np.all(np.abs(b - ref) <= 8 * 2.0 ** -24 * mag)
