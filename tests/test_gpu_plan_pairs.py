"""Online transfers read the recorded samples of a Philox unit in pairs where
the samples per element are even (2D), one by one where they are odd: both
equal sft_transfer's load vector (same samples; only the order of the FP64
atomic sums differs, bound 1e-14)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402


@pytest.mark.parametrize("prec", [sft.SFT_PREC_FP32, sft.SFT_PREC_FP64])
@pytest.mark.parametrize("N", [1, 2, 3, 6, 7, 34, 63])
def test_pairs_equal_transfer(prec, N):
    dt = np.float64 if prec == sft.SFT_PREC_FP64 else np.float32
    src = W.as_precision(W.with_values(W.jittered_tri_mesh(11, 1), [W.paper_f1, W.paper_f2, W.paper_f3]), dt)
    tgt = W.as_precision(W.jittered_tri_mesh(9, 2), dt)
    s, t = sft.mesh_source(src), sft.mesh_target(tgt)
    for nf in (1, 3):
        pl = sft.sft_plan_create(s, t, N, precision=prec, seed=5, field_count=nf)
        bp, bs = np.zeros((nf, tgt.nnodes)), np.zeros((nf, tgt.nnodes))
        sft.sft_plan_transfer(pl, b_out=bp)
        sft.sft_transfer(s, t, N, prec, seed=5, field_count=nf, b_out=bs)
        assert np.linalg.norm(bp - bs) < 1e-14 * np.linalg.norm(bs)
        pl.close()
