"""Mesh intersection with its pairs spread over the lanes of a warp: fewer
targets than lanes, one warp's worth and one more, more targets than the first
warps hold; targets under far more and far fewer source triangles than the
part of a walk that is kept in shared memory (20). Against the oracle's brute
force clipping, to the bounds of the general-position pairs (1e-13, 1e-12)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n_src,n_tgt", [(1, 1), (2, 1), (12, 1), (5, 3), (3, 4), (22, 4), (30, 5), (4, 37), (31, 33)])
def test_pairs_over_lanes_match_oracle(orc, n_src, n_tgt):
    src = W.with_values(W.jittered_tri_mesh(n_src, 2, 0.2), [W.paper_f1, W.paper_f2])
    tgt = W.jittered_tri_mesh(n_tgt, 7, 0.2)
    s, t = sft.mesh_source(src, device=DEV), sft.mesh_target(tgt, device=DEV)
    for field in (0, 1):
        f = W.Mesh(src.coords, src.conn, src.values[field:field + 1])
        b, b_o = sft.sft_mi_load_vector(s, t, field), orc.mi_load_vector_2d(f, tgt)
        assert np.linalg.norm(b - b_o) < 1e-13 * np.linalg.norm(b_o)
        u = np.random.default_rng(field).standard_normal(tgt.nnodes)
        e, n = sft.sft_mi_l2_error(s, t, u, field)
        e_o, n_o = orc.l2_error_2d(f, tgt, u)
        assert e == pytest.approx(e_o, rel=1e-12) and n == pytest.approx(n_o, rel=1e-12)


def test_l2_error_is_the_same_every_time():
    src = W.with_values(W.jittered_tri_mesh(70, 2, 0.2), [W.paper_f2])
    tgt = W.jittered_tri_mesh(50, 7, 0.2)
    s, t = sft.mesh_source(src, device=DEV), sft.mesh_target(tgt, device=DEV)
    u = np.random.default_rng(0).standard_normal(tgt.nnodes)
    assert len({sft.sft_mi_l2_error(s, t, u) for _ in range(3)}) == 1
