"""Mesh intersection where source and target share vertices and edges: the same
mesh on both sides, nested regular refinements either way (every target edge
is a source edge or halves one), one triangle under a fan of more source
triangles than the shared part of the walk's queue holds (16), and the walk's
limit (256), beyond which the call is refused. Against the oracle's brute
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


def _src(n, jitter=0.0, seed=1):
    return W.with_values(W.jittered_tri_mesh(n, seed, jitter), [W.paper_f2])


PAIRS = {
    "same": lambda: (_src(12, 0.2), W.jittered_tri_mesh(12, 1, 0.2)),
    "source_refines": lambda: (_src(16), W.jittered_tri_mesh(4, 1, 0.0)),
    "target_refines": lambda: (_src(4), W.jittered_tri_mesh(16, 1, 0.0)),
    "thirds": lambda: (_src(9), W.jittered_tri_mesh(3, 1, 0.0)),
    "fine_source": lambda: (_src(14, 0.2), W.jittered_tri_mesh(2, 3, 0.2)),   # 49 triangles under each of 8
}


@pytest.mark.parametrize("name", list(PAIRS))
def test_shared_edges_match_oracle(orc, name):
    src, tgt = PAIRS[name]()
    s, t = sft.mesh_source(src, device=DEV), sft.mesh_target(tgt, device=DEV)
    b, b_o = sft.sft_mi_load_vector(s, t), orc.mi_load_vector_2d(src, tgt)
    assert np.linalg.norm(b - b_o) < 1e-13 * np.linalg.norm(b_o)
    assert np.abs(b - b_o).max() < 1e-13 * np.abs(b_o).max()
    u = np.random.default_rng(0).standard_normal(tgt.nnodes)
    e, n = sft.sft_mi_l2_error(s, t, u)
    e_o, n_o = orc.l2_error_2d(src, tgt, u)
    assert e == pytest.approx(e_o, rel=1e-12) and n == pytest.approx(n_o, rel=1e-12)


def test_too_many_source_triangles_are_refused():
    s, t = sft.mesh_source(_src(60, 0.2), device=DEV), sft.mesh_target(W.jittered_tri_mesh(2, 3, 0.0), device=DEV)
    with pytest.raises(sft.SftError) as e:
        sft.sft_mi_load_vector(s, t)
    assert e.value.status == sft.SFT_ERR_UNSUPPORTED
