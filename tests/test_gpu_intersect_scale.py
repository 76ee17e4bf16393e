"""Mesh intersection of meshes of extreme scale: lengths near 2^-400 .. 2^400
(areas within FP64, their squares far outside), powers of two off and on the
scale of the areas. Everything of the integrals scales by a power of two, so
load vector, error and norm are those of the mesh at scale 1 within the bounds
that its general-position pairs have against the oracle (1e-13, 1e-12)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("p", [-400, -301, -160, -20, 0, 17, 160, 301, 400])
def test_scale(orc, p):
    src = W.with_values(W.jittered_tri_mesh(14, 1, 0.2), [W.paper_f2])
    tgt = W.jittered_tri_mesh(11, 3, 0.2)
    u = np.random.default_rng(0).standard_normal(tgt.nnodes)
    s = sft.sft_source_create(np.ldexp(src.coords, p), src.conn, src.values)
    t = sft.sft_target_create(np.ldexp(tgt.coords, p), tgt.conn)
    b, b_o = np.ldexp(sft.sft_mi_load_vector(s, t), -2 * p), orc.mi_load_vector_2d(src, tgt)
    assert np.linalg.norm(b - b_o) < 1e-13 * np.linalg.norm(b_o)
    assert np.abs(b - b_o).max() < 1e-13 * np.abs(b_o).max()
    e, n = (float(np.ldexp(x, -p)) for x in sft.sft_mi_l2_error(s, t, u))
    e_o, n_o = orc.l2_error_2d(src, tgt, u)
    assert e == pytest.approx(e_o, rel=1e-12) and n == pytest.approx(n_o, rel=1e-12)
