"""Grid registration of elements whose boxes have more than 64 cells: masks of
several words on fine grids (by the grid scale), and the list of elements beyond
their masks, which a warp takes up to 32 at a time. Few such elements, and all of
a mesh; boxes around the edges of the words and of some thousands of cells, one
to three cells high, of cells with very different sides; coordinates beyond the
FP32 filter's range. Cell lists and start elements equal to the oracle's, entry
for entry."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

FP32, FP64 = sft.SFT_PREC_FP32, sft.SFT_PREC_FP64
DEV = torch.device("cuda:0")


def _mesh(dim, n, kind):
    m = W.jittered_tri_mesh(n, 3, 0.15) if dim == 2 else W.jittered_kuhn_mesh(n, 3, 0.08)
    x = m.coords
    if kind == "graded":          # the largest elements take thousands of cells, the smallest one
        x = x ** 3
    elif kind == "rows":          # boxes over the whole width and one to three cells high
        keep = x[m.conn][:, :, 0].max(1) < 1.4 / n
        used, c = np.unique(m.conn[keep], return_inverse=True)
        m = W.Mesh(x[used], c.reshape(-1, dim + 1).astype(np.int32), None)
        x = m.coords
    elif kind == "anisotropic":   # cells of very different sides
        x = x * ([4.0] + [1.0] * (dim - 2) + [1e-6])
    elif kind == "huge":
        x = x * 2.0 ** (55 if dim == 2 else 52)
    return W.with_values(W.Mesh(np.ascontiguousarray(x), m.conn, None), [lambda p: p[:, 0]])


CASES = [(2, 3, "plain", 7.0), (2, 40, "plain", 5.5), (2, 60, "plain", 7.0), (2, 20, "graded", 2.0), (2, 12, "graded", 9.0),
         (2, 12, "anisotropic", 8.0), (2, 100, "rows", 8.0), (2, 12, "huge", 7.0), (3, 2, "plain", 4.0), (3, 9, "plain", 2.0), (3, 9, "plain", 2.7),
         (3, 6, "graded", 2.0), (3, 5, "huge", 2.5), (2, 3, "plain", 30.0), (2, 5, "huge", 30.0), (3, 2, "plain", 8.0),
         (3, 4, "graded", 4.0), (3, 3, "huge", 6.5), (2, 30, "plain", 4.1), (3, 12, "plain", 1.62), (2, 50, "graded", 1.0),
         (3, 10, "graded", 1.0)]


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("dim,n,kind,L", CASES)
def test_large_boxes_equal_oracle(orc, dim, n, kind, L, prec):
    m = _mesh(dim, n, kind)
    if prec == FP32:
        if (dim, kind) == (3, "huge"):
            m.coords[:] *= 2.0 ** -30   # the largest scale whose FP32 determinants are finite
        m = W.as_precision(m, np.float32)
    s = sft.mesh_source(m, L, device=DEV)
    nc, start, items = sft.sft_source_grid(s, prec)
    g = orc.Grid(1 if prec == FP32 else 0, m.coords, m.conn, L)
    start_o, items_o = g.csr()
    assert list(nc) == list(g.shape()[0])
    assert np.array_equal(start, start_o)
    cell = np.repeat(np.arange(len(start) - 1), np.diff(start))
    assert np.array_equal(items[np.lexsort((items, cell))], items_o[np.lexsort((items_o, cell))])
    first = sft.sft_source_cell_first(s, prec)
    nonempty = np.diff(start_o) > 0
    assert np.array_equal(first[nonempty], items_o[start_o[:-1][nonempty]])
    assert np.all(first[~nonempty] == -1)
