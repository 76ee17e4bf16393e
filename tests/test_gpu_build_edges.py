"""Grid registration and mass rows where their kernels change path: elements
whose box has more cells than the bit mask (64), cells whose centres lie on
faces (ties of the start element, thresholds the FP32 bound cannot settle),
coordinates far from the origin (a wide bound) and of extreme scale (no bound
at all), one element, and rows at the edges of the hash tables (half and full).
Everything equal to the oracle, entry for entry."""
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


def _mesh(dim, kind):
    jitter = 0.0 if kind.startswith("regular") else 0.15 if dim == 2 else 0.08
    n = {"one": 1}.get(kind, 13 if dim == 2 else 5)
    m = W.jittered_tri_mesh(n, 3, jitter) if dim == 2 else W.jittered_kuhn_mesh(n, 3, jitter)
    x, c = m.coords, m.conn
    if kind == "one":
        c = c[:1]
        x, c = x[c[0]], np.arange(dim + 1, dtype=np.int32)[None]
    elif kind == "graded":
        x = x ** 2
    elif kind == "offset":
        x = x + 64.0
    elif kind == "tiny":
        x = x * 2.0 ** -40
    elif kind == "huge":
        x = x * 2.0 ** 55   # beyond the range the FP32 bound is used in
    m = W.Mesh(np.ascontiguousarray(x), np.ascontiguousarray(c), None)
    return W.with_values(m, [lambda p: p[:, 0]])


CASES = [("jittered", 1.0), ("jittered", 4.5), ("regular", 1.0), ("regular", 0.708), ("regular", 2.0), ("graded", 1.5),
         ("offset", 1.0), ("tiny", 1.0), ("huge", 1.0), ("one", 1.0), ("one", 3.0), ("one", 12.0)]


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("kind,L", CASES)
def test_registration_equals_oracle(orc, dim, prec, kind, L):
    m = _mesh(dim, kind)
    if prec == FP32:
        m = W.as_precision(m, np.float32)
    if (dim, prec, kind) == (3, FP32, "huge"):   # its determinants exceed FP32: refused
        with pytest.raises(sft.SftError):
            sft.mesh_source(m, L, device=DEV)
        return
    s = sft.mesh_source(m, L, device=DEV)
    n, start, items = sft.sft_source_grid(s, prec)
    g = orc.Grid(1 if prec == FP32 else 0, m.coords, m.conn, L)
    start_o, items_o = g.csr()
    assert list(n) == list(g.shape()[0])
    assert np.array_equal(start, start_o)
    cell = np.repeat(np.arange(len(start) - 1), np.diff(start))
    assert np.array_equal(items[np.lexsort((items, cell))], items_o[np.lexsort((items_o, cell))])
    first = sft.sft_source_cell_first(s, prec)
    nonempty = np.diff(start_o) > 0
    assert np.array_equal(first[nonempty], items_o[start_o[:-1][nonempty]])
    assert np.all(first[~nonempty] == -1)
    assert np.array_equal(sft.sft_source_adjacency(s, prec), g.adjacency())


@pytest.mark.parametrize("k", [3, 6, 7, 8, 14, 15, 16, 40])
def test_row_lengths_at_table_edges(orc, k):
    """A hub of k triangles: its row has k + 1 entries."""
    ang = 2 * np.pi * np.arange(k) / k
    x = np.vstack([[0.0, 0.0], np.stack([np.cos(ang), np.sin(ang)], 1)])
    c = np.array([[0, 1 + i, 1 + (i + 1) % k] for i in range(k)], np.int32)
    perm = np.random.default_rng(k).permutation(k + 1).astype(np.int32)   # hub anywhere in the numbering
    xp = np.empty_like(x)
    xp[perm] = x
    m = W.Mesh(xp, perm[c], None)
    rp, col, val, lump = sft.sft_target_mass(sft.mesh_target(m, device=DEV))
    rp_o, col_o, val_o = orc.mass_csr(m.coords, m.conn)
    assert np.array_equal(rp, rp_o) and np.array_equal(col, col_o)
    assert np.max(np.abs(val - val_o)) <= 1e-15 * np.max(np.abs(val_o))
    assert np.max(np.abs(lump - orc.lumped_mass(m.coords, m.conn))) <= 1e-15
