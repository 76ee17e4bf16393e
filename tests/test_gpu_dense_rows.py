"""Mass rows of a mesh in which every node of one line meets every node of a
skew line: rows of up to 64 entries, so a block of the copy pass has more
entries than it holds in shared memory (m = 60), about as many (m = 18, 19) or
few (m = 4). Against the oracle, entry for entry."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,m", [(60, 60), (300, 18), (300, 19), (130, 4), (1, 1)])
def test_rows_equal_oracle(orc, n, m):
    a = np.arange(n + 1)[:, None] * [1.0, 0, 0] / n
    b = np.arange(m + 1)[:, None] * [0, 1.0, 0] / m + [0, 0, 1.0]
    c = [[i, i + 1, n + 1 + j, n + 2 + j] for i in range(n) for j in range(m)]
    mesh = W.Mesh(np.vstack([a, b]), np.array(c, np.int32), None)
    W._fix_orientation(mesh)
    if max(n, m) > 60:   # keep the rows of the short line's nodes within 64 entries: parts of 58 along the long one
        parts, conn = [], []
        for k in range(0, n, 58):
            w = min(58, n - k)
            off = sum(len(p) for p in parts)
            parts.append(np.vstack([a[k:k + w + 1], b]) + [0, 0, 2.0 * k])
            conn += [[off + i, off + i + 1, off + w + 1 + j, off + w + 2 + j] for i in range(w) for j in range(m)]
        mesh = W.Mesh(np.vstack(parts), np.array(conn, np.int32), None)
        W._fix_orientation(mesh)
    rp, col, val, lump = sft.sft_target_mass(sft.mesh_target(mesh, device=DEV))
    rp_o, col_o, val_o = orc.mass_csr(mesh.coords, mesh.conn)
    assert np.diff(rp_o).max() <= 64
    assert np.array_equal(rp, rp_o) and np.array_equal(col, col_o)
    assert np.max(np.abs(val - val_o)) <= 1e-15 * np.max(np.abs(val_o))
    assert np.max(np.abs(lump - orc.lumped_mass(mesh.coords, mesh.conn))) <= 1e-15
