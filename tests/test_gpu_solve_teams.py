"""The mixed-precision solve over the sizes at which its kernel changes shape:
one block, a cluster or the whole grid per system (by nonzeros x fields), row
counts off the slice of 32, 1 to 8 fields (padded to 1, 2, 4, 8), rows of y in
shared memory or only in global memory, long rows and nodes of no element.

The stopping test is on the FP64 residual, so the residual recomputed on the
host from the oracle's CSR matrix is held to 2 tol (its own FP64 rounding is
some 1e-15 of ||b||)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")


def _spmv(rp, col, val, x):
    rows = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    return np.bincount(rows, weights=val * x[col], minlength=len(rp) - 1)


def _check(orc, m, nrhs, tol=1e-12, seed=1):
    t = sft.mesh_target(m, device=DEV)
    rp, col, val = orc.mass_csr(m.coords, m.conn)
    rng = np.random.default_rng(seed)
    b = np.stack([_spmv(rp, col, val, rng.standard_normal(m.nnodes)) for _ in range(nrhs)])
    u, it, rr = sft.sft_mass_solve(t, b, tol=tol, max_iter=500)
    assert rr <= tol and it > 0
    for f in range(nrhs):
        assert np.linalg.norm(b[f] - _spmv(rp, col, val, u[f])) <= 2 * tol * np.linalg.norm(b[f])
    return u


# nonzeros x padded fields: a block up to 10,000, a cluster up to 110,000
@pytest.mark.parametrize("dim,n,nrhs", [(2, 2, 1), (2, 3, 8), (2, 36, 1), (2, 38, 1), (2, 26, 2), (2, 27, 2), (2, 60, 1),
                                        (2, 124, 1), (2, 126, 1), (2, 40, 7), (2, 130, 3), (3, 3, 1), (3, 9, 1),
                                        (3, 18, 1), (3, 19, 1), (3, 11, 5), (2, 210, 6), (2, 400, 1)])
def test_teams(orc, dim, n, nrhs):
    m = W.jittered_tri_mesh(n, 3) if dim == 2 else W.jittered_kuhn_mesh(n, 3)
    _check(orc, m, nrhs)


def test_rows_of_y_in_global_memory(orc):
    _check(orc, W.jittered_tri_mesh(570, 2), 8, tol=1e-11)   # 326,041 rows x 8 fields


@pytest.mark.parametrize("scale", [1, 12])
def test_long_rows_and_unused_nodes(orc, scale):
    # a fan of 40 triangles round the centre (a row of 41), a strip of many
    # fans beside it, and three nodes of no element
    k = 40
    parts, conn, base = [], [], 0
    for c in range(scale):
        a = 2 * np.pi * np.arange(k) / k
        parts.append(np.concatenate([[[3.0 * c, 0.0]], np.stack([3.0 * c + np.cos(a), np.sin(a)], 1)]))
        i = np.arange(k)
        conn.append(base + np.stack([np.zeros(k, int), 1 + i, 1 + (i + 1) % k], 1))
        base += k + 1
    coords = np.concatenate(parts + [np.array([[9e3, 1.0], [9e3, 2.0], [9e3, 3.0]])])
    m = W.Mesh(coords, np.concatenate(conn).astype(np.int32), None)
    u = _check(orc, m, 3)
    assert np.all(u[:, -3:] == 0.0)


@pytest.mark.parametrize("n", [20, 100, 300])
def test_warm_start_and_budget_on_every_team(orc, n):
    src = W.with_values(W.jittered_tri_mesh(40, 0), [W.field_sincos])
    s, t = sft.mesh_source(src, device=DEV), sft.mesh_target(W.jittered_tri_mesh(n, 1), device=DEV)
    u = torch.zeros((1, (n + 1) ** 2), dtype=torch.float64, device=DEV)
    sft.sft_transfer(s, t, 8, sft.SFT_PREC_FP64, cg_tol=1e-12, u_out=u)
    cold = u.clone()
    _, st, _ = sft.sft_transfer(s, t, 8, sft.SFT_PREC_FP64, cg_tol=1e-12, u_out=u, cg_warm_start=True)
    assert st["cg_iters"] == 0 and torch.equal(u, cold)
    b = torch.randn((1, (n + 1) ** 2), dtype=torch.float64, device=DEV)
    with pytest.raises(sft.SftError) as e:
        sft.sft_mass_solve(t, b, tol=1e-12, max_iter=3, u_out=u)
    assert e.value.status == sft.SFT_ERR_NOT_CONVERGED
