"""The wait limit of the mixed solve on each of its teams. On a cluster of blocks
every barrier overruns a limit of 1 ns; the overrun is noted and all blocks
leave at the next barrier, so the call reports SFT_ERR_DEVICE_STATUS, and the
target solves again once the limit is restored. One block waits for no other
and solves under any limit."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")


# nonzeros x fields (padded to 1, 2, 4, 8): a block up to 10,000, a cluster up to 110,000
@pytest.mark.parametrize("dim,n,nrhs,team", [(2, 20, 1, "block"), (2, 60, 1, "cluster"), (2, 100, 1, "cluster"),
                                             (2, 60, 2, "cluster"), (2, 40, 7, "cluster"), (3, 12, 1, "cluster"),
                                             (2, 200, 1, "grid"), (2, 100, 3, "grid")])
@pytest.mark.parametrize("warm", [False, True])
def test_limit_on_every_team(orc, dim, n, nrhs, team, warm):
    m = W.jittered_tri_mesh(n, 3) if dim == 2 else W.jittered_kuhn_mesh(n, 3)
    t = sft.mesh_target(m, device=DEV)
    rp, col, val = orc.mass_csr(m.coords, m.conn)
    work = len(col) * (nrhs if nrhs <= 2 else 4 if nrhs <= 4 else 8)
    assert team == ("block" if work <= 10000 else "cluster" if work <= 110000 else "grid")
    src = W.with_values(m, [W.field_sincos if dim == 2 else (lambda p: p[:, 0])] * nrhs)
    s = sft.mesh_source(src, device=DEV)
    u = torch.zeros((nrhs, m.nnodes), dtype=torch.float64, device=DEV)

    def solve(tol):   # through the transfer: with and without a warm start
        return sft.sft_transfer(s, t, 4, sft.SFT_PREC_FP32, cg_tol=tol, u_out=u, cg_warm_start=warm)[1]

    sft.sft_target_set_wait_limit(t, 1e-9)
    for _ in range(2):
        if team == "block":
            assert solve(1e-12)["cg_rel_resid"] <= 1e-12
            continue
        with pytest.raises(sft.SftError) as e:
            solve(1e-12)
        assert e.value.status == sft.SFT_ERR_DEVICE_STATUS
    sft.sft_target_set_wait_limit(t, 2.0)
    u.zero_()
    assert solve(1e-12)["cg_rel_resid"] <= 1e-12
    b = np.random.default_rng(5).standard_normal((nrhs, m.nnodes))
    x, _, rr = sft.sft_mass_solve(t, b, tol=1e-12, max_iter=500)
    assert rr <= 1e-12
    rows = np.repeat(np.arange(m.nnodes), np.diff(rp))
    for f in range(nrhs):
        r = b[f] - np.bincount(rows, weights=val * x[f][col], minlength=m.nnodes)
        assert np.linalg.norm(r) <= 2e-12 * np.linalg.norm(b[f])
