"""The batched mixed-precision solve by 32-row slices: pieces that start and
end inside a slice, systems smaller than one, every padded field count, both
dimensions and tolerances of one and of several cycles in one batch. Every
system's true residual (FP64, from the load vector that comes back) meets its
tolerance (the solver tests the same quantity; 1e-3 relative for the order of
the sums), and an iteration limit below what is needed is kept and reported."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")
FIELDS = [lambda x, k=k: np.cos((k + 1) * x[:, 0]) + x[:, 1] * (k + 2) for k in range(8)]


def _requests(max_iter):
    s2 = sft.mesh_source(W.as_precision(W.with_values(W.jittered_tri_mesh(20, 3), FIELDS), np.float32), device=DEV)
    s3 = sft.mesh_source(W.as_precision(W.with_values(W.jittered_kuhn_mesh(6, 3), FIELDS), np.float32), device=DEV)
    srcs, tgts, opts = [], [], []
    for k, (dim, n, nf, tol) in enumerate([(2, 1, 1, 1e-10), (2, 4, 2, 1e-6), (2, 5, 3, 1e-12), (2, 15, 4, 1e-3),
                                           (2, 30, 5, 1e-10), (2, 61, 8, 1e-10), (3, 1, 8, 1e-10), (3, 2, 7, 1e-12),
                                           (3, 7, 1, 1e-2), (3, 10, 6, 1e-10), (2, 40, 1, 1e-10), (3, 9, 2, 1e-8)]):
        m = W.jittered_tri_mesh(n, 50 + k) if dim == 2 else W.jittered_kuhn_mesh(n, 50 + k)
        srcs.append(s2 if dim == 2 else s3)
        tgts.append(sft.mesh_target(W.as_precision(m, np.float32), device=DEV))
        opts.append(dict(samples_per_elem=8, seed=k, field_count=nf, cg_tol=tol, cg_max_iter=max_iter))
    return srcs, tgts, opts


def test_every_system_meets_its_tolerance():
    srcs, tgts, opts = _requests(2000)
    b = sft.sft_batch_create(srcs, tgts, opts)
    for _ in range(2):
        _, st = sft.sft_batch_run(b)
        assert st["nonconverged"] == 0
        for r, o in enumerate(opts):
            rp, col, val, _ = sft.sft_target_mass(tgts[r])
            n = len(rp) - 1
            u, bb = sft.sft_batch_result(b, r, b_out=np.zeros((o["field_count"], n)))
            rows = np.repeat(np.arange(n), np.diff(rp))
            for f in range(o["field_count"]):
                res = bb[f] - np.bincount(rows, weights=val * u[f][col], minlength=n)
                assert np.linalg.norm(res) <= 1.001 * o["cg_tol"] * np.linalg.norm(bb[f]) + 1e-15, (r, f)
    b.close()


def test_iteration_limit_is_reported():
    srcs, tgts, opts = _requests(2)
    b = sft.sft_batch_create(srcs, tgts, opts)
    with pytest.raises(sft.SftError) as e:
        sft.sft_batch_run(b)
    assert e.value.status == 5 and "iteration cap" in str(e.value)
    b.close()
