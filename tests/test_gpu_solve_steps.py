"""Step counts of the mixed solve's first cycle at their edges. From u = 0 the
cycle asks for e = 0.1 tol (clamped to 1e-5 .. 1/4), and takes the smallest K
with T_K(s1) >= 1 / e (s1 of the spectrum interval, formed in FP32 as the
kernel does). Tolerances 1e-9 to either side of 10 / T_K tell the counts of
64-bit arithmetic from those of 32; an easy right-hand side (one smooth mode)
converges within the cycle, so the reported iterations are the count. On a
block, a cluster and the grid."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_00538_gb300 as sft  # noqa: E402

DEV = torch.device("cuda:0")


def _chebyshev(dim):
    f = np.float32
    a, b = f(0.5) * (f(1) - f(1e-3)), f(2.0 if dim == 2 else 2.5) * (f(1) + f(1e-3))
    s1 = float((f(0.5) * (a + b)) / (f(0.5) * (b - a)))
    t = [1.0, s1]
    while len(t) < 16:
        t.append(2 * s1 * t[-1] - t[-2])
    return t


def _steps(dim, tol):
    t = _chebyshev(dim)
    e = min(0.25, max(float(np.float32(1e-5)), 0.1 * tol))
    return next(k for k in range(1, 16) if t[k] * e >= 1.0)


@pytest.mark.parametrize("dim,n", [(2, 20), (2, 60), (2, 140), (3, 7), (3, 12), (3, 22)])
def test_steps_of_the_first_cycle(orc, dim, n):
    m = W.jittered_tri_mesh(n, 3) if dim == 2 else W.jittered_kuhn_mesh(n, 3)
    t = sft.mesh_target(m, device=DEV)
    rp, col, val = orc.mass_csr(m.coords, m.conn)
    rows = np.repeat(np.arange(m.nnodes), np.diff(rp))
    b = np.bincount(rows, weights=val, minlength=m.nnodes)[None]   # M 1
    cheb = _chebyshev(dim)
    tols = [10.0 / cheb[k] * (1 + s) for k in range(3, 13) for s in (1e-9, -1e-9)]
    for tol in (x for x in tols if 1.001e-4 < x < 1.0):
        _, it, rr = sft.sft_mass_solve(t, b, tol=tol, max_iter=100)
        assert rr <= tol
        assert it == _steps(dim, tol), tol


@pytest.mark.parametrize("tol", [0.0, 1e-12, 1e153, 1e160, 1e308])
def test_zero_right_hand_side_converges_at_any_tolerance(tol):
    """||r|| <= tol ||b|| holds with both zero, whatever tol (its square overflows above 1e154)."""
    t = sft.mesh_target(W.jittered_tri_mesh(8, 3), device=DEV)
    u, it, rr = sft.sft_mass_solve(t, np.zeros((2, 81)), tol=tol, max_iter=50)
    assert it == 0 and rr == 0.0 and not u.any()


@pytest.mark.parametrize("n,nrhs", [(1960, 1), (1950, 2)])
def test_systems_that_hold_little_of_their_matrix(n, nrhs):
    """More than 26 M nonzeros: k_mixed keeps 12,000 entries of a block's 175,000. Against the FP64 CG
    (each residual below tol ||b||, and cond(M) of this mesh's Jacobi-scaled matrix is at most 4;
    the areas differ by less than a factor of 10, which bounds the unscaled one by 40)."""
    t = sft.mesh_target(W.jittered_tri_mesh(n, 3), device=DEV)
    g = torch.Generator(device=DEV)
    g.manual_seed(n)
    b = torch.randn((nrhs, (n + 1) ** 2), dtype=torch.float64, device=DEV, generator=g)
    u, v = torch.zeros_like(b), torch.zeros_like(b)
    _, _, rr = sft.sft_mass_solve(t, b, tol=1e-11, u_out=u)
    sft.sft_mass_solve(t, b, tol=1e-11, u_out=v, cg_mode=sft.SFT_CG_FP64)
    assert rr <= 1e-11
    for f in range(nrhs):
        assert float((u[f] - v[f]).norm() / v[f].norm()) <= 2 * 40 * 1e-11
