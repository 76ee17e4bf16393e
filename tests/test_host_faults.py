"""The library's host code against a CUDA runtime on the host (fake_cuda.cpp):
limits, failed allocations and launches, several devices. The library's own
object files are linked with the fake runtime; no GPU."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    from paper_2603_00538_gb300 import _build
    _build.build()
    objs = [os.path.join(_build.OUT_DIR, s.replace(".cu", ".o")) for s in _build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        _build.build(force=True)
    so = str(tmp_path_factory.mktemp("fake") / "libsft_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(_build._nvcc())), "include")
    # (the library's own copies of these names are bound inside the object)
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-Wl,-Bsymbolic", f"-I{inc}", "-o", so,
                    os.path.join(ROOT, "tests", "fake_cuda.cpp"), *objs, "-lpthread"], check=True)
    return ctypes.CDLL(so)


@pytest.fixture
def fake(fake_lib, monkeypatch):
    """The package bound to the fake library, and the fake's controls."""
    import paper_2603_00538_gb300 as sft
    for name, (args, res) in sft._SIGS.items():
        fn = getattr(fake_lib, name)
        fn.argtypes, fn.restype = args, res
    monkeypatch.setattr(sft, "_lib", fake_lib)
    monkeypatch.setattr(sft, "_current_stream", lambda: None)
    fake_lib.fake_reset()
    yield fake_lib
    fake_lib.fake_reset()


def _mesh(dim):
    import workloads as W
    m = W.jittered_tri_mesh(2, 1) if dim == 2 else W.jittered_kuhn_mesh(1, 1)
    return W.with_values(m, [lambda p: p[:, 0]])


# 2D: 8 triangles, n^2 <= 8 L^2; 3D: 6 tetrahedra, n^3 <= 6 L^3. The cells' linear
# index is a 32-bit integer, so 2^31 - 1 of them and more are refused, at any scale.
@pytest.mark.parametrize("dim,L", [(2, 16385.0), (2, 1e6), (2, 1e200), (2, float("inf")),
                                   (3, 711.0), (3, 1e4), (3, 1e150), (3, float("inf"))])
def test_grids_beyond_the_cell_index_are_refused(fake, dim, L):
    import paper_2603_00538_gb300 as sft
    m = _mesh(dim)
    live = fake.fake_live()
    with pytest.raises(sft.SftError) as e:
        sft.sft_source_create(m.coords, m.conn, m.values, grid_scale_L=L)
    assert e.value.status == sft.SFT_ERR_UNSUPPORTED
    assert fake.fake_live() == live


@pytest.mark.parametrize("dim,L", [(2, 16383.5), (3, 710.0)])
def test_the_largest_grids_are_still_built(fake, dim, L):
    """Just below the limit the build goes on to its cell arrays (8.6 GB, more than the fake gives)."""
    import paper_2603_00538_gb300 as sft
    m = _mesh(dim)
    with pytest.raises(sft.SftError) as e:
        sft.sft_source_create(m.coords, m.conn, m.values, grid_scale_L=L)
    assert e.value.status == sft.SFT_ERR_OOM
    assert fake.fake_live() == 0


def test_network_calls_on_several_devices(fake):
    """The kernels' shared-memory opt-in belongs to a device: first calls on each of three
    (one beyond the table of devices), then again on the first."""
    n = fake.sft_mlp_nparam()
    params, pts = np.zeros(n, np.float32), np.zeros((300, 3), np.float32)
    out, grad, loss = np.zeros(300, np.float32), np.zeros(n, np.float32), ctypes.c_double()
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    for dev in (0, 1, 70, 0):
        fake.fake_device(dev)
        h = ctypes.c_void_p()
        assert fake.sft_mlp_create(p(params), 1, None, ctypes.byref(h)) == 0
        ran = fake.fake_ran()
        assert fake.sft_mlp_forward(h, 300, p(pts), p(out), 1, None) == 0, (dev, fake.sft_last_error())
        assert fake.sft_mlp_loss_grad(h, 300, p(pts), p(out), p(grad), ctypes.byref(loss), 1, None) == 0, dev
        assert fake.sft_mlp_train(h, 300, p(pts), p(out), 1, 128, 1e-3, 1e-4, None, 1, None) == 0, dev
        assert fake.fake_ran() >= ran + 5
        fake.sft_mlp_destroy(h)
    assert fake.fake_live() == 0


@pytest.mark.parametrize("what", ["alloc", "launch"])
def test_a_solve_that_fails_half_way_can_be_repeated(fake, what):
    """Each allocation and each launch of a target's first mixed solve fails once: nothing stays
    behind, and the next solve launches the whole preparation."""
    import paper_2603_00538_gb300 as sft

    def solve(t):   # the fake's kernels do nothing, so a solve that ran reports no convergence
        with pytest.raises(sft.SftError) as e:
            sft.sft_mass_solve(t, np.ones((1, 9)), u_out=np.zeros((1, 9)))
        return e.value.status

    def first_solve():
        m = _mesh(2)
        return sft.sft_target_create(m.coords, m.conn)

    t = first_solve()
    live, ran = fake.fake_live(), fake.fake_ran()
    assert solve(t) == sft.SFT_ERR_NOT_CONVERGED
    kept, launches = fake.fake_live() - live, fake.fake_ran() - ran
    assert launches == 3 and kept == 5
    t.close()
    for k in range(1, 20) if what == "alloc" else ("k_jacobi_sqrt", "k_scaled_slices", "k_mixed"):
        t = first_solve()
        live = fake.fake_live()
        if what == "alloc":
            fake.fake_fail_alloc(k)
        else:
            fake.fake_fail_launch(k.encode())
        status = solve(t)
        fake.fake_reset()
        if status == sft.SFT_ERR_NOT_CONVERGED:   # the k-th allocation is beyond the call's last
            assert what == "alloc" and k > kept
            t.close()
            break
        assert status == (sft.SFT_ERR_OOM if what == "alloc" else sft.SFT_ERR_CUDA)
        assert fake.fake_live() - live in (0, kept)
        ran = fake.fake_ran()
        prepared = fake.fake_live() - live == kept
        assert solve(t) == sft.SFT_ERR_NOT_CONVERGED
        assert fake.fake_ran() - ran == (1 if prepared else launches)
        assert fake.fake_live() - live == kept
        t.close()
