"""A wait of the network tile that runs out (2 s): the kernel records it in its
error word, every thread passes the same barriers and leaves, and the context
stays usable (net_wait.cu, a kernel of the tile's own device functions)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def test_expired_network_wait_is_reported(tmp_path):
    from paper_2603_00538_gb300 import _build
    exe = str(tmp_path / "net_wait")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "net_wait.cu")
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, f"-I{_build.CSRC}", "-o", exe, src], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
