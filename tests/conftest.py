import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)
HERE = os.path.dirname(os.path.abspath(__file__))
if HERE not in sys.path:
    sys.path.insert(0, HERE)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300) and the built library")
    config.addinivalue_line("markers", "slow: longer CPU statistical test")


@pytest.fixture(scope="session")
def internal(tmp_path_factory):
    """(torch, tests/internal.cu linked with the library's object files)."""
    import ctypes
    import glob
    import subprocess

    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_02242_gb300 import build as b

    b.build()
    so = str(tmp_path_factory.mktemp("internal") / "internal.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-I", os.path.join(ROOT, "include"), "-shared", "-cudart", "shared",
                    "-o", so, os.path.join(HERE, "internal.cu"), *sorted(glob.glob(os.path.join(b.BUILD, "*.o")))],
                   check=True, capture_output=True)
    torch.zeros(1, device="cuda")
    return torch, ctypes.CDLL(so)
