"""The bounded waits of the persistent decode step: a poll whose flag nothing sets gives up
after its limit of looks, sets DEVERR_TIMEOUT and the abort words, and later waits return
at once. One CTA, no ring and no copies in flight; the status is read on the host."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
DEVERR_TIMEOUT = 8


def test_poll_gives_up_and_reports(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_19889_gb300 import build
    so = str(tmp_path / "poll_bound.so")
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-I" + build.CSRC,
                    os.path.join(HERE, "poll_bound.cu"), "-o", so], check=True)
    out = (ctypes.c_int * 4)()
    assert ctypes.CDLL(so).run_poll(8192, out) == 0
    assert list(out) == [0, 1, 1, DEVERR_TIMEOUT]
