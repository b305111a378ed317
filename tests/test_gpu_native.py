"""Device code that the C interface does not reach on its own (native_checks.cu)."""
import os
import subprocess

import pytest

from paper_2405_05446_gb300 import build as B

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("native") / "native_checks")
    cmd = [B._nvcc()] + B.ARCH + B.FLAGS + ["-o", exe, os.path.join(HERE, "native_checks.cu"),
                                            os.path.join(B.CSRC, "diag.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return exe


@pytest.mark.parametrize("what", ["sort", "div"])
def test_native(checks, what):
    """sort: behind a bounded wait that gave up no pass of either sort runs, also where the
    status already holds another error (the lists they would read were never written); div:
    the packed division gives CUDA's quotient over the transmittances of 1 to 2^-100."""
    r = subprocess.run([checks, what], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
