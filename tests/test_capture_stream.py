"""A gradient run that cannot make its capture stream goes on without graphs: the failed
creation leaves no error for the next launch to report (on a fake of the failing call)."""
import os
import subprocess

from conftest import ROOT
from paper_1407_6704_gb300 import build


def test_no_error_stays_behind(tmp_path):
    exe = str(tmp_path / "capture_stream")
    src = os.path.join(ROOT, "tests", "native", "capture_stream.cu")
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, src, "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
