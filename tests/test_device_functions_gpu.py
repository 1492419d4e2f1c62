"""Device functions on their own, in programs built from the library's headers: the ordered
spreading by strips against the per-cell form to the bit, and the FP64 helpers against the
plain operations."""
import os
import subprocess

import pytest

from conftest import ROOT
from paper_1407_6704_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["strips_vs_cells", "fp64_helpers"])
def test_program(name, tmp_path):
    exe = str(tmp_path / name)
    src = os.path.join(ROOT, "tests", "native", name + ".cu")
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, src, "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    print(res.stdout)
    assert res.returncode == 0, res.stdout
