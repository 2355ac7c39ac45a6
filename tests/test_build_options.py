"""Build options of csrc/ that compile code of their own: the sources build
with them (no GPU)."""
import os

import pytest

from paper_1711_00231_gb300 import _build


@pytest.mark.parametrize("src,flags", [("lb_serve.cu", ["-DLB_SERVE_PROFILE=1"])])
def test_builds_with(src, flags, tmp_path):
    import subprocess
    cmd = [_build._nvcc(), *_build.NVCC_FLAGS, *flags, "-ptx", os.path.join(_build.CSRC, src), "-o", str(tmp_path / "x.ptx")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
