"""The backward's record capacity is a build-time choice of 32 records a lane
or several: the sources compile for values other than the default."""
import os
import subprocess

import pytest

from paper_2412_04459_gb300 import build


@pytest.mark.parametrize("cap", (32, 96))
def test_record_capacities_compile(cap, tmp_path):
    src = os.path.join(build.CSRC, "render.cu")
    cmd = [build.nvcc(), "-arch=compute_103a", *build.FLAGS, "-Xcicc", "-O0", f"-DSVR_BWD_REC_CAP={cap}", "-ptx", src,
           "-o", str(tmp_path / "render.ptx")]
    out = subprocess.run(cmd, capture_output=True, text=True)
    assert out.returncode == 0, out.stderr[-2000:]
