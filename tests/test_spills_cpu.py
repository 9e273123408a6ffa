"""Register spills of the kernels that are launched at their register limit: ptxas reports none. The decode
FFN's builds of 9 to 64 tokens take all 128 registers of two CTAs per SM, so a change as small as another
order of its parameters can push values to local memory."""
import os
import re
import subprocess

import pytest

from paper_2609_34077_gb300 import build


@pytest.mark.parametrize("src", ["ffn_decode.cu"])
def test_no_spills(src, tmp_path):
    cmd = [build._nvcc(), *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, src),
           "-o", str(tmp_path / "x.o")]
    r = subprocess.run(cmd, capture_output=True, text=True, check=True)
    spills = re.findall(r"(\d+) bytes spill stores, (\d+) bytes spill loads", r.stdout + r.stderr)
    assert spills and all(s == ("0", "0") for s in spills), spills
