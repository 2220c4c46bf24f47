"""What the fused joiner's instances keep outside their registers, from ptxas: a change of its epilogue that helps one segment size can
cost another one.  The epilogue holds 64 exponentials a lane with 256 columns to a CTA, 32 with 128 and 16 with 64, of 96 registers."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2302_14357_b200 import build as tw_build

# spill-store bytes a thread by (columns, logits bounded): at most these for any segment size
LIMIT = {(64, False): 0, (64, True): 0, (128, False): 16, (128, True): 20, (256, False): 164, (256, True): 72}


@pytest.fixture(scope="module")
def ptxas_output(tmp_path_factory):
    nvcc = tw_build._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    out = str(tmp_path_factory.mktemp("joiner") / "fused_joiner.o")
    res = subprocess.run([nvcc] + tw_build.NVCC_FLAGS + ["-Xptxas", "-v", "-c", os.path.join(tw_build.CSRC, "fused_joiner.cu"), "-o", out],
                         capture_output=True, text=True, check=True)
    return res.stdout + res.stderr


def test_spills_of_every_instance(ptxas_output):
    spills, at = {}, None
    for line in ptxas_output.splitlines():
        m = re.search(r"fused_joiner_kernelILi(\d+)ELb([01])ELi(\d+)E", line)
        if m:
            at = (int(m[3]), m[2] == "1", int(m[1]))
        m = re.search(r"(\d+) bytes spill stores", line)
        if m and at is not None:
            spills[at], at = int(m[1]), None
    assert len(spills) == 3 * 2 * 12
    over = {k: v for k, v in spills.items() if v > LIMIT[k[:2]]}
    assert not over, over


def test_compiles_without_warnings(ptxas_output):
    assert "warning" not in ptxas_output
