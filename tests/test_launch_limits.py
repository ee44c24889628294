"""What no GPU run can be made to show: launches of two threads that meet in a moment, waits that give up."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_01219_gb300", "csrc")


def test_only_the_keeper_of_limits_sets_them():
    """Shared-memory limits of kernels are process-wide: a launch that sets a kernel's limit to its own need can lower it
    under a launch that another thread is about to make.  Every limit goes through fit.cu, which holds a mutex and never
    lowers one."""
    sets = [os.path.basename(f) for f in sorted(glob.glob(os.path.join(CSRC, "*")))
            if re.search(r"\b(cudaFuncSetAttribute|cudaKernelSetAttributeForDevice)\b", open(f).read())]
    assert sets == ["fit.cu"]


def test_a_result_names_its_own_error(tmp_path):
    """A TAM wait that gave up is not reported as a scan without a valid beam (no GPU run can make the wait give up)."""
    from paper_2511_01219_gb300 import _build
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build._nvcc()))), "include")
    src = tmp_path / "words.cpp"
    src.write_text('#include <stdio.h>\n#include "relo_internal.h"\n'
                   "int main() { printf(\"%s\\n%s\\n\", relo::result_error(RELO_E_CUDA),"
                   " relo::result_error(RELO_E_NO_VALID_BEAMS)); }\n")
    exe = tmp_path / "words"
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, "-I", cuda, str(src), "-o", str(exe)])
    wait, beams = subprocess.check_output([str(exe)], text=True).splitlines()
    assert "gave up waiting" in wait and "valid beam" not in wait
    assert "valid beam" in beams
    api = open(os.path.join(CSRC, "relo_api.cu")).read()
    assert "result_error(out[i].status)" in api and '"a scan has no valid beam"' not in api
