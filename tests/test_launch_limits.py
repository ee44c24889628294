"""Shared-memory limits of kernels are process-wide: a launch that sets a kernel's limit to its own need can lower it under
a launch that another thread is about to make."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_01219_gb300", "csrc")


def test_only_the_keeper_of_limits_sets_them():
    """Every kernel's limit goes through fit.cu, which holds a mutex and never lowers one."""
    sets = [os.path.basename(f) for f in sorted(glob.glob(os.path.join(CSRC, "*")))
            if re.search(r"\b(cudaFuncSetAttribute|cudaKernelSetAttributeForDevice)\b", open(f).read())]
    assert sets == ["fit.cu"]
