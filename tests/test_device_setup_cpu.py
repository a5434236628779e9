"""Kernel set-up is kept per device: a shared-memory limit raised while one GPU is current does not
hold on another one that the process drives.  No machine of these tests has two GPUs, so the launch
code itself is looked at."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2603_20889_gb300", "csrc")
FILES = [p for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))) if "cudaFuncSetAttribute" in open(p).read()]


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_limits_are_not_guarded_by_process_wide_state(path):
    src = open(path).read()
    for at in (m.start() for m in re.finditer("cudaFuncSetAttribute", src)):
        launch = src[src.rfind("\n}", 0, at):at]  # the launching function up to the call
        guards = re.findall(r"if \(!?(\w+)(?: == 0)?\) \{\n[^}]*$", launch)
        for g in guards:
            assert re.search(r"& %s = \w+\[device_slot\(\)\]" % g, launch), (os.path.basename(path), g)
