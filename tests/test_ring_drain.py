"""A kernel whose bounded wait ran out leaves only once the copies it issued
have landed (CPU: a timeout is not provoked on a GPU).  The phases it waits
for are checked against a model of the barriers (tests/native/
ring_drain_check.cpp); that the kernels wait for them, in their source."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_15171_gb300", "csrc")


def test_waits_cover_every_copy_in_flight(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path / "ring_drain_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I",
                    "/usr/local/cuda/include", os.path.join(ROOT, "tests", "native", "ring_drain_check.cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], capture_output=True, text=True).stdout
    assert out.strip() == "ok", out


@pytest.mark.parametrize("source,kernel,wait", [
    ("gateup.cu", "gateup_swiglu_kernel", "ring_pair_newest("),
    ("gateup.cu", "gateup_few_kernel", "ring_land("),
    ("attn_prefill.cu", "prefill_cta", "ring_land(bar(q ? B_Q : v ? B_VFULL : B_KFULL)"),
])
def test_kernels_wait_for_them(source, kernel, wait):
    with open(os.path.join(CSRC, source)) as f:
        text = f.read()
    start = re.search(rf"^[^/\n]*\b{kernel}\(.*$", text, re.M).start()
    body = text[start:text.index("\n}\n", start)]
    assert wait in body
