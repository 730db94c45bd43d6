"""plan_step() makes no plan twice, whatever the workspace (CPU, see
tests/native/plan_calls_check.cpp): planning is host time of every iteration."""
import os
import shutil
import subprocess

import pytest

from paper_2608_15171_gb300 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2608_15171_gb300")


def test_each_plan_once(tmp_path):
    if not os.path.exists(os.path.join(PKG, "libppas.so")):
        pytest.skip("libppas.so is not built")
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path / "plan_calls_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(PKG, "csrc"), "-I",
                    "/usr/local/cuda/include", os.path.join(ROOT, "tests", "native", "plan_calls_check.cpp"), "-o", exe,
                    "-L", PKG, "-lppas", f"-Wl,-rpath,{PKG}", "-L/usr/local/cuda/lib64", "-lcudart", "-ldl"],
                   check=True, capture_output=True, text=True)
    hp, lo = wl.high_pressure_step(0), wl.llama_lo_step(0)
    cases = [(16, 2, [512] * 4, [512, 9000, 20000, 25000]), (16, 2, hp.q_lens, hp.ctx_lens),
             (32, 8, lo.q_lens, lo.ctx_lens), (16, 2, [1] * 8, [25000] * 8), (16, 2, [16384], [16384]),
             (16, 2, [1] * 130 + [700], [4000] * 130 + [9000]),      # more decode rows than a mixed launch takes
             (8, 8, [1] * 3 + [300] * 140, [900] * 143),             # several prefill launches
             (16, 2, [1, 1, 40], [20000, 300, 500])]
    text = "".join(f"{hq} {hk} {len(q)} " + " ".join(map(str, q)) + " " + " ".join(map(str, c)) + "\n"
                   for hq, hk, q, c in cases)
    lines = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    assert lines[:-1] == ["ok"] * len(cases), list(zip(cases, lines))
