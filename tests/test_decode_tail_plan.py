"""Decode splits of mixed steps: the last third of the rows in halves (CPU, see
tests/native/decode_tail_check.cpp)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2608_15171_gb300 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2608_15171_gb300")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if not os.path.exists(os.path.join(PKG, "libppas.so")):
        pytest.skip("libppas.so is not built")
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("tail") / "decode_tail_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(PKG, "csrc"), "-I",
                    "/usr/local/cuda/include", os.path.join(ROOT, "tests", "native", "decode_tail_check.cpp"), "-o",
                    exe, "-L", PKG, "-lppas", f"-Wl,-rpath,{PKG}", "-L/usr/local/cuda/lib64", "-lcudart"],
                   check=True, capture_output=True, text=True)
    return exe


def _run(exe, cases, sms):
    text = "".join(f"{sms} {hq} {hk} {len(q)} " + " ".join(map(str, q)) + " " + " ".join(map(str, c)) + "\n"
                   for hq, hk, q, c in cases)
    lines = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    return [x for x in lines if x]


@pytest.mark.parametrize("sms", [152, 31, 256])
def test_random_mixed_and_decode_only_steps(checker, sms):
    rng = np.random.default_rng(sms)
    cases = []
    for _ in range(80):
        nd, npf = int(rng.integers(0, 130)), int(rng.integers(0, 5))
        hk = int(rng.choice([1, 2, 8]))
        q = [1] * nd + [int(rng.integers(2, 700)) for _ in range(npf)]
        c = [x + int(rng.integers(0, rng.choice([40, 3000, 40000]))) for x in q]
        if q:
            cases.append((hk * int(rng.choice([1, 4, 8])), hk, q, c))
    # rows at the longest context: their splits stay as they are
    cases.append((16, 2, [1] * 6 + [64], [1 << 25] * 6 + [64]))
    for case, line in zip(cases, _run(checker, cases, sms)):
        assert line.startswith("ok"), (case, line)


def test_paper_workloads(checker):
    hp, lo = wl.high_pressure_step(0), wl.llama_lo_step(0)
    got = _run(checker, [(16, 2, list(hp.q_lens), list(hp.ctx_lens)), (32, 8, list(lo.q_lens), list(lo.ctx_lens))], 152)
    assert got[0].startswith("ok") and got[1].startswith("ok"), got
    assert [int(x.split()[2]) > int(x.split()[1]) for x in got] == [True, True]
