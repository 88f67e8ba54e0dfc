"""Host logic: pointer tables of a plan run serve the next one only where every plane's
scratch lies in the present arena (tests/host/tables_check.cpp), and the engine asks for
that with the arena's own sizes and forgets the tables when it gives an arena back.  No GPU
involved."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1712_08872_gb300", "csrc")


def test_tables_serve_only_within_the_arena(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "tables_check")
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "tables_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout


def test_engine_forgets_tables_of_an_arena_given_back():
    with open(os.path.join(CSRC, "acr_engine.cu")) as fh:
        text = fh.read()
    free = re.search(r"void free_work\(Work& k\) \{(.*?)\n  \}", text, re.S).group(1)
    assert "tabs.epoch = -1" in free
