"""Host logic: plans built with the engine's own parameters (one core stage per plan, and one
basis stage for float factors), executed on the CPU as the kernels read them
(tests/host/plan_stages.cpp), reproduce exact operations, alone and merged; bundles
and target ranges cover their stages once; and every kind of stage that a plan of the
engine holds is one that it runs.  No GPU involved."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1712_08872_gb300", "csrc")


@pytest.fixture(scope="module")
def stages(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("plan") / "plan_stages")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "tests", "host"),
                    os.path.join(ROOT, "tests", "host", "plan_stages.cpp"),
                    os.path.join(CSRC, "acr_plan.cpp"), os.path.join(CSRC, "acr_structure.cpp"),
                    "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n,eta,leaf", [(16, 2.0, 16), (16, 2.0, 32), (16, 1.0, 16),
                                        (20, 2.0, 64), (32, 2.0, 64)])
@pytest.mark.parametrize("fused", [0, 1])
def test_plans_as_the_engine_runs_them(stages, n, eta, leaf, fused):
    r = subprocess.run([stages, str(n), str(eta), str(leaf), str(fused)], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.count(" ok") == 6, r.stdout


def test_engine_refuses_stages_it_does_not_run():
    """Only Cholesky stages reach the Cholesky launch; any other kind is an error."""
    with open(os.path.join(CSRC, "acr_engine.cu")) as fh:
        text = fh.read()
    run = text[text.index("for (const Stage& sg : pl.stages)"):text.index("launch_pchol<T>(pl, sg.beg")]
    assert re.search(r"sg\.kind != ST_PCHOL && sg\.kind != ST_PCHOL \+ 16\)\s*\n\s*throw AcrError", run)
