"""The launch plan (csrc/plan.h), compiled for the host: the bounded search finds
the chunk that a search over every chunk count finds, and a plan for 30,000
planes takes no longer than one for 256 (within a factor of 4; a search over
every count took 100 times as long and was made for every launch).  The back
end plans once per call, outside its loop over steps.  CPU only."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1705_10045_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    out = tmp_path_factory.mktemp("plan") / "plan_host"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-I", CSRC,
                           os.path.join(ROOT, "tests", "c", "plan_host.cc"), "-o", str(out)])
    text = subprocess.check_output([str(out)], text=True)
    return {line.split()[0]: float(line.split()[1]) for line in text.splitlines()}


def test_bounded_search_finds_what_the_full_search_finds(program):
    assert program["checked"] == 20 * 8 * 8 * 2 and program["wrong"] == 0


def test_plan_time_does_not_grow_with_the_planes(program):
    assert program["long_us"] <= 4.0 * program["short_us"], program


def test_a_call_plans_outside_its_loop_over_steps():
    with open(os.path.join(CSRC, "backend.cuh")) as f:
        text = f.read()
    for name in ("step", "profile"):
        body = text[re.search(r"static int %s\(lbm_handle\* h, int n" % name, text).start():]
        body = body[: body.index("\n    }\n")]
        loop = body.index("for (int s = 0; s < n")
        assert body.index("plan(h)") < loop and "plan(" not in body[loop:], name
    for name in ("launch", "launch_fused", "launch_phase"):
        body = text[re.search(r"static void %s\(lbm_handle\* h" % name, text).start():]
        body = body[: body.index("\n    }\n")]
        assert not re.search(r"\b(plan|march_chunk|row_chunk|strip_rows)\(", body), name
