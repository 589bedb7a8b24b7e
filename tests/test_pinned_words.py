"""The pinned words that pair queries copy their results to (csrc/pinned_words.h), on the host
with plain memory: words go back to the pool only when no copy into them can be under way."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    exe = tmp_path_factory.mktemp("pinned") / "harness"
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-Wall", "-I",
                    os.path.join(ROOT, "paper_2301_00611_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "pinned_words_harness.cpp"), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stderr
    return res.stdout.splitlines()


@pytest.mark.parametrize("name", ["reused", "withheld", "bounded"])
def test_scenario(harness, name):
    assert f"{name} ok" in harness
