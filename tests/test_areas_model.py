"""First keys of an attention phase against the sums of the QKV phase before it, which lie in the same shared memory: the header
that the pass kernel takes its addresses and its rule from (csrc/ada_areas.h), driven on the host by warps in random order."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("areas") / "areas_model")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2412_18910_b200", "csrc"), "-o", exe,
                           os.path.join(ROOT, "tests", "areas_model.cpp")])
    return exe


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("rows", [1, 8, 9, 16, 17, 18, 24, 25, 33, 48])
def test_no_key_lands_on_sums_still_needed(model, rows, head_dim):
    r = subprocess.run([model, str(rows), str(2 * head_dim), "50"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
