"""The file of timed y-pass forms (tune_file.h): only choices that were timed on
this library's own pass code are taken from it.  Host code only."""
import json
import os
import shutil
import subprocess

import pytest

from test_engine_host import BUILD, CSRC, HERE

from paper_1106_0557_gb300 import build

ENTRIES = [[0, 512, 256, 256, 256, 103, 1, 1], [2, 768, 384, 300, 300, 103, 0, 2]]


@pytest.fixture(scope="module")
def exe():
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    os.makedirs(BUILD, exist_ok=True)
    out = os.path.join(BUILD, "tune_file_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", out, os.path.join(HERE, "tune_file_check.cpp")],
                   check=True)
    return out


def _taken(exe, tmp_path, content, code=77):
    a, b = tmp_path / "a.json", tmp_path / "b.json"
    a.write_text(content)
    subprocess.run([exe, str(a), str(code), str(b), "5"], check=True)
    got = json.loads(b.read_text())
    assert got["code"] == 5
    return got["y_pass_forms"]


def test_choices_of_the_same_code_are_taken(exe, tmp_path):
    assert _taken(exe, tmp_path, json.dumps({"code": 77, "y_pass_forms": ENTRIES})) == ENTRIES
    # entries that name no form of this library are left out
    bad = ENTRIES + [[0, 64, 32, 32, 32, 103, 3, 0], [1, 64, 32, 32, 32, 103, 0, -1]]
    assert _taken(exe, tmp_path, json.dumps({"code": 77, "y_pass_forms": bad})) == ENTRIES


@pytest.mark.parametrize("content", [
    json.dumps({"code": 78, "y_pass_forms": ENTRIES}),  # other code
    json.dumps({"y_pass_forms": ENTRIES}),              # none named
    json.dumps({"code": 77, "y_pass_forms": [ENTRIES[0][:5]]}), "", "[]", "{"])
def test_choices_of_other_code_are_not(exe, tmp_path, content):
    assert _taken(exe, tmp_path, content) == []


def test_the_digest_covers_the_pass_code():
    assert build._pass_code() != build._spectrum_code()
    assert any("-DISOFFT_PASS_CODE=" + build._pass_code() in u[2] for u in build._units() if u[0] == "api")
