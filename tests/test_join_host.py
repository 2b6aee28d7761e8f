"""Rules of the join kernel that need no GPU to be checked (host build)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not installed")
    exe = tmp_path_factory.mktemp("join") / "join_host_check"
    subprocess.check_call(["nvcc", "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2101_07690_gb300", "csrc"),
                           "-o", str(exe), os.path.join(ROOT, "tests", "join_host_check.cu")])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    return dict(line.rsplit(" ", 1) for line in out.stdout.splitlines())


def test_debug_checks_an_index_against_its_own_list(report):
    assert report["bounds"] == "0"


def test_tables_as_the_device_fills_them_match_the_rule(report):
    """Both tables of every stored size, that of size 5 by its own way over the 2^21 graphs of 7 vertices."""
    assert int(report["kept"]) > 1000
    assert report["acc"] == "0" and report["any"] == "0"
