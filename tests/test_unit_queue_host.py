"""The hand-over of units of work between the roles of a kernel, run on the host: in the usual course, and when a wait runs out."""
import os
import subprocess

from tests.conftest import ROOT


def test_hand_over_of_units(tmp_path):
    exe = tmp_path / "unit_queue"
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2410_09397_b200", "csrc"),
                    os.path.join(ROOT, "tests", "unit_queue_host.cpp"), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
