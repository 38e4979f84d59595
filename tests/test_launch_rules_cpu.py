"""The host rules that choose priorities and launch shapes, compiled alone
(tests/launch_rules.cu)."""
import os
import subprocess

import pytest

from paper_2101_06769_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("launch_rules") / "launch_rules")
    subprocess.run([B._nvcc()] + B.ARCH + B.FLAGS + ["-I", B.CSRC, os.path.join(HERE, "launch_rules.cu"), "-o", exe],
                   check=True)

    def ask(*queries):
        out = subprocess.run([exe, *queries], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]
        return [[int(v) for v in line.split()] for line in out]
    return ask


def test_second_branch_of_a_batch_is_one_level_above_its_stream(rules):
    """never further before the caller's other work, never above the device's greatest"""
    assert rules("priority,0,-5", "priority,-2,-5", "priority,-5,-5", "priority,0,0") == [[-1], [-3], [-5], [0]]
