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


# dims and LBMP_OPT_CHUNK of test_gpu_load_ahead.py's cases, and whether f' is loaded ahead
LOAD_AHEAD = [((37, 11, 13), 4, 0), ((37, 11, 13), 5, 1), ((37, 11, 13), 6, 1), ((37, 11, 13), 13, 1), ((32, 4, 11), 5, 1),
              ((5, 3, 64), 0, 0), ((72, 72, 72), 0, 1), ((130, 66, 131), 0, 0)]


def ahead(rules, domains):  # (planes per item, loaded ahead, work items) of (dims, chunk)
    tiles = [-(-nx // 32) * -(-ny // 4) for (nx, ny, _), _ in domains]
    out = rules(*(f"ahead,{t},{dims[2]},{chunk}" for t, (dims, chunk) in zip(tiles, domains)))
    return [(c, a, t * -(-dims[2] // c)) for (c, a), t, (dims, _) in zip(out, tiles, domains)]


def test_load_ahead_cases_reach_both_kernels(rules):
    """The choice is an estimate of the launch's time, and its constants may
    change; the domains that compare the two kernels with the reference pair must
    lie on both sides of it, and in several rounds of the 3 x 152 CTAs."""
    from test_gpu_load_ahead import test_loading_ahead_is_bitwise_the_reference_pair as one_round
    from test_gpu_load_ahead_rounds import DOMAINS
    assert [(c[0], c[2]) for c in one_round.pytestmark[0].args[1]] == [c[:2] for c in LOAD_AHEAD]
    out = ahead(rules, [c[:2] for c in LOAD_AHEAD])
    assert [a for _, a, _ in out] == [a for _, _, a in LOAD_AHEAD]
    assert all(c == chunk for (c, _, _), (_, chunk, _) in zip(out, LOAD_AHEAD) if chunk)
    assert all(a and items > 3 * 152 for _, a, items in ahead(rules, [(dims, 0) for dims, _ in DOMAINS]))
