"""Kernels' own sources compiled for the host and run as one CTA on threads
(host/cuda_runtime.h): schedules of the warps and operands that a GPU run does not
choose."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _program(tmp, name):
    out = os.path.join(str(tmp), name)
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("needs g++")
    subprocess.run([cc, "-std=c++20", "-O1", "-ffp-contract=off", "-pthread", "-w", "-I", os.path.join(HERE, "host"), "-I",
                    os.path.join(ROOT, "paper_2602_15838_gb300", "csrc"), os.path.join(HERE, "host", name + ".cpp"), "-o", out],
                   check=True, capture_output=True, text=True)
    return out


@pytest.fixture(scope="module")
def polish(tmp_path_factory):
    return _program(tmp_path_factory.mktemp("host"), "polish")


@pytest.mark.parametrize("what,want", [(0, "0 1 0 0 0 0 1"), (1, "0 0 0 0 0 256 1"), (2, "0 0 0 0 0 0 1")])
def test_polishing_round_under_every_late_warp(polish, what, want):
    """One polishing round changes one row, whichever warp comes late after whichever
    barrier: the row it takes is found in two searches, and a warp that reads the
    first one's result must not see the second one's."""
    for warp in range(4):
        for at in range(8):
            r = subprocess.run([polish, str(what), str(warp), str(at)], capture_output=True, text=True, timeout=60)
            assert r.returncode == 0 and r.stdout.strip() == want, (warp, at, r.returncode, r.stdout)


@pytest.fixture(scope="module")
def ratio(tmp_path_factory):
    return _program(tmp_path_factory.mktemp("host"), "ratio")


@pytest.mark.parametrize("what", ["near", "1", "2", "3"])
def test_ratio_scan_equals_ratio_test(ratio, what):
    """The ratio test over the lanes takes the blocking input of the test in index
    order: beside inputs whose distance to a bound float32 cannot tell from 0, and on
    random steps on either side of what stays in registers (128 inputs)."""
    r = subprocess.run([ratio, what], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert int(r.stdout) >= 20


def test_graph_state_after_a_failed_allocation(tmp_path):
    """Whichever block of the graph mode's state cannot be allocated, the handle keeps
    none, and the next solve starts over (a later one failing must not leave the first
    as the mark of a complete state)."""
    r = subprocess.run([_program(tmp_path, "graph_state")], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and int(r.stdout) == 8, (r.returncode, r.stdout, r.stderr)


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    return _program(tmp_path_factory.mktemp("host"), "rules")


@pytest.mark.parametrize("scenarios,want", [
    ([(14, 20, 1)], 1), ([(2, 20, 1)], 1), ([(14, 24, 1)], 1), ([(14, 25, 1)], 0), ([(32, 20, 1)], 0), ([(8, 80, 1)], 0),
    ([(32, 1280, 1)], 0), ([(32, 20, 64)], 0), ([(32, 20, 256)], 1), ([(4, 20, 300), (32, 2560, 1)], 0), ([(33, 2, 1)], 0),
    ([(4, 70000, 1)], 1)])
def test_tail_rule_of_the_graph_mode(rules, scenarios, want):
    """One CTA per scenario for what comes after the x-update only where the measured
    times (beside the rule) have it ahead or level: not for long horizons."""
    r = subprocess.run([rules, "tail", "152"] + [str(v) for s in scenarios for v in s], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and int(r.stdout) == want, r.stdout


# batches of which every shape was timed (beside the rule): CTAs of 128, 64 and 32 threads
# that an SM holds, groups (agents, steps, how many), the fastest
@pytest.mark.parametrize("resident,groups,want", [
    ((2, 4, 8), [(16, 30, 800), (64, 30, 1), (200, 30, 1)], 128), ((2, 3, 3), [(16, 30, 800), (64, 30, 1)], 128),
    ((2, 2, 2), [(16, 30, 800), (90, 30, 1)], 128), ((2, 3, 3), [(32, 30, 2200), (64, 30, 1)], 64),
    ((2, 4, 8), [(32, 30, 2200), (100, 30, 1)], 64), ((2, 4, 7), [(40, 25, 1500)], 64),
    ((2, 4, 5), [(48, 40, 20), (41, 30, 280)], 128), ((2, 4, 8), [(90, 22, 200)], 128), ((2, 2, 2), [(90, 40, 1)], 128)])
def test_threads_with_large_scenarios(rules, resident, groups, want):
    r = subprocess.run([rules, "threads", "152", *map(str, resident), "0"] + [str(v) for g in groups for v in g],
                       capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and int(r.stdout) == want, r.stdout


@pytest.mark.parametrize("groups,relaxed,want", [(190, 0, 128), (304, 0, 128), (305, 0, 64), (608, 0, 64), (609, 0, 32),
                                                 (2223, 0, 32), (2223, 1, 128)])
def test_threads_of_small_groups(rules, groups, relaxed, want):
    r = subprocess.run([rules, "threads", "152", "0", "0", "0", str(relaxed), "20", "30", str(groups)],
                       capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and int(r.stdout) == want, r.stdout
