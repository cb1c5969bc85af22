"""A step on host weights in parts when something cannot be queued half-way (``csrc/ciera_host_step.hpp``), played
through on the CPU with an object that fails one call after the other."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2609_04609_b200", "csrc")
PARTS = 3


@pytest.fixture(scope="module")
def play(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("host_step") / "host_step_order")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, os.path.join(HERE, "host_step_order.cpp"), "-o", exe],
                   check=True)

    def run(failing, sticky=0):
        words = subprocess.run([exe, str(PARTS), str(failing), str(sticky)], check=True, capture_output=True, text=True).stdout.split()
        return words[:-1], int(words[-1][2:])

    return run


def test_order_without_a_failure(play):
    ops, rc = play(0)
    assert rc == 0
    assert ops == ["in0", "in1", "in2", "step0", "out0", "step1", "out1", "step2", "out2", "join0"]


@pytest.mark.parametrize("k", range(PARTS))
def test_a_range_that_cannot_be_copied_in_leaves_everything_as_it_was(play, k):
    ops, rc = play(k + 1)
    assert rc == -101 - k
    assert ops == [f"in{i}" for i in range(k)] + [f"in{k}!", "join0"]  # nothing stepped


@pytest.mark.parametrize("k", range(PARTS))
def test_a_part_that_cannot_be_launched_has_the_workspace_emptied(play, k):
    call = PARTS + 2 * k + 1
    ops, rc = play(call)
    assert rc == -100 - call
    done = [x for i in range(k) for x in (f"step{i}", f"out{i}")]
    assert ops == ["in0", "in1", "in2"] + done + [f"step{k}!", "clear", "join0"]


@pytest.mark.parametrize("sticky", [0, 1])
@pytest.mark.parametrize("k", range(PARTS))
def test_a_range_that_cannot_be_copied_out_does_not_end_the_step_on_the_device(play, k, sticky):
    call = PARTS + 2 * k + 2
    ops, rc = play(call, sticky)
    assert rc == -100 - call  # the first error
    assert [x.rstrip("!") for x in ops] == play(0)[0]


def test_a_failing_join_is_reported(play):
    assert play(3 * PARTS + 1)[1] == -100 - (3 * PARTS + 1)
