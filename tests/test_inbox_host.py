"""The inboxes of a list chain (csrc/inbox.h) under adversarial interleavings
of the blocks, on the host: inbox_model.cpp compiled against the header."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2607_15906_gb300", "csrc")


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("inbox") / "inbox_model")
    subprocess.run([cxx, "-O1", "-std=c++17", f"-I{CSRC}", os.path.join(HERE, "inbox_model.cpp"), "-o", exe],
                   check=True)
    return lambda rule, runs: int(subprocess.run([exe, str(rule), str(runs)], check=True, capture_output=True,
                                                 text=True).stdout)


def test_a_step_sees_exactly_the_entries_of_earlier_steps(model):
    assert model(0, 20000) == 0


def test_the_model_finds_a_word_that_is_written_while_it_is_read(model):
    """One length word, raised by the step that is being read, and a flag
    without its step: the schedules reach the fault."""
    assert model(1, 2000) > 0
