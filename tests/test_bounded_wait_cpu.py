"""The give-up path of the device code's bounded wait, run on CPU threads.

Every wait in the kernels goes through ``csrc/bounded_wait.h``.  The same source is compiled here for the host:
two threads play two warps, one arrival is withheld, and the waits must end by themselves; four threads play the lanes
of one warp, which must all leave a wait with the same result.  Another test maps
the sticky device-side error word to the status the host reports.  Nothing is withheld on a GPU."""
import glob
import os
import re
import subprocess

import pytest

from paper_2503_05931_b200 import binding, build_ext

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    exe = tmp_path_factory.mktemp("wait") / "wait_host_check"
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", os.path.join(HERE, "wait_host_check.cpp"), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")
    return {l.split()[0]: [int(v) for v in l.split()[1:]] for l in out if l.strip()}


def test_wait_gives_up_and_raises_the_abort_word(rows):
    assert rows["complete"][:3] == [1, 1, 0]                 # both waits satisfied, abort word untouched
    r0, r1, abort_word, ms1 = rows["withheld"]
    assert (r0, r1, abort_word) == (0, 0, 1)                 # both gave up, the abort word is raised
    assert ms1 < 2000                                        # the second waiter left through the abort word, not its 5 s limit


def test_lanes_of_a_warp_leave_a_wait_together(rows):
    """Where lanes that decide for themselves would leave with different results, the vote gives all of them one."""
    for what in ("phase", "clock"):
        *alone, _, _ = rows[f"lanes_{what}_alone"]
        assert len(set(alone)) == 2, "the schedule should be one that splits the lanes"
        *lanes, abort_word, left_behind = rows[f"lanes_{what}"]
        assert (lanes, abort_word, left_behind) == ([0, 0, 0, 0], 1, 0)


def test_every_device_wait_takes_the_vote():
    calls = 0
    for path in glob.glob(os.path.join(build_ext.CSRC, "*.cu*")):
        with open(path) as f:
            source = f.read()
        for m in re.finditer(r"\bbounded_poll\(", source):
            calls += 1
            assert "WarpVote()" in source[m.start():source.index("kWaitCycles", m.start()) + 60], path
        # the one other form of the instruction: poll loops of a warp's own
        assert "mbarrier.try_wait" not in source or "bounded_poll" in source, path
    assert calls == 2


def test_error_word_maps_to_a_status():
    build_ext.build()
    lib = binding.load_library()
    assert lib.aed_dec_status_of_error_word(0) == binding.AED_OK
    assert lib.aed_dec_status_of_error_word(1) == binding.AED_ERR_CAPACITY
    for word in (2, 3, 77):                                  # 2 is what a kernel writes when a wait ran out
        assert lib.aed_dec_status_of_error_word(word) == binding.AED_ERR_TIMEOUT
