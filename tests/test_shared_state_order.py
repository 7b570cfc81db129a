"""The memory order of tour 0's kept states in split_shared.cu, read from the
source: warp 0 writes a state with all its lanes, a warp barrier, then lane 0's
release of the count; a warp that resumes acquires the count with lane 0, and
every lane reads the state.  An acquire orders the reads of the lane that made
it; a warp barrier between it and the resumed tour carries that to the other
lanes, which __shfl_sync does not."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2602_05179_gb300", "csrc", "split_shared.cu")


def _code():
    return re.sub(r"//[^\n]*", "", open(SRC).read())


def test_every_lane_is_ordered_behind_the_acquire():
    code = _code()
    assert code.count("ld_acquire_shared(&snap_ready)") == 1
    behind = code[code.index("ld_acquire_shared(&snap_ready)"):]
    resumed = behind.index("run_tour<QT, false, false>")
    assert 0 <= behind.find("__syncwarp();") < resumed


def test_the_state_is_written_before_its_release():
    code = _code()
    keep = code[code.index("save_state(st,"):]
    assert 0 <= keep.find("__syncwarp();") < keep.index("st_release_shared(snap.ready")
