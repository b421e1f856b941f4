"""Rules of ordering that the kernels keep, checked in their sources: breaking one is a race, which a run need not show (no GPU needed)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_15919_b200", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _between(src, start, end):
    i = src.index(start)
    return src[i:src.index(end, i)]


def test_simulator_orders_an_admission_before_its_commit():
    # single lanes note what is admitted (s_park, s_word, s_byte); the commit reads the notes with other lanes
    src = _source("hfx_sim.cu")
    last_note = src.rindex("park(adm_cnt", 0, src.index("parked(e0"))
    between = src[last_note:src.index("parked(e0")]
    # in a block that every iteration with an admission passes (not inside `if (from_list)` or a loop over the list)
    assert re.search(r"if \(adm_cnt > 0\) __syncwarp\(\);", between)


def test_simulator_orders_reading_a_slot_before_the_samples_overwrite_it():
    # the TTFT samples are closed up over the slots of the same 32 rows, of which those in flight are read just before
    src = _source("hfx_sim.cu")
    assert "__syncwarp();" in _between(src, "s_slot[i] >> 32);\n            last", "s_slot[n_ttft")
