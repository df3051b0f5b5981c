"""Rules of the kernels' sources that a run on the GPU cannot show: breaking one gives a wrong sum or a hang
only when warps happen to be scheduled badly, so the sources themselves are read (no GPU needed)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_13846_gb300", "csrc")


def _source(name):
    """A source file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_warp_collectives_name_their_lanes():
    """No collective takes the lanes that happen to be converged for the lanes that take part."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert "__activemask" not in _source(os.path.basename(path)), path


def test_flag_of_other_teams_is_read_by_one_thread():
    """ChainState::failed changes while blocks run: threads that read it for themselves could part at a barrier."""
    text = _source("search.cuh")
    reads = [m.start() for m in re.finditer(r"volatile int\*>\(&[\w.>-]*failed\)", text)]
    assert len(reads) == 2
    for pos in reads:
        start = max(text.rfind(c, 0, pos) for c in ";{}")
        block, depth = [], 0
        for i in range(pos, -1, -1):          # heads of the blocks around the statement
            depth += (text[i] == "}") - (text[i] == "{")
            if depth < 0:
                depth = 0
                block.append(text[max(text.rfind(c, 0, i) for c in ";{}") + 1:i])
        assert "tid == 0" in text[start:pos] or any("tid == 0" in b for b in block)


def test_failed_item_ends_at_a_team_barrier():
    """The exact optimum's blocks copy block 0's status after a step; block 0 resets it for the next item, so no
    way out of an item after the step may skip the barrier of the team."""
    text = _source("search.cuh")
    body = text[text.index("global_items_kernel(const float*"):]
    body = body[body.index("team_neuron_step<DT, SM>"):body.index("template <")]
    assert body.count("continue;") == 1
    for part in body.split("continue;")[:-1]:
        assert "team_sync(tm)" in part[part.rindex("if (sh.status != DTP_OK)"):]
    assert "team_sync(tm)" in body.split("continue;")[-1]
