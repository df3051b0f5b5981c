"""Rules of the kernels' sources that a run on the GPU cannot show: breaking one gives a wrong sum or a hang
only when warps happen to be scheduled badly, so the sources themselves are read (no GPU needed)."""
import glob
import os
import re
import subprocess

import pytest

from paper_2609_13846_gb300 import build

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


@pytest.mark.parametrize("budget,builds", [(184, True), (166, True), (160, False), (4, False)])
def test_shared_memory_budget_and_workspace_rule_agree(tmp_path, budget, builds):
    """Layers that ask for no workspace must fit one block: a budget too small for that does not build."""
    text = open(os.path.join(CSRC, "search.cuh")).read()
    line = "constexpr size_t kSmemBudget = 184 * 1024;"
    assert text.count(line) == 1
    (tmp_path / "search.cuh").write_text(text.replace(line, f"constexpr size_t kSmemBudget = {budget} * 1024;"))
    (tmp_path / "t.cu").write_text('#include "search.cuh"\n')
    cmd = [build.nvcc(), *build.ARCH, "-std=c++17", "-I", os.path.join(build.ROOT, "include"), "-I", CSRC, "-c",
           str(tmp_path / "t.cu"), "-o", str(tmp_path / "t.o")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert (r.returncode == 0) == builds, r.stderr
    assert builds or "layers without a workspace fit one block" in r.stderr
