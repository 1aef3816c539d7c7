"""A model of the weight-row kernels' stage waits, on the CPU: copies land in any order, groups of row threads run at any
relative speed, and a wait by parity passes whenever the number of completed phases has the other parity.  A group must
never read a stage whose codes have not landed (csrc/wide.cu, csrc/slim.cu)."""
import os
import random
import re

import pytest

from conftest import ROOT

WIDE = [(4, 5, 1, True), (4, 6, 1, True), (4, 7, 1, True), (4, 8, 1, True)]    # groups, stages, runs per box, MMAs first
SLIM = [(2, 2, 2, False), (2, 3, 2, False), (2, 4, 2, False),                  # two groups: one run of every box
        (3, 3, 2, True), (3, 2, 2, True)]


def read_early(groups, stages, runs_per_box, nruns, mmas_first, seed):
    rnd = random.Random(seed)
    boxes = -(-nruns // runs_per_box)
    landed, reads, expanded, issued, mma = set(), [0] * boxes, set(), 0, 0
    run, waiting = list(range(groups)), [True] * groups
    for _ in range(200000):
        if all(r >= nruns for r in run):
            return False
        event = rnd.choice(["issue", "land", "mma"] + 2 * list(range(groups)))
        if event == "issue":
            before = issued - stages
            if issued < boxes and (before < 0 or (reads[before] == runs_per_box and mma >= (before + 1) * runs_per_box)):
                issued += 1
        elif event == "land":
            flying = [b for b in range(issued) if b not in landed]
            if flying:
                landed.add(rnd.choice(flying + flying[-1:]))
        elif event == "mma":
            if mma < nruns and mma in expanded and mma // runs_per_box in landed:
                mma += 1
        elif run[event] < nruns:
            r = run[event]
            box, mmas_done = r // runs_per_box, r < groups or mma > r - groups
            if waiting[event]:
                phases = sum(1 for b in landed if b % stages == box % stages)
                if (mmas_first and not mmas_done) or phases % 2 == (box // stages) % 2:
                    continue
                if box not in landed:
                    return True
                reads[box] += 1
                waiting[event] = False
            elif mmas_done:
                expanded.add(r)
                run[event], waiting[event] = r + groups, True
    raise AssertionError("stuck")


@pytest.mark.parametrize("groups,stages,runs_per_box,mmas_first", WIDE + SLIM)
def test_no_stage_is_read_before_its_codes_have_landed(groups, stages, runs_per_box, mmas_first):
    assert not any(read_early(groups, stages, runs_per_box, 24, mmas_first, s) for s in range(150))


def test_the_model_sees_the_mistake():
    """Waiting for the stage before the MMAs of the group's run before lets a wait pass on the phase before."""
    assert any(read_early(4, 7, 1, 40, False, s) for s in range(150))
    assert any(read_early(3, 2, 2, 40, False, s) for s in range(150))


def source(name):
    text = open(os.path.join(ROOT, "paper_2407_11062_b200", "csrc", name)).read()
    return re.sub(r"//[^\n]*", "", text)


def constant(text, name):
    return re.search(r"\b%s = ([^;]+);" % name, text).group(1)


def test_the_model_is_of_the_pair_kernel():
    """Its groups, every number of stages that fits, and the order of its waits."""
    text = source("wide.cu")
    assert {g for g, *_ in WIDE} == {int(constant(text, "kGroups"))} and constant(text, "kRun") == "128"
    assert "return kRows * code_bytes(bits) + tn * 128;" in text and "return 16 * bits;" in text
    room = int(constant(text, "kMaxSmem")) - 1024 - 512
    assert {min(8, room // (128 * 16 * bits + tn * 128)) for bits in (2, 3, 4) for tn in range(32, 257, 32)} == {s for _, s, *_ in WIDE}
    rows = text[text.index("for (int r = g; r < nruns; r += kGroups)"):]
    assert rows.index("ctl->empty[before % stages]") < rows.index("ctl->full_c[st]") < rows.index("load_run<BITS>")
    assert constant(rows, "before") == "r - kGroups" and constant(rows, "st") == "r % stages"


def test_the_model_is_of_the_weight_row_kernel():
    text = source("slim.cu")
    assert constant(text, "kGroups") == "NT <= 2 ? 2 : 3" and constant(text, "kBoxRuns") == "2"
    assert constant(text, "kStages") == "NT == 1 ? (BITS == 2 ? 4 : 3) : (NT == 3 ? 3 : 2)"
    used = {(2 if nt <= 2 else 3, (4 if bits == 2 else 3) if nt == 1 else (3 if nt == 3 else 2)) for bits in (2, 3, 4) for nt in (1, 2, 3, 4)}
    assert used == {(g, s) for g, s, *_ in SLIM}
    rows = text[text.index("for (int r = g; r < nruns; r += kGroups)"):]
    assert rows.index("kGroups > 2 && r != g && !(ok = collect())") < rows.index("ctl->full[st]") < rows.index("load_run<BITS>")
